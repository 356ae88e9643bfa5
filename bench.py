#!/usr/bin/env python3
"""Benchmark of the IIM Poisson hot path: solves/s on the single-cylinder workload at 1024^2
cells to a relative un-reduced residual of 1e-10 (chosen form: FP32 transforms inside FP64
iterative refinement), with the plain FP64 iteration timed beside it.

One step = B independent iim_poisson_solve calls (omega -> psi, u) in flight together through the
C ABI (iim_poisson_solve_batched) with inputs resident in HBM.  L2 is flushed (256 MiB write)
before every timed step; the flush is outside the step's CUDA events.  Under torchrun each rank
runs independent solves on its own GPU (replicas, weak scaling): time = max over ranks, solves
= sum over ranks; rank 0 prints one JSON line.

--impl reference times the CPU oracle (Schur-form GMRES with scipy's DST-I, FP64) on the
host cores on the same workload, metric and unit.
"""
import argparse
import hashlib
import json
import math
import os
import statistics
import subprocess
import tempfile
import sys
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

METRIC = "IIM Poisson solves/s at 1024² to 1e-10 residual: chosen form vs plain FP64"
UNIT = "solves/s"
N_CELLS = 1024
RTOL = 1e-10
WORKLOAD = ("c1_cylinder_1024: [-2,2]^2, 1024x1024 cells (1023^2 unknowns), one cylinder R=0.5 at the origin, "
            "manufactured psi = sin(pi x/2) sin(pi y/2) + 0.1 log r, Dirichlet box and body data from psi, "
            "fixed-psibar body, solve to un-reduced FP64 relative residual 1e-10")
# DRAM traffic per launch of the dominant kernel from the committed ncu captures, valid for the hash of the
# kernel's source files (null otherwise).
NCU_TRAFFIC = {
    # python -m paper_2109_13628_gb300.passes --n 1024 --col 0 (column DSTs) or 1 --batch 40 under ncu --metrics
    # (DRAM and L2 sector counters, -k regex:<kernel> -c 1): 40 fields in one launch; scaled by the fields to
    # the roofline's launch of 95 fields
    # k_cols: DRAM 167.7 MB read + 112.3 MB written, L2 12.92 M + 5.24 M sectors
    "dst_cols_f32": {"bytes_per_launch": 280002816 / 40 * 95, "l2_bytes_per_launch": 18161676 * 32 / 40 * 95,
                     "launches": 1, "tile_width": 8, "source_hash": "fb6051612007d295",
                     "note": "one launch over 40 fields of 1023^2 (cold caches under ncu), scaled to 95 fields"},
    # k_cols_scan: DRAM 167.7 MB read + 111.7 MB written, L2 10.99 M + 5.24 M sectors
    "tri_cols_f32": {"bytes_per_launch": 279393024 / 40 * 95, "l2_bytes_per_launch": 16229570 * 32 / 40 * 95,
                     "launches": 1, "tile_width": 8, "source_hash": "fb6051612007d295",
                     "note": "one launch over 40 fields of 1023^2 (cold caches under ncu), scaled to 95 fields"},
    # k_sine_rows_fwd (FP64 rows in, FP32 out): DRAM 335.3 MB read + 134.8 MB written, L2 15.07 M + 5.24 M sectors
    "dst_rows_fwd_f32": {"bytes_per_launch": 470086656 / 40 * 95, "l2_bytes_per_launch": 20304869 * 32 / 40 * 95,
                         "launches": 1, "tile_width": None, "source_hash": "fb6051612007d295",
                         "note": "one launch over 40 fields of 1023^2 (cold caches under ncu), scaled to 95 fields"},
    # k_sine_rows_inv (FP32 store, the form iim_time_box_passes times): DRAM 167.7 MB read + 120.5 MB written,
    # L2 8.71 M + 5.24 M sectors
    "dst_rows_inv_f32": {"bytes_per_launch": 288142080 / 40 * 95, "l2_bytes_per_launch": 13950553 * 32 / 40 * 95,
                         "launches": 1, "tile_width": None, "source_hash": "fb6051612007d295",
                         "note": "one launch over 40 fields of 1023^2 (cold caches under ncu), scaled to 95 fields"},
    # k_residual of a 1024^2 solve with one cylinder: DRAM 17.1 MB read (17 B per node), the 8 B per node it writes
    # still in L2; L2 0.93 M + 0.26 M sectors
    "residual_f64": {"bytes_per_launch": 17050624, "l2_bytes_per_launch": 1191620 * 32, "launches": 1,
                     "tile_width": None, "sources": ("iim_ops.cuh",), "source_hash": "e035dce4d191b813",
                     "note": "one launch on 1023^2 (cold caches under ncu)"},
}
TRANSFORM_SOURCES = ("dst.cuh", "sine.cuh", "tri.cuh")


L2_BYTES = 126 * 1024 * 1024
# kernel names of the three passes of iim_time_box_passes, per column pass (0 DSTs, 1 scans)
PASS_NAMES = {0: ("dst_rows_fwd_f32", "dst_cols_f32", "dst_rows_inv_f32"),
              1: ("dst_rows_fwd_f32", "tri_cols_f32", "dst_rows_inv_f32")}


def kernel_source_hash(files=TRANSFORM_SOURCES):
    """Hash of the files holding a captured kernel's code (the launch shape of a capture is recorded
    beside it: tile width, fields per launch)."""
    h = hashlib.sha256()
    for f in files:
        with open(os.path.join(ROOT, "paper_2109_13628_gb300", "csrc", f), "rb") as fh:
            h.update(fh.read())
    return h.hexdigest()[:16]


def parse():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=100)
    ap.add_argument("--warmup", type=int, default=5)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--n", type=int, default=N_CELLS)
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-e2e", action="store_true")
    ap.add_argument("--inner-rtol", type=float, default=0.0, help="mixed-mode Krylov tolerance (0: library default)")
    ap.add_argument("--restart", type=int, default=64)
    ap.add_argument("--sweep", action="store_true", help="print iterations/time for a grid of inner tolerances and exit")
    ap.add_argument("--no-precond", action="store_true", help="chosen form without the dense Schur preconditioner")
    ap.add_argument("--precond", type=int, default=3,
                    help="chosen form's iim_opts.precond: 1 dense inverse as right preconditioner of the transform "
                         "operator, 3 the same with the dense Schur matrix as the inner operator")
    ap.add_argument("--batch", type=int, default=8, help="independent problems in flight per step")
    ap.add_argument("--no-c4", action="store_true", help="skip the mixed-size batched workload")
    ap.add_argument("--c4-count", type=int, default=96)
    ap.add_argument("--no-learned", action="store_true", help="skip the learned-guess leg")
    ap.add_argument("--no-rk3", action="store_true", help="skip the RK3 step leg")
    ap.add_argument("--no-c3", action="store_true", help="skip the 2048^2 multi-body leg")
    ap.add_argument("--tiles", type=int, default=0, help="column-pass tile width (0: tuned on the batch)")
    ap.add_argument("--no-cufft", action="store_true", help="skip the cuFFT box-solve cross-check")
    ap.add_argument("--no-free", action="store_true", help="skip the free-space (unbounded) leg")
    ap.add_argument("--no-pressure", action="store_true", help="skip the total-pressure (Sec. 5.4) leg")
    ap.add_argument("--col-solver", type=int, default=-1,
                    help="column pass of the chosen form: 1 tridiagonal scans, 0 column DSTs, -1 tuned on the batch")
    return ap.parse_args()


def replica_totals(local_ms, local_units, device="cpu"):
    """Whole-job figures of independent replicas: (max over ranks of the timed milliseconds,
    sum over ranks of the units processed).  Without an initialised process group: the local
    figures."""
    import torch
    import torch.distributed as dist
    if not (dist.is_available() and dist.is_initialized()) or dist.get_world_size() == 1:
        return float(local_ms), float(local_units)
    t = torch.tensor([float(local_ms)], dtype=torch.float64, device=device)
    u = torch.tensor([float(local_units)], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    dist.all_reduce(u, op=dist.ReduceOp.SUM)
    return float(t.item()), float(u.item())


def dist_env():
    ws = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return ws, rank, local


class ClockSampler:
    """nvidia-smi clock / throttle samples while the timed region runs."""

    FIELDS = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, index):
        self.index = index
        self.proc = None
        out_dir = os.environ.get("IIM_CLOCKS_DIR") or tempfile.gettempdir()
        self.path = os.path.join(out_dir, f"iim_clocks_rank{index}.csv")

    def __enter__(self):
        try:
            os.makedirs(os.path.dirname(self.path), exist_ok=True)
            self.fh = open(self.path, "w")
            self.proc = subprocess.Popen(["nvidia-smi", f"--id={self.index}", f"--query-gpu={self.FIELDS}",
                                          "--format=csv,noheader,nounits", "-lms", "100"], stdout=self.fh,
                                         stderr=subprocess.DEVNULL)
        except Exception:
            self.proc = None
        return self

    def __exit__(self, *exc):
        if self.proc is not None:
            self.proc.terminate()
            try:
                self.proc.wait(timeout=5)
            except Exception:
                self.proc.kill()
            self.fh.close()

    def summary(self):
        if self.proc is None or not os.path.exists(self.path):
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["unavailable"]}
        sm, smax, reasons = [], [], set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for line in open(self.path):
            parts = [p.strip() for p in line.split(",")]
            if len(parts) < 9:
                continue
            try:
                sm.append(float(parts[1]))
                smax.append(float(parts[2]))
            except ValueError:
                continue
            for nm, v in zip(names, parts[5:9]):
                if v.lower() == "active":
                    reasons.add(nm)
        if not sm:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["no samples"]}
        return {"sm_mhz": statistics.median(sm), "sm_max_mhz": max(smax), "samples": len(sm),
                "reasons": sorted(reasons)}


def measured_peaks():
    try:
        with open(os.path.join(ROOT, "MEASURED_PEAKS.json")) as fh:
            return json.load(fh), "measured"
    except Exception:
        return {"hbm_gbs": 6800.0, "bf16_tflops": 1900.0}, "fallback"


_ORACLE_BARRIER = None


def _oracle_init(barrier):
    global _ORACLE_BARRIER
    _ORACLE_BARRIER = barrier
    for v in ("OMP_NUM_THREADS", "OPENBLAS_NUM_THREADS", "MKL_NUM_THREADS"):
        os.environ[v] = "1"


def _oracle_solves(task):
    """One host core: set up the workload, `warm` untimed oracle solves, wait for the other
    cores, then `reps` timed solves.  Returns (start, end, reps, GMRES iterations, residual)."""
    n, reps, warm = task
    import numpy as np

    from oracle import poisson as op
    from paper_2109_13628_gb300 import inputs
    P = inputs.c1_cylinder(n)
    S = op.Setup(P)
    O = op.SchurOperators(S)
    for _ in range(warm):
        op.solve_schur(S, psibar=np.zeros(1), tol=RTOL / 10, ops=O)
    if _ORACLE_BARRIER is not None:
        _ORACLE_BARRIER.wait(timeout=600)
    t0 = time.time()
    for _ in range(reps):
        psi, pb, it, rel = op.solve_schur(S, psibar=np.zeros(1), tol=RTOL / 10, ops=O)
    t1 = time.time()
    return t0, t1, reps, it, float(op.residual(S, psi, pb))


def oracle_throughput(n, reps, warm, cores=None):
    """The oracle as it stands (Schur-form GMRES, scipy DST-I, FP64, one thread per process) on
    `cores` host cores at once (default: every core this process may use), one independent
    solve stream per core in spawned processes, timed from the common start to the last end.
    Returns (solves/s, cores, GMRES iterations, worst residual, seconds)."""
    import multiprocessing as mp
    cores = cores or len(os.sched_getaffinity(0))
    ctx = mp.get_context("spawn")
    barrier = ctx.Barrier(cores)
    with ctx.Pool(cores, initializer=_oracle_init, initargs=(barrier,)) as pool:
        out = pool.map(_oracle_solves, [(n, reps, warm)] * cores)
    start, end = min(o[0] for o in out), max(o[1] for o in out)
    return sum(o[2] for o in out) / (end - start), cores, out[0][3], max(o[4] for o in out), end - start


def cpu_baseline(n, reps=8):
    v, cores, it, res, el = oracle_throughput(n, reps, 1)
    return {"value": v, "unit": UNIT, "cores": cores, "kind": "oracle",
            "sample": f"{cores} processes x {reps} oracle solves of the {n}^2 single-cylinder workload, one per host "
                      f"core (GMRES {it} iterations, residual {res:.2e}), geometry setup and one warm-up solve "
                      f"excluded, {el:.1f} s"}


def run_reference(args):
    ws, rank, _ = dist_env()
    if rank != 0:
        return
    steps = max(1, args.steps)
    v, cores, it, res, el = oracle_throughput(args.n, steps, args.warmup)
    line = {"impl": "reference", "metric": METRIC, "value": v, "unit": UNIT, "n_gpus": args.gpus,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": 1e3 * el / steps,
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
            "config": {"workload": WORKLOAD},
            "cpu_baseline": {"value": v, "unit": UNIT, "cores": cores, "kind": "oracle",
                             "sample": f"each step one full oracle solve on each of {cores} host cores at once "
                                       f"({it} GMRES iterations, FP64, scipy DST-I, residual {res:.2e})"},
            "e2e": {"value": v, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line))


def c4_batch(iim, inputs, T, dev, count, seed, precond):
    """The mixed-size batched workload: geometries, inputs, outputs (under-resolved draws skipped)."""
    import numpy as np
    import torch
    probs = inputs.batched_c4(count=count, seed=seed)
    geos, om, pb, gm, pbar, out, kept = [], [], [], [], [], [], []
    redraws = 0
    for k0, P in enumerate(probs):
        g = P.grid
        try:
            geo = iim.iim_setup_geometry(iim.make_grid(g.x0, g.x1, g.y0, g.y1, g.nx, g.ny), T(P.phi), P.regions, P.modes)
        except iim.IIMError:
            # under-resolved draw: another seeded draw of the same grid size takes its place
            geo = None
            for r in range(1, 50):
                P = inputs.ellipses_problem(g.nx, seed * 1000 + 100000 * r + k0)
                redraws += 1
                try:
                    geo = iim.iim_setup_geometry(iim.make_grid(g.x0, g.x1, g.y0, g.y1, g.nx, g.ny), T(P.phi),
                                                 P.regions, P.modes)
                    break
                except iim.IIMError:
                    continue
            if geo is None:
                continue
        cp = iim.iim_geometry_control_points(geo)
        geos.append(geo)
        kept.append(P)
        om.append(T(P.omega.ravel()))
        pb.append(T(np.zeros(geo.n_control)))
        h = g.h
        gm.append(T(np.array([h * h * P.omega[r[2] - 1:r[3], r[0] - 1:r[1]].sum() for r in P.regions])))
        pbar.append(torch.zeros(len(P.regions), dtype=torch.float64, device=dev))
        out.append(torch.empty(P.omega.size, dtype=torch.float64, device=dev))
        del cp
    t0 = time.perf_counter()
    if precond:
        # one-time per-geometry set-up, built concurrently on worker streams (ctypes releases the GIL)
        import concurrent.futures as cf
        order = sorted(range(len(geos)), key=lambda k: -kept[k].grid.nx)

        def build(ks):
            torch.cuda.set_device(dev)
            st = torch.cuda.Stream(device=dev)
            for k in ks:
                iim.iim_build_preconditioner(geos[k], stream=st)
            st.synchronize()

        nw = 8
        with cf.ThreadPoolExecutor(nw) as ex:
            list(ex.map(build, [order[w::nw] for w in range(nw)]))
    torch.cuda.synchronize()
    c4_batch.redraws = redraws
    return kept, geos, om, pb, gm, pbar, out, time.perf_counter() - t0


def learned_c5(iim, dev, opts_for, train_n=128, train_count=256, train_s=30.0, eval_n=1024, eval_count=4):
    """The learned initial guess: the net trained on the method's own solves (train_n^2, grid
    symmetries as augmentation, time-bounded), evaluated on unseen eval_n^2 geometries against
    the plain iteration (zero guess).  Guess time (body-free box solve, net input, forward,
    composition) counts against the learned solve."""
    import numpy as np
    import torch
    from paper_2109_13628_gb300 import learned
    t0 = time.perf_counter()
    data = learned.make_dataset(train_count, train_n, 1000, dev)
    t_data = time.perf_counter() - t0
    net = learned.Net(seed=5)
    t0 = time.perf_counter()
    losses = learned.train(net, data, epochs=1000, batch=8, lr=2e-3, time_budget_s=train_s)
    t_train = time.perf_counter() - t0
    del data
    rows, seed = [], 90000
    T = lambda a: torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device=dev)
    while len(rows) < eval_count and seed < 90000 + 8 * eval_count:
        P = learned.training_problem(eval_n, seed)
        seed += 1
        g = P.grid
        try:
            geo = iim.iim_setup_geometry(iim.make_grid(g.x0, g.x1, g.y0, g.y1, g.nx, g.ny), T(P.phi), P.regions,
                                         P.modes)
        except iim.IIMError:
            continue
        om, pb, gm = T(P.omega.ravel()), T(np.zeros(geo.n_control)), T(learned.gamma_of(P))
        phi_d = T(P.phi)
        out = torch.empty(P.omega.size, dtype=torch.float64, device=dev)
        pbar = torch.zeros(len(P.regions), dtype=torch.float64, device=dev)
        res = {}
        for tag in ("zero", "learned", "zero", "learned"):   # second pass timed (first warms graphs)
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            torch.cuda.synchronize()
            e0.record()
            guess = None
            if tag == "learned":
                S = learned.Sample(P, dev, omega=om, phi=phi_d, mask=False, box_prec=iim.IIM_MIXED)
                guess = S.guess(net, dev)
            st = iim.iim_poisson_solve(geo, om, pb, None, gm, pbar, out, psi_guess=guess,
                                       opts=iim.default_opts(prec=iim.IIM_MIXED, rtol=1e-10,
                                                             guess=0 if guess is None else 2))
            e1.record()
            torch.cuda.synchronize()
            res[tag] = (st["iters"], e0.elapsed_time(e1), st["seed_rel_res"], st["rel_res"], st["iters_first"])
        rows.append(res)
        geo.close()
    net.close()
    if not rows:
        return None
    # the net alone at the evaluation size: tensor-core and CUDA-core hidden layers
    fwd = {name: learned.time_forward(eval_n - 1, tensor_cores=tc)
           for name, tc in (("tensor_cores", 2), ("tensor_cores_hidden_only", 1), ("cuda_cores", 0))}
    mean = lambda tag, k: float(np.mean([r[tag][k] for r in rows]))
    return {"config": f"train {train_count} method solves at {train_n}^2 (random 2-5 circles/ellipses, Gaussian "
                      f"vortices; 8 grid symmetries), eval {len(rows)} unseen {eval_n}^2 geometries, mixed to 1e-10",
            "train_s": t_train, "dataset_s": t_data, "loss_first": losses[0],
            "loss_last": float(np.mean(losses[-10:])), "train_steps": len(losses),
            "zero_guess": {"krylov_iters": mean("zero", 0), "first_correction_iters": mean("zero", 4),
                           "ms_per_solve": mean("zero", 1),
                           "solves_per_s": 1e3 / mean("zero", 1)},
            "learned_guess": {"krylov_iters": mean("learned", 0), "first_correction_iters": mean("learned", 4),
                              "ms_per_solve": mean("learned", 1),
                              "solves_per_s": 1e3 / mean("learned", 1),
                              "seed_rel_res_mean": mean("learned", 2),
                              "max_rel_res": max(r["learned"][3] for r in rows)},
            "net_forward": {k: {"ms": v["forward_ms"], "kernels": v["kernels"]} for k, v in fwd.items()},
            "guess_path": "body-free box solve (FP32 transforms) of the device omega, net input, forward pass "
                          "(every layer on the tensor cores), composition; all inside the learned solve's events"}


def rk3_c2(iim, inputs, dev, steps=3):
    """One RK3 step of flow past a cylinder (1024 x 512, Re 200, CFL 0.5): the plain FP64 path
    and the mixed path, each timed over `steps` steps from the same initial state."""
    import numpy as np
    import torch
    P = inputs.c2_cylinder_flow(1024, 512)
    g = P.grid
    T = lambda a: torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device=dev)
    h = g.h
    lx, rx, ly, ry = P.regions[0]
    gam0 = np.array([h * h * P.omega[ly - 1:ry, lx - 1:rx].sum()])
    inside = np.zeros(P.omega.shape, dtype=bool)
    inside[ly - 1:ry, lx - 1:rx] = True
    ring = T(P.psi_box)
    w0d, g0d = T(P.omega.ravel()), T(gam0)
    out = {}
    # the geometry does not move, so its dense Schur preconditioner is built once for all steps
    geo = iim.iim_setup_geometry(iim.make_grid(g.x0, g.x1, g.y0, g.y1, g.nx, g.ny), T(P.phi), P.regions, P.modes)
    pc_ms = iim.iim_build_preconditioner(geo)
    for name, prec, pc in (("fp64", iim.IIM_FP64, 0), ("mixed", iim.IIM_MIXED, 0),
                           ("mixed_precond", iim.IIM_MIXED, 1), ("mixed_dense_op", iim.IIM_MIXED, 3)):
        w, gam, pbar = T(P.omega.ravel()), T(gam0), torch.zeros(1, dtype=torch.float64, device=dev)
        opts = iim.default_opts(prec=prec, rtol=1e-10, precond=pc)

        def step():
            w.copy_(w0d)
            gam.copy_(g0d)
            pbar.zero_()
            return iim.iim_rk3_step(geo, w, gam, pbar, None, None, ring, (1.0, 0.0), 0.005, 0.5, opts=opts)

        step()
        torch.cuda.synchronize()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        for _ in range(steps):
            dt, stats, _ = step()
        e1.record()
        torch.cuda.synchronize()
        w1 = w.cpu().numpy().reshape(P.omega.shape)
        kelvin = (gam.cpu().numpy().sum() + h * h * w1[~inside].sum()) - (gam0.sum() + h * h * P.omega[~inside].sum())
        out[name] = {"ms_per_step": e0.elapsed_time(e1) / steps, "dt": dt,
                     "krylov_iters_per_stage": [s["iters"] for s in stats],
                     "circ_err_max": max(s["circ_err_max"] for s in stats),
                     "kelvin_invariant_drift": float(abs(kelvin)), "omega": w1}
    w64, w32, wpc, wdo = (out[k].pop("omega") for k in ("fp64", "mixed", "mixed_precond", "mixed_dense_op"))
    geo.close()
    rel = lambda a: float(np.abs(a - w64).max() / np.abs(w64).max())
    return {"config": "flow past a cylinder R 0.5, [-2,6]x[-2,2], 1024 x 512, U 1, Re 200, CFL 0.5, noise 1e-3 seed 0",
            **out, "precond_setup_ms": pc_ms, "mixed_vs_fp64_rel_linf": rel(w32),
            "mixed_precond_vs_fp64_rel_linf": rel(wpc), "mixed_dense_op_vs_fp64_rel_linf": rel(wdo),
            "speedup_mixed_dense_op_vs_fp64": out["fp64"]["ms_per_step"] / out["mixed_dense_op"]["ms_per_step"],
            "speedup_mixed_vs_fp64": out["fp64"]["ms_per_step"] / out["mixed"]["ms_per_step"],
            "speedup_mixed_precond_vs_fp64": out["fp64"]["ms_per_step"] / out["mixed_precond"]["ms_per_step"],
            "kelvin_note": "box-wide invariant (Gamma + h^2 sum omega off the bodies' regions) also moves by the "
                           "vorticity flux through the box edges"}


def total_pressure_c2(iim, inputs, dev, flow_steps=30, steps=3):
    """The global surface-pressure method (Sec. 5.4) on the impulsively started cylinder of the
    1024 x 512 flow-past-a-cylinder workload: `flow_steps` RK3 steps from rest (mixed, dense
    Schur preconditioner), then the total-pressure problem -- right-hand side and Neumann wall
    datum from the flow, the IIM solve with the Neumann stencils on a second geometry of the same
    level set, surface values -- timed per call in FP64 and in the mixed forms."""
    import numpy as np
    import torch
    P = inputs.c2_cylinder_flow(1024, 512)
    g = P.grid
    T = lambda a: torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device=dev)
    mk = lambda modes: iim.iim_setup_geometry(iim.make_grid(g.x0, g.x1, g.y0, g.y1, g.nx, g.ny), T(P.phi), P.regions,
                                              modes)
    nu, U = 0.005, (1.0, 0.0)
    flow = mk(P.modes)
    iim.iim_build_preconditioner(flow)
    h = g.h
    lx, rx, ly, ry = P.regions[0]
    w = T(P.omega.ravel())
    gam = T([h * h * P.omega[ly - 1:ry, lx - 1:rx].sum()])
    pbar = torch.zeros(1, dtype=torch.float64, device=dev)
    ring = T(P.psi_box)
    fopts = iim.default_opts(prec=iim.IIM_MIXED, rtol=1e-10, precond=1)
    t = 0.0
    for _ in range(flow_steps):
        dt, _, _ = iim.iim_rk3_step(flow, w, gam, pbar, None, None, ring, U, nu, 0.5, opts=fopts)
        t += dt
    psi = torch.empty_like(w)
    ux, uy = torch.empty_like(w), torch.empty_like(w)
    iim.iim_poisson_solve(flow, w, torch.zeros(flow.n_control, dtype=torch.float64, device=dev), ring, gam, pbar, psi,
                          ux, uy, opts=fopts)
    flow.close()
    geo = mk([0])
    iim.iim_geometry_set_wall_condition(geo, 1)
    t0 = time.perf_counter()
    pc_ms = iim.iim_build_preconditioner(geo)
    t_pc = time.perf_counter() - t0
    H = torch.empty_like(w)
    Hw = torch.empty(geo.n_control, dtype=torch.float64, device=dev)
    out = {"config": f"impulsively started cylinder (R 0.5, U 1, Re 200) after {flow_steps} RK3 steps (t = {t:.4f}), "
                     f"1024 x 512, |C| = {geo.n_control}, |A| = {geo.n_affected}; H = 0 on the box",
           "precond_setup_s": t_pc, "precond_setup_gpu_ms": pc_ms}
    walls = {}
    for name, prec, pc in (("fp64", iim.IIM_FP64, 0), ("mixed", iim.IIM_MIXED, 0), ("mixed_precond", iim.IIM_MIXED, 1),
                           ("mixed_dense_op", iim.IIM_MIXED, 3)):
        opts = iim.default_opts(prec=prec, rtol=1e-10, precond=pc, max_iter=4000, max_refine=30)
        iim.iim_total_pressure(geo, w, ux, uy, U, nu, H, H_wall_out=Hw, opts=opts)
        torch.cuda.synchronize()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        for _ in range(steps):
            st = iim.iim_total_pressure(geo, w, ux, uy, U, nu, H, H_wall_out=Hw, opts=opts)
        e1.record()
        torch.cuda.synchronize()
        walls[name] = Hw.cpu().numpy().copy()
        out[name] = {"ms_per_call": e0.elapsed_time(e1) / steps, "krylov_iters": st["iters"],
                     "refinements": st["refinements"], "rel_res": st["rel_res"]}
    geo.close()
    ref = walls["fp64"]
    for k in ("mixed", "mixed_precond", "mixed_dense_op"):
        out[k]["wall_H_vs_fp64_max_abs"] = float(np.abs(walls[k] - ref).max())
    # static pressure coefficient on the wall, 2 (p - p_inf) / U^2 = 2 H / U^2 + 1
    cp = 2.0 * ref + 1.0
    out["wall_cp_range"] = [float(cp.min()), float(cp.max())]
    out["speedup_mixed_dense_op_vs_fp64"] = out["fp64"]["ms_per_call"] / out["mixed_dense_op"]["ms_per_call"]
    out["speedup_mixed_precond_vs_fp64"] = out["fp64"]["ms_per_call"] / out["mixed_precond"]["ms_per_call"]
    return out


PLAIN_INNER = (1e-10, 5e-11, 2e-11, 1e-11, 5e-12)


def calibrate_inner(solve_at, candidates, reps=2):
    """The Krylov tolerance (of `candidates`) whose solve reaches the FP64 residual target in
    the fewest milliseconds; each candidate is solved once untimed, then `reps` times under
    CUDA events.  Returns (tolerance, [per-candidate record])."""
    import torch
    rows, best = [], None
    for inner in candidates:
        solve_at(inner)
        torch.cuda.synchronize()
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        for _ in range(reps):
            st = solve_at(inner)
        b.record()
        torch.cuda.synchronize()
        ms = a.elapsed_time(b) / reps
        ok = st["rel_res"] <= RTOL
        rows.append({"inner_rtol": inner, "ms": ms, "krylov_iters": st["iters"], "refinements": st["refinements"],
                     "rel_res": st["rel_res"], "reaches_target": ok})
        if ok and (best is None or ms < best[1]):
            best = (inner, ms)
    return (best[0] if best else candidates[-1]), rows


def free_space_c43(iim, inputs, dev, n=1024, steps=3):
    """Free-space velocity reconstruction (Sec. 4.3's case: Lamb-Oseen vortex, two notched bodies
    in circulation mode, unbounded exterior) at n^2: mixed solve with the dense inner operator
    and the plain FP64 iteration, and the velocity error against the exact Lamb-Oseen field."""
    import numpy as np
    import torch
    c = inputs.FREE_SPACE_TWO_BODIES
    P = inputs.lamb_oseen_two_bodies(n)
    g = P.grid
    T = lambda a: torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device=dev)
    geo = iim.iim_setup_geometry(iim.make_grid(g.x0, g.x1, g.y0, g.y1, g.nx, g.ny), T(P.phi), P.regions, P.modes)
    t0 = time.perf_counter()
    iim.iim_geometry_set_outer(geo, 1)
    t_lgf = time.perf_counter() - t0
    cp = iim.iim_geometry_control_points(geo)
    pb = T(P.psi_b_fn(cp["x"].cpu().numpy(), cp["y"].cpu().numpy(), None))
    om, gam = T(P.omega.ravel()), T(P.gamma)
    psi = torch.empty(P.omega.size, dtype=torch.float64, device=dev)
    ux, uy = torch.empty_like(psi), torch.empty_like(psi)
    pbar = torch.zeros(2, dtype=torch.float64, device=dev)
    t0 = time.perf_counter()
    pc_ms = iim.iim_build_preconditioner(geo)
    t_pc = time.perf_counter() - t0
    X, Y = g.nodes()
    _, ex, ey = inputs.lamb_oseen(X, Y, c["x0"][0], c["x0"][1], c["gamma"], c["nu_t"])
    fl = (P.phi >= 0)[1:-1, 1:-1]
    out = {"config": f"Sec. 4.3 case in free space (unbounded exterior), {n}^2 cells, |A| = {geo.n_affected}",
           "lgf_table_and_buffers_s": t_lgf, "precond_setup_s": t_pc, "precond_setup_gpu_ms": pc_ms}
    # column pass per leg: FP64 on the tridiagonal scans (its fastest); mixed on both passes (in
    # free space their FP32 rounding changes the number of refinements)
    for name, prec, pc, col in (("fp64", iim.IIM_FP64, 0, 1), ("mixed_dense_op", iim.IIM_MIXED, 3, 0),
                                ("mixed_dense_op_tri", iim.IIM_MIXED, 3, 1)):
        iim.iim_geometry_set_column_solver(geo, col)
        opts = iim.default_opts(prec=prec, rtol=1e-10, precond=pc, max_iter=4000, max_refine=30)
        iim.iim_poisson_solve(geo, om, pb, None, gam, pbar, psi, ux, uy, opts=opts)
        torch.cuda.synchronize()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        for _ in range(steps):
            st = iim.iim_poisson_solve(geo, om, pb, None, gam, pbar, psi, ux, uy, opts=opts)
        e1.record()
        torch.cuda.synchronize()
        e = np.hypot(ux.cpu().numpy().reshape(P.omega.shape) - ex[1:-1, 1:-1],
                     uy.cpu().numpy().reshape(P.omega.shape) - ey[1:-1, 1:-1])[fl]
        out[name] = {"ms_per_solve": e0.elapsed_time(e1) / steps, "column_pass": ["column DSTs", "tridiagonal scans"][col],
                     "krylov_iters": st["iters"],
                     "refinements": st["refinements"], "rel_res": st["rel_res"], "circ_err_max": st["circ_err_max"],
                     "velocity_err_max": float(e.max()), "velocity_err_l2": float(np.sqrt((e * e).sum()) * g.h)}
    out["speedup_mixed_dense_op_vs_fp64"] = out["fp64"]["ms_per_solve"] / min(
        out["mixed_dense_op"]["ms_per_solve"], out["mixed_dense_op_tri"]["ms_per_solve"])
    geo.close()
    return out


def cufft_dst1(x, dim):
    """DST-I along `dim` by cuFFT (torch.fft): X_k = sum_j x_j sin(pi j k / n), j, k = 1..n-1,
    from the real FFT of the odd extension (0, x, 0, -x reversed) of length 2n, X_k = -Im Y_k / 2.
    The library's own transforms never call this: it is the timed library cross-check."""
    import torch
    n = x.shape[dim] + 1
    shape = list(x.shape)
    shape[dim] = 1
    z = torch.zeros(shape, dtype=x.dtype, device=x.device)
    y = torch.cat([z, x, z, -x.flip(dim)], dim)
    return torch.fft.rfft(y, dim=dim).imag.narrow(dim, 1, n - 1) * -0.5


def cufft_box_poisson(f, h):
    """Dirichlet-box solve -lap_h u = f (zero box data) on an (ny-1) x (nx-1) interior array by
    cuFFT DST-I along both axes, division by lam_x(k) + lam_y(l), lam(k) = (2 - 2 cos(pi k/n))/h^2,
    and the inverse DST-I (the same transform times 2/n per axis)."""
    import math
    import torch
    ny, nx = f.shape[0] + 1, f.shape[1] + 1
    kx = torch.arange(1, nx, dtype=torch.float64, device=f.device)
    ky = torch.arange(1, ny, dtype=torch.float64, device=f.device)
    lam = ((2 - 2 * torch.cos(math.pi * ky / ny))[:, None] + (2 - 2 * torch.cos(math.pi * kx / nx))[None, :]) / h**2
    scale = (2.0 / nx) * (2.0 / ny) / lam
    F = cufft_dst1(cufft_dst1(f, 1), 0) * scale.to(f.dtype)
    return cufft_dst1(cufft_dst1(F, 0), 1)


def gpu_ms_per_call(fn, reps, dev):
    """Device milliseconds per call of `fn`: the stream is first held by a sleep kernel long
    enough for the host to queue all `reps` calls, so the events bracket device time only."""
    import torch
    fn()
    torch.cuda.synchronize()
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    torch.cuda._sleep(int(2e8))   # ~0.1 s at 2 GHz
    a.record()
    for _ in range(reps):
        fn()
    b.record()
    torch.cuda.synchronize()
    return a.elapsed_time(b) / reps


def cufft_crosscheck(iim, dev, sizes=(1024, 2048), reps=20):
    """The library's DST-I box solve (FP64 and FP32 transforms) against a cuFFT-based box solve
    on the same seeded fields: agreement and device time per solve."""
    import numpy as np
    import torch
    out = {}
    for n in sizes:
        h = 4.0 / n
        g = iim.make_grid(-2, 2, -2, 2, n, n)
        NXY = (n - 1) ** 2
        rng = np.random.default_rng(n)
        f64 = torch.as_tensor(rng.normal(size=(n - 1, n - 1)), dtype=torch.float64, device=dev)
        f32 = f64.float()
        work = torch.empty(2 * NXY, dtype=torch.float64, device=dev)
        u = {p: torch.empty(NXY, dtype=torch.float64, device=dev) for p in (iim.IIM_FP64, iim.IIM_MIXED)}
        ref = cufft_box_poisson(f64, h)
        r32 = cufft_box_poisson(f32, h)
        fl = f64.reshape(-1)
        row = {}
        scale = ref.abs().max().item()
        for prec, tag in ((iim.IIM_FP64, "f64"), (iim.IIM_MIXED, "f32")):
            iim.iim_box_poisson(g, fl, None, u[prec], prec, work)
            torch.cuda.synchronize()
            err = (u[prec].reshape(n - 1, n - 1) - ref).abs().max().item() / scale
            ms = gpu_ms_per_call(lambda: iim.iim_box_poisson(g, fl, None, u[prec], prec, work), reps, dev)
            row[f"ours_{tag}"] = {"ms": ms, "rel_linf_vs_cufft_f64": err}
        row["cufft_f64"] = {"ms": gpu_ms_per_call(lambda: cufft_box_poisson(f64, h), reps, dev)}
        row["cufft_f32"] = {"ms": gpu_ms_per_call(lambda: cufft_box_poisson(f32, h), reps, dev),
                            "rel_linf_vs_cufft_f64": (r32.double() - ref).abs().max().item() / scale}
        xs = torch.zeros((n - 1, 2 * n), dtype=torch.float32, device=dev)
        row["cufft_f32_rfft_only"] = {"ms": 4 * gpu_ms_per_call(lambda: torch.fft.rfft(xs, dim=1), reps, dev),
                                      "note": "four batched real FFTs of 2n points over n-1 lines, no packing"}
        row["speedup_ours_f32_vs_cufft_f32"] = row["cufft_f32"]["ms"] / row["ours_f32"]["ms"]
        row["speedup_ours_f64_vs_cufft_f64"] = row["cufft_f64"]["ms"] / row["ours_f64"]["ms"]
        out[f"{n}x{n}"] = row
    out["note"] = ("cuFFT (through torch.fft) DST-I by the real FFT of the odd extension, zero box data; the "
                   "library's solve includes its box-data step; device time per solve with the host queued ahead")
    return out


def c3_multibody(iim, inputs, dev, steps=3):
    """The 2048^2 multi-body workload (three circles, an annulus, a five-petal star; 50 Gaussian
    vortices; circulation mode): plain FP64 solve and mixed solve to 1e-10, their difference,
    and the per-kernel profile of one mixed solve (a 2048^2 FP64 field is 32 MB, the solve's
    working set about 0.2 GB, beyond the 129 MB L2)."""
    import numpy as np
    import torch
    P = inputs.multibody(2048)
    g = P.grid
    T = lambda a: torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device=dev)
    geo = iim.iim_setup_geometry(iim.make_grid(g.x0, g.x1, g.y0, g.y1, g.nx, g.ny), T(P.phi), P.regions, P.modes)
    h = g.h
    gam = T([h * h * P.omega[r[2] - 1:r[3], r[0] - 1:r[1]].sum() for r in P.regions])
    om, pb = T(P.omega.ravel()), T(np.zeros(geo.n_control))
    out, res = {}, {}
    t0 = time.perf_counter()
    pc_ms = iim.iim_build_preconditioner(geo)
    out["precond_setup_s"] = time.perf_counter() - t0
    out["precond_setup_gpu_ms"] = pc_ms
    for name, prec, pc in (("fp64", iim.IIM_FP64, 0), ("mixed", iim.IIM_MIXED, 0),
                           ("mixed_precond", iim.IIM_MIXED, 1), ("mixed_dense_op", iim.IIM_MIXED, 3)):
        psi = torch.empty(P.omega.size, dtype=torch.float64, device=dev)
        pbar = torch.zeros(len(P.regions), dtype=torch.float64, device=dev)
        opts = iim.default_opts(prec=prec, rtol=1e-10, max_iter=4000, precond=pc)
        iim.iim_poisson_solve(geo, om, pb, None, gam, pbar, psi, opts=opts)
        torch.cuda.synchronize()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        for _ in range(steps):
            st = iim.iim_poisson_solve(geo, om, pb, None, gam, pbar, psi, opts=opts)
        e1.record()
        torch.cuda.synchronize()
        res[name] = psi
        out[name] = {"ms_per_solve": e0.elapsed_time(e1) / steps, "krylov_iters": st["iters"],
                     "refinements": st["refinements"], "rel_res": st["rel_res"], "circ_err_max": st["circ_err_max"]}
    for k in ("mixed", "mixed_precond", "mixed_dense_op"):
        out[f"{k}_vs_fp64_rel_linf"] = float((res[k] - res["fp64"]).abs().max() / res["fp64"].abs().max())
        out[f"speedup_{k}_vs_fp64"] = out["fp64"]["ms_per_solve"] / out[k]["ms_per_solve"]
    iim.iim_profile_begin()
    psi = torch.empty(P.omega.size, dtype=torch.float64, device=dev)
    pbar = torch.zeros(len(P.regions), dtype=torch.float64, device=dev)
    torch.cuda.nvtx.range_push("profile_c3")
    iim.iim_poisson_solve(geo, om, pb, None, gam, pbar, psi, opts=iim.default_opts(prec=iim.IIM_MIXED, rtol=1e-10,
                                                                                    max_iter=4000))
    torch.cuda.synchronize()
    torch.cuda.nvtx.range_pop()
    kern = sorted(iim.iim_profile_end(), key=lambda r: -r["ms"])
    tot = sum(r["ms"] for r in kern)
    peaks, src = measured_peaks()
    mem = [r for r in kern if r["bytes"] > 0]
    if mem:
        d = mem[0]
        us = d["ms"] * 1e3 / d["launches"]
        ach = d["bytes"] / d["launches"] / (us * 1e-6) / 1e9
        out["roofline"] = {"bound": "hbm", "kernel": d["name"], "achieved": ach, "peak": peaks["hbm_gbs"],
                           "unit": "GB/s", "frac": ach / peaks["hbm_gbs"], "peak_source": src,
                           "alg_bytes_per_launch": d["bytes"] / d["launches"], "avg_launch_us": us,
                           "share_of_kernel_time": d["ms"] / tot if tot else None}
    out["kernels"] = [{"name": r["name"], "launches": r["launches"], "ms": r["ms"], "share": r["ms"] / tot if tot else None}
                      for r in kern[:6]]
    out["config"] = ("multibody_2048: [-4,4]^2, 2048^2 cells, 3 circles R~U(0.3,0.6), annulus 0.4/0.8, star "
                     "r = 0.5 + 0.15 cos 5 theta; 50 Gaussian vortices sigma 0.1; circulation mode; "
                     f"|A| = {geo.n_affected}, |C| = {geo.n_control}")
    geo.close()
    return out


def main():
    args = parse()
    if args.impl == "reference":
        run_reference(args)
        return
    import numpy as np
    import torch

    ws, rank, local = dist_env()
    if ws > 1:
        import torch.distributed as dist
        torch.cuda.set_device(local)
        dist.init_process_group("nccl")
    dev = torch.device("cuda", local)
    torch.cuda.set_device(dev)
    import paper_2109_13628_gb300 as iim
    from paper_2109_13628_gb300 import autotune, inputs

    P = inputs.c1_cylinder(args.n)
    g = P.grid
    T = lambda a: torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device=dev)
    grid = iim.make_grid(g.x0, g.x1, g.y0, g.y1, g.nx, g.ny)
    precond = 0 if args.no_precond else args.precond
    NXY = (g.nx - 1) * (g.ny - 1)
    B = max(1, args.batch)
    # B independent problems (each its own geometry workspace) on the same cylinder workload
    t_setup = time.perf_counter()
    geos = [iim.iim_setup_geometry(grid, T(P.phi), P.regions, P.modes) for _ in range(B)]
    t_setup = (time.perf_counter() - t_setup) / B
    col_mode, col_tuned = (args.col_solver if args.col_solver >= 0 else 1), None
    for gg in geos:
        iim.iim_geometry_set_column_solver(gg, col_mode)
    cp = iim.iim_geometry_control_points(geos[0])
    psi_b_h = P.psi_b_fn(cp["x"].cpu().numpy(), cp["y"].cpu().numpy(), None)
    omega, psi_b, ring = T(P.omega.ravel()), T(psi_b_h), T(P.psi_box)
    psibars = [torch.zeros(1, dtype=torch.float64, device=dev) for _ in range(B)]
    psis = [torch.empty(NXY, dtype=torch.float64, device=dev) for _ in range(B)]
    uxs = [torch.empty(NXY, dtype=torch.float64, device=dev) for _ in range(B)]
    uys = [torch.empty(NXY, dtype=torch.float64, device=dev) for _ in range(B)]
    t_pc = time.perf_counter()
    pc_ms = [iim.iim_build_preconditioner(geo) if precond else 0.0 for geo in geos][0]
    t_pc = (time.perf_counter() - t_pc) / B
    flush = torch.empty(64 * 1024 * 1024, dtype=torch.float32, device=dev)   # 256 MiB > L2
    stream = torch.cuda.current_stream()
    geo = geos[0]

    def opts_for(prec, inner=None, pc=None):
        use_pc = (precond if prec == iim.IIM_MIXED else 0) if pc is None else pc
        return iim.default_opts(prec=prec, rtol=RTOL, restart=args.restart, precond=use_pc,
                                inner_rtol=args.inner_rtol if inner is None else inner)

    def solve(prec, inner=None, pc=None, on=None):
        # the plain FP64 comparator is the unpreconditioned paper iteration
        return iim.iim_poisson_solve(geo if on is None else on, omega, psi_b, ring, None, psibars[0], psis[0], uxs[0],
                                     uys[0], opts=opts_for(prec, inner, pc))

    def solve_batch(n_streams):
        return iim.iim_poisson_solve_batched(geos, [omega] * B, [psi_b] * B, [ring] * B, None, psibars, psis, uxs, uys,
                                             opts=opts_for(iim.IIM_MIXED), n_streams=n_streams)

    if args.sweep:
        for prec, pc in ((iim.IIM_MIXED, 3), (iim.IIM_MIXED, 1), (iim.IIM_FP64, 3), (iim.IIM_FP64, 1),
                         (iim.IIM_MIXED, 0), (iim.IIM_FP64, 0)):
            if pc and not precond:
                continue
            for inner in ((1e-3, 1e-4, 1e-5, 1e-6, 3e-7) if prec == iim.IIM_MIXED else (5e-12, 5e-11)):
                for _ in range(2):
                    solve(prec, inner, pc)
                torch.cuda.synchronize()
                t0 = time.perf_counter()
                for _ in range(5):
                    st = solve(prec, inner, pc)
                torch.cuda.synchronize()
                print(json.dumps({"prec": prec, "precond": pc, "inner": inner,
                                  "ms": (time.perf_counter() - t0) / 5 * 1e3, "iters": st["iters"],
                                  "refinements": st["refinements"], "rel_res": st["rel_res"]}))
        return

    window = {}   # library launches before / inside the last timed region

    def timed(step, k, warm, nvtx="timed"):
        for _ in range(warm):
            step()
        torch.cuda.synchronize()
        if ws > 1:
            torch.distributed.barrier()
        torch.cuda.synchronize()
        ms, outs = [], []
        window["before"] = iim.iim_launch_count()
        torch.cuda.nvtx.range_push(nvtx)   # lets a profiler select the timed launches
        for _ in range(k):
            flush.zero_()
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record(stream)
            outs.append(step())
            b.record(stream)
            b.synchronize()
            ms.append(a.elapsed_time(b))
        torch.cuda.synchronize()
        torch.cuda.nvtx.range_pop()
        window["timed"] = iim.iim_launch_count() - window["before"]
        if ws > 1:
            torch.distributed.barrier()
        return ms, outs


    # ---- concurrency autotuning of the batched form (untimed)
    n_streams = B
    tuned = None
    tile_w, tiles_tuned = 4, None
    if args.tiles:
        tile_w = args.tiles
        for gg in geos:
            iim.iim_geometry_set_tiles(gg, tile_w)
    group, group_tuned = 1, None
    if B > 1:
        # the per-problem form's tile width and streams, then the lockstep group size
        prev = iim.iim_set_lockstep(0)
        if args.col_solver < 0:
            col_mode, col_tuned = autotune.tune_column_solver(geos, lambda: solve_batch(B), rebuild_precond=bool(precond))
        if not args.tiles:
            tile_w, tiles_tuned = autotune.tune_tiles_batch(geos, lambda: solve_batch(B))
        n_streams, tuned = autotune.tune_streams(solve_batch, tuple(c for c in (1, 2, 4, 8, 12, 16) if c <= B))
        iim.iim_set_lockstep(prev)
        group, group_tuned = autotune.tune_lockstep(lambda: solve_batch(n_streams),
                                                    tuple(c for c in (1, 2, 4, 8) if c <= B))
    # ---- chosen form: B problems per step in flight (the timed region), clocks sampled
    with ClockSampler(local) as clk:
        ms, outs = timed(lambda: solve_batch(n_streams)[1] if B > 1 else [solve(iim.IIM_MIXED)], args.steps,
                         args.warmup, nvtx="value")
        launches = window["timed"]
        launch_window = dict(window)
    stats = [s for step_stats in outs for s in step_stats]
    total_ms, total_solves = replica_totals(sum(ms), B * args.steps, dev)
    value = total_solves / (total_ms * 1e-3)
    # ---- the same form one problem at a time (latency view)
    ms1, outs1 = timed(lambda: solve(iim.IIM_MIXED), args.steps, 2)
    single = args.steps / (sum(ms1) * 1e-3)
    # ---- plain FP64 iteration (the comparator: unpreconditioned, one problem at a time), at its
    # loosest Krylov tolerance that still ends at the same FP64 residual target (no over-solve)
    # (FP64 legs on a geometry of their own with their fastest column pass, the tridiagonal scans)
    geo64 = iim.iim_setup_geometry(grid, T(P.phi), P.regions, P.modes)
    iim.iim_geometry_set_column_solver(geo64, 1)
    inner64, calib64 = calibrate_inner(lambda inner: solve(iim.IIM_FP64, inner, 0, geo64), PLAIN_INNER)
    k64 = max(3, args.steps // 5)
    ms64, stats64 = timed(lambda: solve(iim.IIM_FP64, inner64, 0, geo64), k64, 2)
    plain = k64 / (sum(ms64) * 1e-3)
    # ---- FP64 transforms with the same dense preconditioner (isolates the mixed-precision gain)
    inner64p, calib64p = (None, None)
    fp64_pc = None
    if precond:
        iim.iim_build_preconditioner(geo64)
        inner64p, calib64p = calibrate_inner(lambda inner: solve(iim.IIM_FP64, inner, 1, geo64), PLAIN_INNER)
        msp, statsp = timed(lambda: solve(iim.IIM_FP64, inner64p, 1, geo64), k64, 2)
        fp64_pc = {"value": k64 / (sum(msp) * 1e-3), "unit": UNIT, "ms_per_solve": sum(msp) / k64,
                   "inner_rtol": inner64p, "krylov_iters": statistics.mean(s["iters"] for s in statsp),
                   "refinements": statistics.mean(s["refinements"] for s in statsp),
                   "final_rel_res": max(s["rel_res"] for s in statsp), "calibration": calib64p}
    geo64.close()
    # ---- lockstep off: one whole-solve graph per problem on the tuned streams (same B solves)
    per_problem = None
    if B > 1:
        prev = iim.iim_set_lockstep(0)
        kpp = max(3, args.steps // 2)
        mpp, _ = timed(lambda: solve_batch(n_streams)[1], kpp, 2)
        iim.iim_set_lockstep(prev)
        per_problem = {"value": B * kpp / (sum(mpp) * 1e-3), "unit": UNIT, "ms_per_step": sum(mpp) / kpp,
                       "streams": n_streams,
                       "form": "lockstep off: one whole-solve graph per problem, problems overlapping on streams"}

    def kernel_profile(step, k):
        iim.iim_profile_begin()
        torch.cuda.nvtx.range_push("profile")   # every launch direct (host-driven), no graphs
        for _ in range(k):
            flush.zero_()
            step()
        torch.cuda.synchronize()
        torch.cuda.nvtx.range_pop()
        kern = iim.iim_profile_end()
        kern.sort(key=lambda r: -r["ms"])
        return kern, sum(r["ms"] for r in kern)

    # ---- per-kernel timing of the timed form: with lockstep groups, the group's kernels run
    # host-driven under the per-kernel profiler (CUDA events around each launch on its stream,
    # each launch carrying the algorithmic bytes of the whole group); with one whole-solve graph
    # per problem, the same solve's kernels one problem at a time
    kprof = min(args.steps, 10)
    kern, tot_k = kernel_profile(lambda: solve_batch(n_streams) if group > 1 else solve(iim.IIM_MIXED), kprof)
    kern1, tot_k1 = kernel_profile(lambda: solve(iim.IIM_MIXED), kprof)
    peaks, src = measured_peaks()
    mem = [r for r in kern if r["bytes"] > 0]
    dom = mem[0] if mem else None
    # ---- the transform passes of this grid timed alone (iim_time_box_passes: each pass launched
    # back to back inside a CUDA graph, CUDA events around the graph): one field (L2-resident),
    # the B fields of a step in one launch, and enough fields that the working set exceeds L2
    big = max(B, int(math.ceil(3 * L2_BYTES / (4.0 * NXY))))
    passes = {}
    for label, nb in (("single", 1), (f"batch_{B}", B), (f"batch_{big}_beyond_l2", big)):
        r = iim.iim_time_box_passes(geo, iim.IIM_MIXED, nb, 10)
        passes[label] = {k: {"us_per_launch": u, "alg_bytes_per_launch": b, "gbs": b / u / 1e3,
                             "frac_of_hbm": b / u / 1e3 / peaks["hbm_gbs"]}
                         for k, u, b in zip(PASS_NAMES[col_mode], r["us"], r["bytes"])}
    roof = None
    if dom:
        per_launch_s = dom["ms"] * 1e-3 / dom["launches"]
        ev_achieved = dom["bytes"] / dom["launches"] / per_launch_s / 1e9
        tr = NCU_TRAFFIC.get(dom["name"])
        valid = (bool(tr) and tr["source_hash"] == kernel_source_hash(tr.get("sources", TRANSFORM_SOURCES))
                 and tr.get("tile_width") in (None, tile_w))   # the tile width matters for the column pass only
        traffic = tr["bytes_per_launch"] if valid else None
        l2_traffic = tr.get("l2_bytes_per_launch") if valid else None
        alone = passes[f"batch_{big}_beyond_l2"].get(dom["name"])
        achieved = alone["gbs"] if alone else ev_achieved
        roof = {"bound": "hbm", "kernel": dom["name"], "achieved": achieved, "peak": peaks["hbm_gbs"], "unit": "GB/s",
                "frac": achieved / peaks["hbm_gbs"], "traffic": traffic, "l2_traffic": l2_traffic, "peak_source": src,
                "alg_bytes_per_launch": alone["alg_bytes_per_launch"] if alone else dom["bytes"] / dom["launches"],
                "avg_launch_us": alone["us_per_launch"] if alone else per_launch_s * 1e6,
                "share_of_kernel_time": dom["ms"] / tot_k if tot_k else None,
                "event_profile": {"achieved": ev_achieved, "avg_launch_us": per_launch_s * 1e6,
                                  "alg_bytes_per_launch": dom["bytes"] / dom["launches"]},
                "timing": ((f"the dominant kernel by share of the timed form's per-kernel profile, timed alone on "
                            f"this grid: {big} fields per launch (working set beyond L2), launches back to back in a "
                            "CUDA graph, CUDA events around the graph launch on its stream" if alone else
                            "per-kernel profile of the timed form (CUDA events around each launch on its stream)") +
                           "; event_profile: the same kernel in the timed form's per-kernel profile, host-driven "
                           "launches (includes host gaps between launches)")}
    # ---- end to end through the C ABI with host buffers (B problems per step)
    e2e = None
    if not args.no_e2e:
        h_omega = torch.from_numpy(np.ascontiguousarray(P.omega).ravel()).pin_memory()
        h_psib = torch.from_numpy(np.ascontiguousarray(psi_b_h)).pin_memory()
        h_ring = torch.from_numpy(np.ascontiguousarray(P.psi_box)).pin_memory()
        h_out = [[torch.empty(NXY, dtype=torch.float64).pin_memory() for _ in range(3)] for _ in range(B)]
        d_in = [(torch.empty_like(omega), torch.empty_like(psi_b), torch.empty_like(ring)) for _ in range(B)]

        h_pbar = [torch.zeros(1, dtype=torch.float64).pin_memory() for _ in range(B)]

        e2e_streams = {"n": n_streams}

        def e2e_step():
            if B > 1:
                # host buffers straight through the C ABI: per-problem copies overlap other solves
                iim.iim_poisson_solve_batched_host(geos, [h_omega] * B, [h_psib] * B, [h_ring] * B, None, h_pbar,
                                                   [h[0] for h in h_out], [h[1] for h in h_out],
                                                   [h[2] for h in h_out], opts=opts_for(iim.IIM_MIXED),
                                                   n_streams=e2e_streams["n"])
                return
            for d in d_in:
                d[0].copy_(h_omega, non_blocking=True)
                d[1].copy_(h_psib, non_blocking=True)
                d[2].copy_(h_ring, non_blocking=True)
            iim.iim_poisson_solve(geo, d_in[0][0], d_in[0][1], d_in[0][2], None, psibars[0], psis[0], uxs[0],
                                  uys[0], opts=opts_for(iim.IIM_MIXED))
            for k in range(B):
                for h, d in zip(h_out[k], (psis[k], uxs[k], uys[k])):
                    h.copy_(d, non_blocking=True)

        e2e_tuning = None
        if B > 1:
            # the stream count for host buffers: fewer streams stagger the problems, so that the
            # outputs of early ones cross to the host while later ones compute
            e2e_step()
            best, e2e_tuning = autotune.tune_streams(
                lambda c: (e2e_streams.__setitem__("n", c), e2e_step()), tuple(c for c in (2, 4, 8) if c <= B))
            e2e_streams["n"] = best
        ems, _ = timed(e2e_step, args.steps, args.warmup)
        e_total, e_solves = replica_totals(sum(ems), B * args.steps, dev)
        e2e = {"value": e_solves / (e_total * 1e-3), "unit": UNIT, "streams": e2e_streams["n"],
               "streams_tuning_ms": e2e_tuning,
               "h2d_bytes_per_step": B * 8 * (NXY + psi_b.numel() + ring.numel()), "d2h_bytes_per_step": B * 8 * 3 * NXY,
               "path": "inputs copied from pinned host memory per problem stream; psi, u_x, u_y written into the "
                       "pinned host arrays by each solve's last kernel (B > 1) or copied back (B = 1)"}
    # ---- mixed-size batched workload (96 problems, 128^2 .. 1024^2)
    c4 = None
    if not args.no_c4:
        kept, cgeos, om, pbv, gm, pbar, cout, c4_pc = c4_batch(iim, inputs, T, dev, args.c4_count, 2, precond)
        tiles = autotune.tune_tiles(cgeos, lambda k: iim.iim_poisson_solve(
            cgeos[k], om[k], pbv[k], None, gm[k], pbar[k], cout[k], opts=opts_for(iim.IIM_MIXED)))

        def c4_run(nst):
            return iim.iim_poisson_solve_batched(cgeos, om, pbv, None, gm, pbar, cout, opts=opts_for(iim.IIM_MIXED),
                                                 n_streams=nst)

        prev_group = iim.iim_set_lockstep(0)
        c4_col, c4_col_tuned = autotune.tune_column_solver(cgeos, lambda: c4_run(8), rebuild_precond=bool(precond))
        c4_streams, c4_tuned = autotune.tune_streams(c4_run, (4, 8, 16, 24))
        iim.iim_set_lockstep(prev_group)
        c4_group, c4_group_tuned = autotune.tune_lockstep(lambda: c4_run(c4_streams), (1, 4, 8, 24), reps=1)
        cms, couts = timed(lambda: c4_run(c4_streams)[1], max(2, args.steps // 10), 1)
        unknowns = sum((P.grid.nx - 1) * (P.grid.ny - 1) for P in kept)
        c4 = {"problems": len(kept), "redrawn_underresolved": getattr(c4_batch, "redraws", 0), "solves_per_s": len(kept) * len(cms) / (sum(cms) * 1e-3),
              "unknown_solves_per_s": unknowns * len(cms) / (sum(cms) * 1e-3), "ms_per_batch": sum(cms) / len(cms),
              "streams": c4_streams, "lockstep_group": c4_group, "lockstep_tuning_ms": c4_group_tuned,
              "tiles_by_size": {f"{k[0]}x{k[1]}": v for k, v in tiles.items()},
              "column_pass": ["column DSTs", "tridiagonal scans"][c4_col], "column_pass_tuning_ms": c4_col_tuned,
              "precond_setup_s": c4_pc, "max_rel_res": max(s["rel_res"] for o in couts for s in o),
              "krylov_iters_mean": statistics.mean(s["iters"] for o in couts for s in o)}
        # the same batch with FP64 transforms throughout (same preconditioner and streams)
        def c4_run64():
            return iim.iim_poisson_solve_batched(cgeos, om, pbv, None, gm, pbar, cout,
                                                 opts=opts_for(iim.IIM_FP64, pc=precond), n_streams=c4_streams)

        for gg in cgeos:   # FP64 on its fastest column pass, the tridiagonal scans
            iim.iim_geometry_set_column_solver(gg, 1)
        c4_run64()
        fms, fouts = timed(lambda: c4_run64()[1], 2, 0)
        c4["fp64"] = {"solves_per_s": len(kept) * len(fms) / (sum(fms) * 1e-3), "ms_per_batch": sum(fms) / len(fms),
                      "max_rel_res": max(s["rel_res"] for o in fouts for s in o),
                      "krylov_iters_mean": statistics.mean(s["iters"] for o in fouts for s in o)}
        c4["mixed_vs_fp64_speedup"] = c4["fp64"]["ms_per_batch"] / c4["ms_per_batch"]
        for gg in cgeos:
            gg.close()
    rk3 = None if args.no_rk3 else rk3_c2(iim, inputs, dev)
    c3 = None if args.no_c3 else c3_multibody(iim, inputs, dev)
    cufft = None if args.no_cufft else cufft_crosscheck(iim, dev)
    free = None if args.no_free else free_space_c43(iim, inputs, dev)
    pressure = None if args.no_pressure else total_pressure_c2(iim, inputs, dev)
    c5 = None
    if not args.no_learned:
        c5 = learned_c5(iim, dev, opts_for)
    cpu = None
    if rank == 0 and ws == 1 and not args.no_cpu_baseline:
        cpu = cpu_baseline(args.n)
    line = {
        "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": ws, "steps": args.steps, "warmup": args.warmup,
        "ms_per_step": total_ms / args.steps, "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
        "dtype": "f32 transforms + f64 refinement", "data": "synthetic",
        "config": {"workload": WORKLOAD, "batch": (f"{B} independent problems of this workload per step in "
                                                   f"lockstep groups of {group} (one kernel launch per solve step for "
                                                   "a whole group, one CUDA graph per group, groups concurrent)"
                                                   if group > 1 else
                                                   f"{B} independent problems of this workload per step, one "
                                                   f"whole-solve graph each, in flight on {n_streams} streams"),
                   "l2": "flushed before every timed step (256 MiB write, outside the events)",
                   "form": ("mixed: FP32 DST-I box solves inside FP64 iterative refinement, GMRES("
                            f"{args.restart}) FP64 Krylov" + (", right-preconditioned by the dense FP32 inverse of the"
                                                             " Schur matrix" if precond else "") +
                            (", inner operator the dense FP32 Schur matrix (transforms for each correction's "
                             "right-hand side and recovery)" if precond == 3 else "")),
                   "parallelism": f"replicas x{ws}"},
        "single_problem": {"value": single, "unit": UNIT, "ms_per_solve": sum(ms1) / len(ms1)},
        "plain_fp64": {"value": plain, "unit": UNIT, "ms_per_step": sum(ms64) / k64, "column_pass": "tridiagonal scans",
                       "krylov_iters": statistics.mean(s["iters"] for s in stats64),
                       "refinements": statistics.mean(s["refinements"] for s in stats64),
                       "final_rel_res": max(s["rel_res"] for s in stats64), "inner_rtol": inner64,
                       "calibration": calib64,
                       "rule": "the paper's iteration (FP64 transforms, unpreconditioned GMRES), stopped as soon as "
                               "the un-reduced FP64 residual is <= 1e-10, at the loosest Krylov tolerance of "
                               f"{list(PLAIN_INNER)} that reaches it in the fewest milliseconds"},
        "fp64_precond": fp64_pc,
        "speedup_vs_plain_fp64": value / plain / ws,
        "speedup_single_vs_plain_fp64": single / plain,
        "solver": {"krylov_iters": statistics.mean(s["iters"] for s in stats),
                   "refinements": statistics.mean(s["refinements"] for s in stats),
                   "final_rel_res_max": max(s["rel_res"] for s in stats), "setup_s": t_setup,
                   "precond_setup_s": t_pc, "precond_setup_gpu_ms": pc_ms, "streams_tuning_ms": tuned,
                   "column_pass": "tridiagonal scans" if col_mode == 1 else "column DSTs",
                   "column_pass_tuning_ms": col_tuned,
                   "tile_width": tile_w, "tile_tuning_ms": tiles_tuned, "lockstep_group": group,
                   "lockstep_tuning_ms": group_tuned,
                   "n_control": geo.n_control, "n_affected": geo.n_affected},
        "roofline": roof,
        "transform_passes": passes,
        "kernels": [{"name": r["name"], "launches_per_step": r["launches"] / kprof, "ms_per_step": r["ms"] / kprof,
                     "share": r["ms"] / tot_k if tot_k else None} for r in kern[:12]],
        "kernels_single_problem": [{"name": r["name"], "launches_per_solve": r["launches"] / kprof,
                                    "ms_per_solve": r["ms"] / kprof, "share": r["ms"] / tot_k1 if tot_k1 else None}
                                   for r in kern1[:8]],
        "per_problem_graphs": per_problem,
        "gpu_launches": launches,
        "launch_window": {"library_launches_before_timed": launch_window["before"],
                          "library_launches_timed": launch_window["timed"]},
        "clocks": clk.summary(),
        "e2e": e2e,
        "batched_c4": c4,
        "learned_c5": c5,
        "rk3_c2": rk3,
        "multibody_c3": c3,
        "cufft_crosscheck": cufft,
        "free_space_c43": free,
        "total_pressure_c2": pressure,
        "cpu_baseline": cpu,
    }
    if rank == 0:
        print(json.dumps(line))
    for gg in geos:
        gg.close()
    if ws > 1:
        torch.distributed.destroy_process_group()


if __name__ == "__main__":
    main()
