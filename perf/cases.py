"""Timed cases of the library's public entry points.

A case is one call (or one batch of calls) that a program using the library makes again and again:
a rectangular solve, an immersed-interface solve alone or in a batch, a Runge-Kutta step, the
transport right-hand side, the learned guess's network.  The immersed-interface solves use
streamfunctions for which the discrete equations hold exactly -- a polynomial of degree three in
each variable around the bodies plus Gaussian vortices that vanish within a few cells of every
body -- so that the result is known at every node."""
import math
import random

import torch

import paper_2109_13628_gb300 as iim
from paper_2109_13628_gb300.learned import DILATIONS, HIDDEN, IN_CHANNELS, Net

F64 = torch.float64


def listed():
    return [
        # the smallest call: one Dirichlet-box solve, where launches and latency are all there is
        dict(name="box_64_fp64", kind="box", nx=64, ny=64, prec="fp64", ring=True),
        # one small flow of a parameter sweep: two bodies at the coarsest grid of the batched workload
        dict(name="solve_128_mixed", kind="solve", nx=128, ny=128, bodies=2, prec="mixed", precond=1),
        # the library's default form (plain FP64 iteration) on a medium grid with three bodies
        dict(name="solve_512_fp64", kind="solve", nx=512, ny=512, bodies=3, prec="fp64", precond=0),
        # one solve at a time on the benchmark's grid: latency of the chosen form
        dict(name="solve_1024_dense", kind="solve", nx=1024, ny=1024, bodies=1, prec="mixed", precond=3),
        # the benchmark's throughput form: eight of them in flight, one graph each
        dict(name="batch_8x1024", kind="batch", count=8, lo=1024, hi=1024, lockstep=1, precond=3),
        # a batch of mixed sizes in lockstep groups (the library's default group size)
        dict(name="batch_15_mixed_sizes", kind="batch", count=15, lo=128, hi=1024, lockstep=4, precond=3),
        # the largest grid: five bodies (an annulus and a star among them)
        dict(name="multibody_2048", kind="solve", nx=2048, ny=2048, bodies=5, prec="mixed", precond=1),
        # unbounded domain around two bodies
        dict(name="free_space_512", kind="free", n=512, bodies=2, precond=3),
        # one time step of flow past a cylinder (three solves and three transport evaluations)
        dict(name="rk3_1024x512", kind="rk3", nx=1024, ny=512, precond=3),
        # the transport right-hand side alone, wall vorticity from the velocity
        dict(name="transport_1024x512", kind="transport", nx=1024, ny=512, bodies=1),
        # inference of the learned guess on the benchmark's grid
        dict(name="net_forward_1023", kind="net_forward", batch=1, h=1023, w=1023),
        # one training step of it on a batch of 128^2 grids
        dict(name="net_train_8x127", kind="net_train", batch=8, h=127, w=127),
    ]


def _log_pick(rng, lo, hi):
    return 2 ** rng.randint(int(math.log2(lo)), int(math.log2(hi)))


def draw(rng):
    kind = rng.choice(["box", "box", "solve", "solve", "solve", "batch", "batch", "free", "rk3", "transport",
                       "transport", "net_forward", "net_train"])
    if kind == "box":
        return dict(kind=kind, nx=_log_pick(rng, 16, 2048), ny=_log_pick(rng, 16, 2048),
                    prec=rng.choice(["fp64", "mixed"]), ring=rng.random() < 0.5)
    if kind == "solve":
        if rng.random() < 0.25:
            n = _log_pick(rng, 128, 512)
            return dict(kind=kind, nx=n, ny=n, bodies=rng.randint(1, 4), prec="fp64", precond=0)
        ny = _log_pick(rng, 128, 1024)
        nx = min(1024, ny * rng.choice([1, 1, 2]))
        return dict(kind=kind, nx=nx, ny=ny, bodies=rng.randint(1, 4), prec="mixed", precond=rng.choice([0, 1, 3, 3]))
    if kind == "batch":
        lo = _log_pick(rng, 128, 512)
        return dict(kind=kind, count=rng.randint(2, 11), lo=lo, hi=rng.choice([lo, 512]),
                    lockstep=rng.choice([1, 4, 8]), precond=rng.choice([1, 3]))
    if kind == "free":
        return dict(kind=kind, n=_log_pick(rng, 128, 512), bodies=rng.randint(1, 4), precond=rng.choice([1, 3]))
    if kind == "rk3":
        ny = _log_pick(rng, 128, 512)
        return dict(kind=kind, nx=2 * ny, ny=ny, precond=rng.choice([1, 3]))
    if kind == "transport":
        ny = _log_pick(rng, 128, 1024)
        return dict(kind=kind, nx=min(2048, ny * rng.choice([1, 2])), ny=ny, bodies=rng.randint(1, 4))
    if kind == "net_forward":
        return dict(kind=kind, batch=rng.randint(1, 3), h=int(math.exp(rng.uniform(math.log(63), math.log(700)))),
                    w=int(math.exp(rng.uniform(math.log(63), math.log(700)))))
    return dict(kind=kind, batch=rng.randint(1, 8), h=rng.randint(60, 130), w=rng.randint(60, 130))


# ------------------------------------------------------------------------------- geometry, fields
def _dev():
    return torch.device("cuda", torch.cuda.current_device())


def _bodies(count, L, h, rng):
    """(level set as a function of X, Y) of each body; L: half of the box's shorter side.  Centres
    lie up to a cell off the grid's nodes."""
    def circle(x, y, r):
        return lambda X, Y: torch.hypot(X - x, Y - y) - r

    def ellipse(x, y, a, b, t):
        c, s = math.cos(t), math.sin(t)
        return lambda X, Y: (torch.sqrt(((c * (X - x) + s * (Y - y)) / a) ** 2 +
                                        ((-s * (X - x) + c * (Y - y)) / b) ** 2) - 1.0) * min(a, b)

    def annulus(x, y, ri, ro):
        return lambda X, Y: torch.maximum(ri - torch.hypot(X - x, Y - y), torch.hypot(X - x, Y - y) - ro)

    def star(x, y, r, amp):
        return lambda X, Y: torch.hypot(X - x, Y - y) - (r + amp * torch.cos(5.0 * torch.atan2(Y - y, X - x)))

    def at(x, y):
        return x * L + rng.uniform(-1, 1) * h, y * L + rng.uniform(-1, 1) * h

    if count == 1:
        return [circle(*at(0.0, 0.0), 0.25 * L)]
    if count == 2:
        return [ellipse(*at(-0.42, -0.3), 0.28 * L, 0.18 * L, 0.6), circle(*at(0.42, 0.35), 0.2 * L)]
    if count == 3:
        return [circle(*at(-0.45, -0.4), 0.2 * L), ellipse(*at(0.45, -0.35), 0.24 * L, 0.15 * L, 0.9),
                ellipse(*at(0.0, 0.45), 0.25 * L, 0.17 * L, 2.1)]
    if count == 4:
        return [circle(*at(-0.45, -0.45), 0.18 * L), ellipse(*at(0.45, -0.45), 0.22 * L, 0.15 * L, 0.4),
                circle(*at(0.45, 0.45), 0.15 * L), ellipse(*at(-0.45, 0.45), 0.2 * L, 0.15 * L, 1.3)]
    return [circle(*at(-0.5, -0.5), 0.14 * L), circle(*at(0.5, -0.5), 0.11 * L), circle(*at(0.0, -0.05), 0.09 * L),
            annulus(*at(0.5, 0.45), 0.1 * L, 0.2 * L), star(*at(-0.5, 0.45), 0.125 * L, 0.0375 * L)]


def _smooth(t):
    t = t.clamp(0.0, 1.0)
    return t * t * t * (10.0 - 15.0 * t + 6.0 * t * t)


class _Flow:
    """Grid, bodies and an exact discrete streamfunction of one problem, from the seed alone."""

    def __init__(self, nx, ny, bodies, seed, compact=False, shift=0.0):
        rng = random.Random(seed)
        dev = _dev()
        self.nx, self.ny, self.nb = nx, ny, bodies
        self.L = L = 2.0 if nx <= 1024 else 4.0            # half of the shorter side
        self.h = h = 2.0 * L / min(nx, ny)
        self.x0, self.y0 = -0.5 * h * nx, -0.5 * h * ny
        self.x = self.x0 + h * torch.arange(nx + 1, dtype=F64, device=dev)
        self.y = self.y0 + h * torch.arange(ny + 1, dtype=F64, device=dev)
        Y, X = torch.meshgrid(self.y, self.x, indexing="ij")
        self.X, self.Y = X, Y
        each = [b(X - shift * L, Y) for b in _bodies(bodies, L, h, random.Random(17 * nx + 5 * ny + bodies))]
        self.phi = torch.stack(each).amin(0)
        self.regions = []
        for p in each:
            js = torch.nonzero((p < 0).any(1)).flatten()
            is_ = torch.nonzero((p < 0).any(0)).flatten()
            self.regions.append((int(is_[0]) - 4, int(is_[-1]) + 4, int(js[0]) - 4, int(js[-1]) + 4))
        self.fluid = (self.phi >= 0)[1:-1, 1:-1]
        # 0 within 8 cells of every body (the star's level set is up to 1.8 times the distance), then
        # smoothly 1
        self.away = _smooth((self.phi - 16.0 * h) / (0.25 * L))
        self.rng = rng
        self.c = [[rng.gauss(0, 1) for _ in range(4)] for _ in range(4)]
        self.offsets = [rng.uniform(-0.7, 0.7) for _ in range(bodies)]
        self.psi = self.poly(X, Y) * (self.bump() if compact else 1.0) + self.vortices(0.3) * (
            self.bump() if compact else 1.0) * self.away

    def poly(self, X, Y):
        X, Y = X / self.L, Y / self.L
        out = torch.zeros_like(X)
        for a in range(3, -1, -1):
            col = torch.zeros_like(X)
            for b in range(3, -1, -1):
                col = col * Y + self.c[a][b]
            out = out * X + col
        return out

    def vortices(self, amplitude, count=40):
        """Gaussian blobs of random centre, strength and width, on the nodes."""
        dev, g = self.x.device, self.rng
        cx = torch.tensor([g.uniform(float(self.x[0]), float(self.x[-1])) for _ in range(count)], dtype=F64, device=dev)
        cy = torch.tensor([g.uniform(float(self.y[0]), float(self.y[-1])) for _ in range(count)], dtype=F64, device=dev)
        s = torch.tensor([g.uniform(0.04, 0.12) * self.L for _ in range(count)], dtype=F64, device=dev)
        a = torch.tensor([g.gauss(0, amplitude) for _ in range(count)], dtype=F64, device=dev)
        ex = torch.exp(-((self.x[None, :] - cx[:, None]) / s[:, None]) ** 2 / 2)
        ey = torch.exp(-((self.y[None, :] - cy[:, None]) / s[:, None]) ** 2 / 2) * a[:, None]
        return ey.T @ ex

    def bump(self):
        """1 around the bodies, smoothly 0 before the box: fields of compact support."""
        r = torch.maximum(self.X.abs() / abs(self.x0), self.Y.abs() / abs(self.y0))
        return 1.0 - _smooth((r - 0.75) / 0.2)

    def omega(self):
        p = self.psi
        lap = (p[1:-1, 2:] + p[1:-1, :-2] + p[2:, 1:-1] + p[:-2, 1:-1] - 4.0 * p[1:-1, 1:-1]) / (self.h * self.h)
        return torch.where(self.fluid, -lap, torch.zeros_like(lap)).contiguous()

    def ring(self):
        p = self.psi
        return torch.cat([p[0], p[-1], p[1:-1, 0], p[1:-1, -1]]).contiguous()

    def gamma(self):
        """Discrete circulation of every bounding region from the streamfunction next to its faces."""
        p, out = self.psi, []
        for lx, rx, ly, ry in self.regions:
            s = (p[ly:ry + 1, rx + 1] - p[ly:ry + 1, rx]).sum() - (p[ly:ry + 1, lx] - p[ly:ry + 1, lx - 1]).sum()
            s = s + (p[ry + 1, lx:rx + 1] - p[ry, lx:rx + 1]).sum() - (p[ly, lx:rx + 1] - p[ly - 1, lx:rx + 1]).sum()
            out.append(-s)
        return torch.stack(out)

    def grid(self):
        return iim.make_grid(self.x0, -self.x0, self.y0, -self.y0, self.nx, self.ny)

    def setup(self):
        return iim.iim_setup_geometry(self.grid(), self.phi.contiguous(), self.regions, [1] * self.nb)

    def psi_b(self, geo):
        cp = iim.iim_geometry_control_points(geo)
        off = torch.tensor(self.offsets, dtype=F64, device=self.x.device)
        return (self.poly(cp["x"], cp["y"]) - off[cp["body"].long()]).contiguous()

    def exact(self):
        """psi, u_x, u_y at the interior nodes (0 in the solid) and the body constants."""
        p, z = self.psi, torch.zeros((), dtype=F64, device=self.x.device)
        return {"psi": torch.where(self.fluid, p[1:-1, 1:-1], z),
                "ux": torch.where(self.fluid, (p[2:, 1:-1] - p[:-2, 1:-1]) / (2.0 * self.h), z),
                "uy": torch.where(self.fluid, -(p[1:-1, 2:] - p[1:-1, :-2]) / (2.0 * self.h), z),
                "psibar": torch.tensor(self.offsets, dtype=F64, device=self.x.device)}


def _opts(prec, precond):
    return iim.default_opts(prec=iim.IIM_FP64 if prec == "fp64" else iim.IIM_MIXED, rtol=RTOL, max_iter=4000,
                            max_refine=30, precond=precond)


RTOL = 1e-12


class _Problem:
    """What a program holds for one immersed-interface problem: the geometry handle with its
    preconditioner, the inputs and the output arrays."""

    def __init__(self, flow, prec, precond, outer=0):
        self.geo = flow.setup()
        if outer:
            iim.iim_geometry_set_outer(self.geo, outer)
        if precond:
            iim.iim_build_preconditioner(self.geo)
        self.opts = _opts(prec, precond)
        self.omega, self.psi_b, self.gamma = flow.omega(), flow.psi_b(self.geo), flow.gamma()
        self.ring = None if outer else flow.ring()
        self.psibar = torch.zeros(flow.nb, dtype=F64, device=self.omega.device)
        self.psi, self.ux, self.uy = (torch.empty_like(self.omega) for _ in range(3))

    def out(self):
        return {"psi": self.psi, "ux": self.ux, "uy": self.uy, "psibar": self.psibar}

    def solve(self):
        iim.iim_poisson_solve(self.geo, self.omega, self.psi_b, self.ring, self.gamma, self.psibar, self.psi, self.ux,
                              self.uy, opts=self.opts)
        return self.out()


def _batch_flows(case, seed):
    lo, hi = int(math.log2(case["lo"])), int(math.log2(case["hi"]))
    sizes = [2 ** (lo + (5 * k + 2 * (k // 3)) % (hi - lo + 1)) for k in range(case["count"])]
    return [_Flow(n, n, 1 if lo == hi else 1 + k % 4, 31 * seed + k) for k, n in enumerate(sizes)]


# ------------------------------------------------------------------------------- box solve
def _box_input(case, seed):
    dev = _dev()
    nx, ny = case["nx"], case["ny"]
    h = 4.0 / nx
    rng = random.Random(seed)
    g = torch.Generator(device=dev).manual_seed(seed)
    x = torch.linspace(0, 1, nx + 1, dtype=F64, device=dev)[1:-1]
    y = torch.linspace(0, 1, ny + 1, dtype=F64, device=dev)[1:-1]
    f = 0.1 * torch.randn(ny - 1, nx - 1, dtype=F64, device=dev, generator=g)
    for _ in range(12):
        s = rng.uniform(0.03, 0.15)
        f += rng.gauss(0, 2) * torch.outer(torch.exp(-((y - rng.random()) / s) ** 2 / 2),
                                           torch.exp(-((x - rng.random()) / s) ** 2 / 2))
    ring = None
    if case["ring"]:
        t = torch.arange(2 * (nx + ny), dtype=F64, device=dev)
        ring = 0.3 * torch.sin(0.01 * t + rng.random()) + 0.1 * torch.randn(2 * (nx + ny), dtype=F64, device=dev, generator=g)
    return h, f, ring


def _dst(a):
    """DST-I along the last axis: X_k = sum_j x_j sin(pi j k / n), n - 1 points."""
    n = a.shape[-1] + 1
    z = torch.zeros(*a.shape[:-1], 1, dtype=a.dtype, device=a.device)
    return -0.5 * torch.fft.rfft(torch.cat([z, a, z, -a.flip(-1)], -1)).imag[..., 1:n]


def _box_exact(case, seed):
    h, f, ring = _box_input(case, seed)
    nx, ny = case["nx"], case["ny"]
    f = f * (h * h)
    if ring is not None:
        f[0] += ring[1:nx]
        f[-1] += ring[nx + 2:2 * nx + 1]
        f[:, 0] += ring[2 * nx + 2:2 * nx + 1 + ny]
        f[:, -1] += ring[2 * nx + 1 + ny:]
    lam = [2.0 - 2.0 * torch.cos(math.pi * torch.arange(1, n, dtype=F64, device=f.device) / n) for n in (nx, ny)]
    s = _dst(_dst(f).T.contiguous()) / (lam[0][:, None] + lam[1][None, :])
    return _dst(_dst(s).T.contiguous()) * (4.0 / (nx * ny))


# ------------------------------------------------------------------------------- transport
class _Transport:
    """Velocity and vorticity of a shear flow (divergence-free, of degree two; its curl) around the
    bodies plus random fluctuations away from them: every extension of the scheme reproduces them, so
    the discrete fluxes follow from the node values alone."""

    def __init__(self, case, seed):
        self.f = f = _Flow(case["nx"], case["ny"], case["bodies"], seed)
        rng, L = f.rng, f.L
        g = torch.Generator(device=f.x.device).manual_seed(seed)
        self.c = [rng.gauss(0, 0.4) for _ in range(9)]
        self.U, self.nu = (1.0 + 0.2 * rng.random(), 0.2 * rng.random()), 0.005
        X, Y = f.X[1:-1, 1:-1], f.Y[1:-1, 1:-1]
        away = f.away[1:-1, 1:-1]
        noise = [torch.randn(X.shape, dtype=F64, device=X.device, generator=g) * away for _ in range(3)]
        ux, uy = self.velocity(X, Y)
        self.ux_ext, self.uy_ext = ux + 0.2 * noise[0], uy + 0.2 * noise[1]
        c = self.c
        curl = -(2.0 * c[2] + 2.0 * c[4] + (6.0 * c[5] + 2.0 * c[7]) * X / L + (2.0 * c[6] + 6.0 * c[8]) * Y / L) / L
        self.w_ext = curl + 0.5 * noise[2]
        z = torch.zeros_like(X)
        self.ux, self.uy, self.w = (torch.where(f.fluid, v, z).contiguous() for v in (self.ux_ext, self.uy_ext, self.w_ext))

    def velocity(self, x, y):
        """(P_y, -P_x) of a cubic polynomial P in x / L, y / L."""
        x, y, c = x / self.f.L, y / self.f.L, self.c
        return (self.U[0] + c[1] + c[3] * x + 2.0 * c[4] * y + c[6] * x * x + 2.0 * c[7] * x * y + 3.0 * c[8] * y * y,
                self.U[1] - c[0] - 2.0 * c[2] * x - c[3] * y - 3.0 * c[5] * x * x - 2.0 * c[6] * x * y - c[7] * y * y)

    def prepare(self):
        f = self.f
        geo = f.setup()
        cp = iim.iim_geometry_control_points(geo)
        ub = torch.cat(self.velocity(cp["x"], cp["y"])).contiguous()
        return dict(geo=geo, w=self.w, ux=self.ux, uy=self.uy, ub=ub, U=self.U, nu=self.nu, rhs=torch.empty_like(self.w),
                    wb=torch.empty(geo.n_control, dtype=F64, device=self.w.device),
                    dg=torch.empty(f.nb, dtype=F64, device=self.w.device))

    def _flux(self, axis):
        """Fluxes f + q through the faces along `axis` (0: x), from node values; the box values beyond."""
        f = self.f
        vel = (self.ux_ext, self.uy_ext)[axis]
        NY, NX = vel.shape
        V = torch.full((NY + 4, NX + 4), self.U[axis], dtype=F64, device=vel.device)
        W = torch.zeros_like(V)
        S = torch.zeros_like(V, dtype=torch.bool)
        V[2:-2, 2:-2], W[2:-2, 2:-2], S[2:-2, 2:-2] = vel, self.w_ext, ~f.fluid
        W[2:-2, -2:] = self.w_ext[:, -1:]
        if axis:
            V, W, S = V.T, W.T, S.T
        V, W, S = V[2:-2], W[2:-2], S[2:-2]                   # rows across the faces
        n = V.shape[1] - 3
        v, w, s = ([t[:, k:k + n] for k in range(4)] for t in (V, W, S))   # nodes a - 1, a, b, b + 1 of every face
        pos = (0.5 * (v[1] + v[2])) >= 0
        into = (s[2] & ~s[1] & ~pos) | (s[1] & ~s[2] & pos)
        pos = pos ^ into
        p = [v[k] * w[k] for k in range(4)]
        up = -p[0] / 6.0 + 5.0 * p[1] / 6.0 + p[2] / 3.0
        dn = p[1] / 3.0 + 5.0 * p[2] / 6.0 - p[3] / 6.0
        out = torch.where(pos, up, dn) - self.nu * (w[2] - w[1]) / f.h
        return out.T if axis else out

    def exact(self):
        f = self.f
        fx, fy = self._flux(0), self._flux(1)                  # (NY, NX + 1), (NY + 1, NX)
        rhs = -((fx[:, 1:] - fx[:, :-1]) + (fy[1:] - fy[:-1])) / f.h
        dg = []
        for lx, rx, ly, ry in f.regions:
            s = (fx[ly - 1:ry, rx] - fx[ly - 1:ry, lx - 1]).sum() + (fy[ry, lx - 1:rx] - fy[ly - 1, lx - 1:rx]).sum()
            dg.append(-f.h * s)
        return {"rhs": torch.where(f.fluid, rhs, torch.zeros_like(rhs)), "omega_b": None, "dgamma": torch.stack(dg)}


# ------------------------------------------------------------------------------- learned guess
def _net_params(seed):
    g = torch.Generator().manual_seed(seed)
    out, layers = [], []
    for k in range(len(DILATIONS)):
        ci = IN_CHANNELS if k == 0 else HIDDEN
        co = 1 if k == len(DILATIONS) - 1 else HIDDEN
        w = (torch.rand(co, ci, 3, 3, generator=g) * 2 - 1) * math.sqrt(6.0 / (9 * ci))
        b = 0.05 * torch.randn(co, generator=g)
        out += [w.flatten(), b]
        layers.append((w, b))
    return torch.cat(out), layers


def _net_input(case, seed):
    """Vorticity, level set and a smooth streamfunction on the pixels, the last one also as the target."""
    dev = _dev()
    B, H, W = case["batch"], case["h"], case["w"]
    g = torch.Generator().manual_seed(seed)
    y = torch.linspace(-1, 1, H, device=dev)
    x = torch.linspace(-1, 1, W, device=dev)
    planes = []
    for _ in range(B):
        r = torch.rand(40, 3, generator=g).to(dev)
        a = torch.randn(40, 1, generator=g).to(dev)
        def blobs(width, amp):
            ey = torch.exp(-((y[None] - 2 * r[:, 1:2] + 1) / width) ** 2 / 2)
            ex = torch.exp(-((x[None] - 2 * r[:, 0:1] + 1) / width) ** 2 / 2)
            return (ey * amp).T @ ex
        w = blobs(0.05, a)
        c = r[:4] * 1.2 - 0.6
        phi = torch.stack([torch.hypot(x[None] - c[k, 0], y[:, None] - c[k, 1]) - 0.15 for k in range(4)]).amin(0)
        u = blobs(0.4, a)
        planes.append(torch.stack([torch.where(phi >= 0, w, torch.zeros_like(w)) / w.square().mean().sqrt(), phi,
                                   0.2 * u / u.square().mean().sqrt()]))
    x = torch.stack(planes).contiguous()
    mask = (x[:, 1:2] >= 0).float().contiguous()
    target = (x[:, 2:3] * torch.sigmoid(8.0 * x[:, 1:2])).contiguous()
    return x, target, mask


def _net_exact(case, seed):
    params, layers = _net_params(seed)
    x, target, mask = _net_input(case, seed)
    dev = x.device
    ws = [w.bfloat16().to(dev, F64).requires_grad_() for w, _ in layers]   # the network's weights are BF16
    bs = [b.to(dev, F64).requires_grad_() for _, b in layers]
    v = x.to(F64)
    with torch.set_grad_enabled(case["kind"] == "net_train"):
        for k, d in enumerate(DILATIONS):
            # a 3x3 convolution as nine products with shifted images
            p = torch.nn.functional.pad(v, (d, d, d, d))
            H, W = v.shape[-2:]
            acc = bs[k][None, :, None, None]
            for t in range(9):
                sh = p[:, :, d * (t // 3):d * (t // 3) + H, d * (t % 3):d * (t % 3) + W]
                acc = acc + torch.einsum("oc,bchw->bohw", ws[k][:, :, t // 3, t % 3], sh)
            v = torch.relu(acc) if k < len(DILATIONS) - 1 else acc
    if case["kind"] == "net_forward":
        return {"y": v}
    loss = (mask.to(F64) * (v - target.to(F64)) ** 2).sum() / mask.to(F64).sum()
    grads = torch.autograd.grad(loss, [t for wb in zip(ws, bs) for t in wb])
    g = torch.cat([t.flatten() for t in grads])
    m, s = 0.1 * g / (1 - 0.9), 0.001 * g * g / (1 - 0.999)
    return {"loss": loss.detach(), "params": params.to(dev, F64) - LR * m / (s.sqrt() + 1e-8)}


LR = 1e-3


# ------------------------------------------------------------------------------- the interface
def prepare(case, seed):
    kind = case["kind"]
    s = {"kind": kind}
    if kind == "box":
        h, f, ring = _box_input(case, seed)
        nx, ny = case["nx"], case["ny"]
        s.update(grid=iim.make_grid(0.0, 4.0, 0.0, h * ny, nx, ny), f=f, ring=ring, u=torch.empty_like(f),
                 prec=iim.IIM_FP64 if case["prec"] == "fp64" else iim.IIM_MIXED,
                 work=torch.empty(2 * (nx - 1) * (ny - 1), dtype=F64, device=f.device))
    elif kind == "solve":
        s["p"] = _Problem(_Flow(case["nx"], case["ny"], case["bodies"], seed), case["prec"], case["precond"])
    elif kind == "free":
        s["p"] = _Problem(_Flow(case["n"], case["n"], case["bodies"], seed, compact=True), "mixed", case["precond"], outer=1)
    elif kind == "batch":
        s["lockstep"] = case["lockstep"]
        s["ps"] = [_Problem(f, "mixed", case["precond"]) for f in _batch_flows(case, seed)]
    elif kind == "rk3":
        # impulsively started flow past a cylinder upstream of the middle, with vortices and noise in the fluid
        f = _Flow(case["nx"], case["ny"], 1, seed, shift=-0.5)
        dev = f.x.device
        g = torch.Generator(device=dev).manual_seed(seed)
        noise = 1e-3 * torch.randn(f.fluid.shape, dtype=F64, device=dev, generator=g)
        w = noise + (f.vortices(2.0, 12) * f.away * f.bump())[1:-1, 1:-1]
        f.psi = f.Y.clone()
        geo = f.setup()
        iim.iim_build_preconditioner(geo)
        w0 = torch.where(f.fluid, w, torch.zeros_like(w)).contiguous()
        s.update(geo=geo, w0=w0, omega=w0.clone(), ring=f.ring(), opts=_opts("mixed", case["precond"]),
                 gamma=torch.zeros(1, dtype=F64, device=dev), psibar=torch.zeros(1, dtype=F64, device=dev))
    elif kind == "transport":
        s.update(_Transport(case, seed).prepare())
    else:
        x, target, mask = _net_input(case, seed)
        net = Net()
        net.set(_net_params(seed)[0].numpy())
        s.update(net=net, x=x, target=target, mask=mask, y=torch.empty_like(target))
    return s


def run(s):
    kind = s["kind"]
    if kind == "box":
        iim.iim_box_poisson(s["grid"], s["f"], s["ring"], s["u"], s["prec"], s["work"])
        return s["u"]
    if kind in ("solve", "free"):
        return s["p"].solve()
    if kind == "batch":
        ps = s["ps"]
        iim.iim_set_lockstep(s["lockstep"])
        iim.iim_poisson_solve_batched([p.geo for p in ps], [p.omega for p in ps], [p.psi_b for p in ps],
                                      [p.ring for p in ps], [p.gamma for p in ps], [p.psibar for p in ps],
                                      [p.psi for p in ps], [p.ux for p in ps], [p.uy for p in ps], opts=ps[0].opts,
                                      n_streams=8)
        return [p.out() for p in ps]
    if kind == "rk3":
        # the step starts from a copy: the program keeps the old state to reject the step
        s["omega"].copy_(s["w0"])
        s["gamma"].zero_()
        dt, _, _ = iim.iim_rk3_step(s["geo"], s["omega"], s["gamma"], s["psibar"], None, None, s["ring"], (1.0, 0.0), 0.005,
                                    0.5, opts=s["opts"])
        return {"omega": s["omega"], "gamma": s["gamma"], "psibar": s["psibar"], "dt": dt}
    if kind == "transport":
        iim.iim_transport_rhs(s["geo"], s["w"], s["ux"], s["uy"], s["ub"], s["U"], s["nu"], s["rhs"], omega_b_out=s["wb"],
                              dgamma_out=s["dg"])
        return {"rhs": s["rhs"], "omega_b": s["wb"], "dgamma": s["dg"]}
    if kind == "net_forward":
        s["net"].forward(s["x"], s["y"])
        return {"y": s["y"]}
    loss = s["net"].train_step(s["x"], s["target"], s["mask"], LR)
    return {"loss": loss, "params": s["net"].get()}


def exact(case, seed):
    kind = case["kind"]
    if kind == "box":
        return _box_exact(case, seed)
    if kind == "solve":
        return _Flow(case["nx"], case["ny"], case["bodies"], seed).exact()
    if kind == "free":
        return _Flow(case["n"], case["n"], case["bodies"], seed, compact=True).exact()
    if kind == "batch":
        return [f.exact() for f in _batch_flows(case, seed)]
    if kind == "transport":
        return _Transport(case, seed).exact()
    if kind == "rk3":
        return None          # three immersed-interface solves in 64 bits: minutes
    return _net_exact(case, seed)


def work(case):
    """Bytes: inputs read once, outputs written once.  Flops: of one pass, at the least one
    rectangular solve (a sine transform pair per row, the column solves) for every solve."""
    kind = case["kind"]

    def box(nx, ny):
        return nx * ny * (2 * 2.5 * math.log2(2 * nx) + 14)

    if kind == "box":
        nx, ny = case["nx"], case["ny"]
        return {"bytes": 16.0 * (nx - 1) * (ny - 1) + (16.0 * (nx + ny) if case["ring"] else 0.0), "flops": box(nx, ny)}
    if kind == "solve":
        return {"bytes": 32.0 * case["nx"] * case["ny"], "flops": 2 * box(case["nx"], case["ny"])}
    if kind == "free":
        return {"bytes": 32.0 * case["n"] ** 2, "flops": 4 * box(case["n"], case["n"])}
    if kind == "batch":
        lo, hi = int(math.log2(case["lo"])), int(math.log2(case["hi"]))
        ns = [2 ** (lo + (5 * k + 2 * (k // 3)) % (hi - lo + 1)) for k in range(case["count"])]
        return {"bytes": sum(32.0 * n * n for n in ns), "flops": sum(2 * box(n, n) for n in ns)}
    if kind == "rk3":
        n = case["nx"] * case["ny"]
        return {"bytes": 16.0 * n, "flops": 3 * (2 * box(case["nx"], case["ny"]) + 50 * n)}
    if kind == "transport":
        n = case["nx"] * case["ny"]
        return {"bytes": 32.0 * n, "flops": 50.0 * n}
    n = case["batch"] * case["h"] * case["w"]
    hid = len(DILATIONS) - 2
    macs = 9.0 * n * (IN_CHANNELS * HIDDEN + hid * HIDDEN * HIDDEN + HIDDEN)
    if kind == "net_forward":
        return {"bytes": 4.0 * n * (IN_CHANNELS + 1), "flops": 2 * macs}
    return {"bytes": 4.0 * n * (IN_CHANNELS + 2), "flops": 6 * macs}
