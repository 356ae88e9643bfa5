"""Transport right-hand side and total-pressure data with outputs in the place of inputs: equal, bit for
bit, to the calls with separate arrays (the grid has many blocks, whose halos overlap)."""
import numpy as np
import pytest
import torch

import paper_2109_13628_gb300 as iim
from paper_2109_13628_gb300 import inputs
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu

N = 256
F64 = torch.float64


def flow(modes):
    g = inputs.square_grid(N)
    X, Y = g.nodes()
    a = inputs.phi_circle(X, Y, -0.8, -0.7, 0.45)
    b = inputs.phi_star(X, Y, 0.7, 0.6, 0.45, 0.08, 4)
    P = inputs.Problem(grid=g, phi=inputs.union(a, b), regions=[inputs.region_around(g, a), inputs.region_around(g, b)],
                       modes=modes, omega=np.zeros((N - 1, N - 1)), psi_box=np.zeros(4 * N),
                       psi_b_fn=lambda x, y, k: np.zeros_like(x), psibar=np.zeros(2), gamma=None, exact=None)
    rng = np.random.default_rng(4)
    fl = (P.phi >= 0)[1:-1, 1:-1]
    return gu.setup(P), [gu.T(np.where(fl, rng.normal(size=fl.shape), 0.0).ravel()) for _ in range(3)]


def placements(n):
    """(name, which field, offset): an output of n values over a field, or starting inside one."""
    return [("omega", 0, 0), ("ux", 1, 0), ("uy", 2, 0), ("into omega", 0, 40 * (N - 1) + 7), ("before ux", 1, -300)]


def arrays(fields, which, offset, n):
    """The fields, one of them in a wider buffer, and the output of n values at the offset from it."""
    size = fields[which].numel()
    buf = torch.full((size + 2 * n,), float("nan"), dtype=F64, device=gu.dev())
    lo = n
    buf[lo:lo + size] = fields[which]
    ins = [f.clone() for f in fields]
    ins[which] = buf[lo:lo + size]
    return ins, buf[lo + offset:lo + offset + n]


@pytest.mark.parametrize("name,which,offset", placements(0))
def test_transport_rhs_in_place(name, which, offset):
    geo, fields = flow([1, 1])
    n = fields[0].numel()
    ub = gu.T(np.random.default_rng(5).normal(size=2 * geo.n_control))

    def call(ins, rhs, wb, dg):
        iim.iim_transport_rhs(geo, *ins, ub, (0.8, -0.3), 0.004, rhs, omega_b_out=wb, dgamma_out=dg)
        return [t.clone() for t in (rhs, wb, dg)]

    new = lambda k: torch.empty(k, dtype=F64, device=gu.dev())
    ref = call(fields, new(n), new(geo.n_control), new(2))
    for out in range(3):
        size = (n, geo.n_control, 2)[out]
        outs = [new(n), new(geo.n_control), new(2)]
        ins, outs[out] = arrays(fields, which, max(offset, 1 - size), size)
        for a, b in zip(call(ins, *outs), ref):
            assert torch.equal(a, b), (name, out)
    geo.close()


@pytest.mark.parametrize("name,which,offset", placements(0))
def test_total_pressure_problem_in_place(name, which, offset):
    geo, fields = flow([0, 0])
    iim.iim_geometry_set_wall_condition(geo, 1)
    n = fields[0].numel()

    def call(ins, f, data, wb):
        iim.iim_total_pressure_problem(geo, *ins, None, (0.8, -0.3), 0.004, f, data, omega_b_out=wb)
        return [t.clone() for t in (f, data, wb)]

    new = lambda k: torch.empty(k, dtype=F64, device=gu.dev())
    ref = call(fields, new(n), new(geo.n_control), new(geo.n_control))
    for out in range(3):
        size = (n, geo.n_control, geo.n_control)[out]
        outs = [new(n), new(geo.n_control), new(geo.n_control)]
        ins, outs[out] = arrays(fields, which, max(offset, 1 - size), size)
        for a, b in zip(call(ins, *outs), ref):
            assert torch.equal(a, b), (name, out)
    geo.close()
