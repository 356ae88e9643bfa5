"""Krylov steps on thread-block clusters and the launch that follows a residual, at the sizes where
their layout changes: 512 unknowns and one more (8 or 16 blocks to a cluster), 2560 and one more
(clustered, or the general kernels), 1, 8 and 9 circulation bodies (64 or 16 blocks per region sum),
restart lengths 1, 3 and 64 with each preconditioner form, host-driven and as one graph.

The streamfunction is bicubic, so the discrete solution is known exactly.  Bound of the error: the
solve leaves a residual of 1e-13 ||f||_2 with ||f||_2 about max|psi| / h^2 sqrt(4 n), and the inverse
operator's norm on the box of side 4 is 0.8, so |error| <= 1e-13 * 0.8 * (n^2 / 16) * 2 sqrt(n) max|psi|."""
import numpy as np
import pytest

import paper_2109_13628_gb300 as iim
from oracle import poisson as op
from oracle.geometry import affected_points
from paper_2109_13628_gb300 import inputs
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu


def problem(n, centres, radius, circulation):
    """Circles of the given radius (cells) at the given centres (cells from the middle)."""
    g = inputs.square_grid(n)
    X, Y = g.nodes()
    phis = [inputs.phi_circle(X, Y, x * g.h, y * g.h, radius * g.h) for x, y in centres]
    phi = inputs.union(*phis)
    c = inputs.bicubic_coeffs(n + len(centres))
    psi = inputs.bicubic(X, Y, c)
    offs = np.linspace(-0.4, 0.6, len(centres))
    P = inputs.Problem(
        grid=g, phi=phi, regions=[inputs.region_around(g, p) for p in phis], modes=[int(circulation)] * len(centres),
        omega=inputs._mask_interior(g, phi, inputs.bicubic_neg_laplacian(X, Y, c)), psi_box=inputs.box_ring(g, psi),
        psi_b_fn=lambda x, y, body: inputs.bicubic(x, y, c) - offs[body], psibar=offs, gamma=None, exact=psi)
    gam = np.array([op.discrete_circulation(psi, r) for r in P.regions]) if circulation else None
    return P, gam


def check(P, gam, precond, restart, prec=iim.IIM_MIXED, geo=None):
    n = P.grid.nx
    opts = iim.default_opts(prec=prec, rtol=1e-13, max_iter=4000, restart=restart, precond=precond)
    outs = [gu.solve_opts(P, geo, gamma=gam, psibar=P.psibar if gam is None else None, opts=opts) for _ in range(2)]
    fl = (P.phi >= 0)[1:-1, 1:-1]
    bound = 1e-13 * 0.8 * (n * n / 16) * 2 * np.sqrt(n) * np.abs(P.exact).max()
    for out in outs:
        assert out["stats"]["rel_res"] <= 1e-13
        assert np.abs(out["psi"] - P.exact[1:-1, 1:-1])[fl].max() <= bound, (precond, restart, out["stats"])
        assert np.abs(out["psibar"] - P.psibar).max() <= bound
    assert np.array_equal(outs[0]["psi"], outs[1]["psi"])   # host-driven, then the graph


@pytest.mark.parametrize("n,radius,na", [(256, 45.25, 512), (1024, 226.25, 2560)])
@pytest.mark.parametrize("circulation", [False, True])
def test_cluster_layout_edges(n, radius, na, circulation):
    P, gam = problem(n, [(0.0, 0.2)], radius, circulation)
    plus, minus = affected_points(P.phi)
    assert int((plus | minus).sum()) == na
    geo = gu.setup(P)
    iim.iim_build_preconditioner(geo)
    for precond, restart in ((0, 64), (1, 1), (1, 3), (3, 1), (3, 3), (3, 64)):
        check(P, gam, precond, restart, geo=geo)
    geo.close()


@pytest.mark.parametrize("bodies", [1, 8, 9])
@pytest.mark.parametrize("prec", [iim.IIM_MIXED, iim.IIM_FP64])
def test_region_sums_of_many_bodies(bodies, prec):
    centres = [(70.0 * i + 1.3, 70.0 * j - 0.4) for j in (-1, 0, 1) for i in (-1, 0, 1)][:bodies]
    P, gam = problem(256, centres, 18.3, True)
    geo = gu.setup(P)
    check(P, gam, 0, 64, prec, geo)
    iim.iim_build_preconditioner(geo)
    check(P, gam, 3, 64, prec, geo)
    geo.close()
