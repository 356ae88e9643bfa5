"""Transport right-hand side near the end of the FP64 range on a cell size that is not a power of two:
where a flux difference divided by h overflows, the result is that infinity, as the oracle's division
gives it; elsewhere the oracle's value."""
import numpy as np
import pytest
import torch

import paper_2109_13628_gb300 as iim
from oracle import poisson as op
from oracle import transport as tr
from paper_2109_13628_gb300 import inputs
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("half", [1.5, 2.0])
def test_overflowing_differences_stay_infinite(half):
    n = 64
    g = inputs.square_grid(n, half)
    X, Y = g.nodes()
    phi = inputs.phi_circle(X, Y, -0.4 * half, -0.35 * half, 0.2 * half)
    P = inputs.Problem(grid=g, phi=phi, regions=[inputs.region_around(g, phi)], modes=[1],
                       omega=np.zeros((n - 1, n - 1)), psi_box=np.zeros(4 * n),
                       psi_b_fn=lambda x, y, k: np.zeros_like(x), psibar=np.zeros(1), gamma=None, exact=None)
    S = op.Setup(P)
    fl = (phi >= 0)[1:-1, 1:-1]
    rng = np.random.default_rng(8)
    away = (phi > 8 * g.h)[1:-1, 1:-1]           # the extensions at the wall stay small
    w = np.where(away, 1e307 * rng.normal(size=fl.shape), 0.0)
    ux, uy = (np.where(fl, 0.3 * rng.normal(size=fl.shape), 0.0) for _ in range(2))
    ncp = S.geo["cp"]["t"].size
    with np.errstate(over="ignore"):
        rhs = tr.transport_rhs(tr.TransportSetup(S), w, ux, uy, (np.zeros(ncp), np.zeros(ncp)), (0.0, 0.0), 0.004)[0]
    assert 50 < np.isinf(rhs).sum() < rhs.size / 2 and not np.isnan(rhs).any()
    geo = gu.setup(P)
    out = torch.empty((n - 1) ** 2, dtype=torch.float64, device=gu.dev())
    iim.iim_transport_rhs(geo, gu.T(w.ravel()), gu.T(ux.ravel()), gu.T(uy.ravel()), None, (0.0, 0.0), 0.004, out)
    r = out.cpu().numpy().reshape(rhs.shape)
    inf = np.isinf(rhs)
    assert np.array_equal(r[inf], rhs[inf])
    assert np.abs(r[~inf] - rhs[~inf]).max() <= 1e-11 * 1e307 / g.h
    geo.close()
