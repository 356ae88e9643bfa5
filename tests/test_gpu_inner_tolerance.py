"""How far under the target the preconditioned mixed solves end.  The default Krylov tolerance of a
correction is max(kappa ||r||, last ||f||) with kappa = 1e-5 and last = rtol / 100: of the Schur residual,
which is what the correction leaves at the affected nodes of the un-reduced residual, beside the FP32 noise
of the other rows.  A solve whose corrections are carried much further (inner_rtol) shows that noise: it
ends at s ||f|| after k corrections, each a contraction by about c = s^(1/k), so the residual that the last
one starts from is s / c and the default may end at s + kappa s / c + rtol / 100.  Twice the added terms
are allowed."""
import pytest

import paper_2109_13628_gb300 as iim
from oracle import poisson as op
from paper_2109_13628_gb300 import inputs
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu

RTOL = 1e-12


@pytest.mark.parametrize("precond", [1, 3])
@pytest.mark.parametrize("n", [128, 256, 512, 1024])
def test_default_tolerance_keeps_the_margin(n, precond):
    for seed in range(6):
        P = inputs.bicubic_bodies(n, seed=seed, circulation=True)
        gam = op.gamma_from_regions(P)
        geo = gu.setup(P)
        iim.iim_build_preconditioner(geo)
        opts = lambda inner: iim.default_opts(prec=iim.IIM_MIXED, rtol=RTOL, restart=64, max_iter=4000, max_refine=30,
                                              precond=precond, inner_rtol=inner)
        usual, tight = [gu.solve_opts(P, geo, gamma=gam, opts=opts(inner))["stats"] for inner in (0.0, 1e-9)]
        if usual["refinements"] == tight["refinements"]:
            s = tight["rel_res"]
            c = s ** (1.0 / tight["refinements"])
            assert usual["rel_res"] <= s + 2 * (1e-5 * s / c + RTOL / 100), (n, precond, seed)
        geo.close()
