"""Solves that follow a longer restart length.  The Krylov buffers grow with it, and the whole-solve graph
kept from before holds the old ones: a solve that finds its own arguments again must not replay it."""
import numpy as np
import pytest

import paper_2109_13628_gb300 as iim
from oracle import poisson as op
from paper_2109_13628_gb300 import inputs
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,precond", [(iim.IIM_FP64, 0), (iim.IIM_MIXED, 1), (iim.IIM_MIXED, 3)])
@pytest.mark.parametrize("between", ["guess", "profiled"])
def test_shorter_restart_after_a_longer_one(prec, precond, between):
    P = inputs.bicubic_bodies(128, seed=11, circulation=True)
    gam = gu.T(op.gamma_from_regions(P))
    geo = gu.setup(P)
    n = P.omega.size
    omega, psi_b, ring = gu.T(P.omega.ravel()), gu.T(gu.psi_b_for(P, geo)), gu.T(P.psi_box)
    psi, pb = gu.T(np.zeros(n)), gu.T(np.zeros(len(P.regions)))
    zero = gu.T(np.zeros(n))

    def solve(restart, guess=None):
        o = iim.default_opts(prec=prec, rtol=1e-11, max_iter=4000, restart=restart, precond=precond,
                             guess=0 if guess is None else 1)
        st = iim.iim_poisson_solve(geo, omega, psi_b, ring, gam, pb, psi, None, None, guess, opts=o)
        return psi.cpu().numpy(), st["iters"], st["refinements"]

    first = solve(20)                    # host-driven
    for restart, longer in ((20, 40), (30, 64)):
        ref = solve(restart)
        solve(restart)                   # the graph, its buffers and the caller's arrays unchanged
        if between == "guess":
            solve(longer, zero)
        else:
            iim.iim_profile_begin()
            solve(longer)
            iim.iim_profile_end()
        out = solve(restart)
        assert np.array_equal(out[0], ref[0]) and out[1:] == ref[1:]
    assert np.isfinite(first[0]).all()
    geo.close()
