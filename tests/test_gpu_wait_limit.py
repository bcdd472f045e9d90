"""A grid-wide wait of the PCG that runs out leaves no mixture of solved and
unsolved cameras.  Each limit, from one poll up, gives either the whole answer
or dc = 0 everywhere, and a solve with the limit back at its default gives the
whole answer again.  (The waits end by themselves after so many polls; nothing
is kept from arriving.)"""
import pytest
import torch

import oracle as orc
import scenegen
from gpu_helpers import problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("jacobian", ["auto", "recompute"])  # formed S; the implicit product
def test_no_mixture_when_a_wait_runs_out(jacobian):
    sc = scenegen.arc_scene(310, 1500, seed=4, views_lo=2, views_hi=7)
    pix = orc.pixels_from_scene(sc)
    with problem(sc, pix, "f64", jacobian=jacobian) as prob:
        want, _, its, want_rel = prob.damped_solve(1e-2, 8, 0.0)
        assert its == 8 and torch.all(torch.any(want != 0, dim=1))
        lost = 0
        for polls in [1] * 5 + [2, 3, 4, 6] * 4 + [8, 12, 16, 32, 64, 256, 4096]:
            prob.set_wait_limit(polls)
            dc, _, _, rel = prob.damped_solve(1e-2, 8, 0.0)
            if rel == 1.0:
                lost += 1
                assert torch.all(dc == 0)
            else:
                assert rel == want_rel and torch.equal(dc, want)
        assert lost > 0
        # in a trial (captured), counted
        prob.set_wait_limit(1)
        prob.solve(1)
        s = prob.stats()[-1]
        assert s["pcg_rel_res"] == 1.0 and s["precond_fallbacks"] == 1
        prob.set_wait_limit(0)
        with problem(sc, pix, "f64", jacobian=jacobian) as fresh:
            prob.set_params(torch.from_numpy(sc.cams_init), torch.from_numpy(sc.points_init))
            assert torch.equal(prob.damped_solve(1e-2, 8, 0.0)[0], want)
            assert torch.equal(fresh.damped_solve(1e-2, 8, 0.0)[0], want)
