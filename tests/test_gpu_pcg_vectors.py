"""PCG on the implicit Schur product with its vector work in one launch per
iteration, against the oracle: camera counts around its blocks of 32, frozen
parameters, stopping on the tolerance.  Recomputed FP64 Jacobians keep the
implicit product at every size.  Bounds are those of the other damped-solve
tests (1e-9 in FP64)."""
import pytest
import torch

import oracle as orc
import scenegen
from gpu_helpers import np64, problem, rel_err

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("C,P,tol", [(2, 9, 0.0), (31, 400, 0.0), (32, 400, 0.0), (33, 400, 1e-3), (300, 2500, 0.0)])
@pytest.mark.parametrize("frozen", [False, True])
def test_iterates_match_the_oracle(C, P, tol, frozen):
    sc = scenegen.arc_scene(C, P, seed=C, views_lo=2, views_hi=min(C, 5))
    pix = orc.pixels_from_scene(sc)
    fixed = orc.gauge_mask(C) if frozen else None
    its = 8 if tol == 0.0 else 60
    blk = orc.assemble(sc.cams_init, sc.points_init, sc.cam_idx, sc.pt_idx, pix)
    dc_ref, dp_ref, n_ref, rel_ref = orc.solve_damped(
        blk, sc.cam_idx, sc.pt_idx, 1e-1, orc.LMOptions(solver="pcg", pcg_maxiter=its, pcg_tol=tol), fixed=fixed)
    with problem(sc, pix, "f64", jacobian="recompute") as prob:
        if frozen:
            prob.set_fixed(torch.from_numpy(fixed))
        dc, dp, n, rel = prob.damped_solve(1e-1, its, tol)
        again = prob.damped_solve(1e-1, its, tol)[0]
    assert n == n_ref and abs(rel - rel_ref) <= 1e-7 * abs(rel_ref) + 1e-12
    assert rel_err(np64(dc), dc_ref) < 1e-9 and rel_err(np64(dp), dp_ref) < 1e-9
    assert torch.equal(dc, again)
