"""The reduced camera system formed from sorted observation pairs and the PCG
on it (the route of problems it pays for) against the oracle: block layouts
around the edges of its grid, tasks of one to many rounds of lanes, points of
one and of many views, frozen parameters, cameras without observations, a
camera that observes a point twice; the direct solver's build on the same
blocks.  Bounds are those of the other damped-solve tests (1e-9 in FP64)."""
import numpy as np
import pytest
import torch

import oracle as orc
import paper_2409_12190_gb300 as ba
import scenegen
from gpu_helpers import np64, problem, rel_err

pytestmark = pytest.mark.gpu


def _ragged(C, P, seed, lo=1, hi=9):
    """Cameras on an arc; views from lo to hi, the first point seen by all."""
    sc = scenegen.arc_scene(C, P, seed=seed, views_lo=lo, views_hi=hi)
    seen = sc.cam_idx[sc.pt_idx == 0]
    rest = np.setdiff1d(np.arange(C), seen).astype(np.int32)
    rng = np.random.default_rng(seed)
    return scenegen.Scene(sc.cams_gt, sc.points_gt, np.concatenate([sc.cam_idx, rest]),
                          np.concatenate([sc.pt_idx, np.zeros_like(rest)]),
                          np.concatenate([sc.noise, rng.normal(size=(len(rest), 2))]), sc.cams_init, sc.points_init)


def _launches(prob, call):
    torch.cuda.synchronize()
    n = ba.kernel_launch_count()
    out = call()
    torch.cuda.synchronize()
    return out, ba.kernel_launch_count() - n


@pytest.mark.parametrize("C,P", [(2, 5), (7, 33), (30, 700), (151, 900), (153, 1200), (310, 1500)])
@pytest.mark.parametrize("frozen", [False, True])
def test_iterates_match_the_oracle(C, P, frozen):
    sc = _ragged(C, P, seed=C)
    pix = orc.pixels_from_scene(sc)
    fixed = orc.gauge_mask(C) if frozen else None
    its = 8
    blk = orc.assemble(sc.cams_init, sc.points_init, sc.cam_idx, sc.pt_idx, pix)
    dc_ref, dp_ref, n_ref, rel_ref = orc.solve_damped(
        blk, sc.cam_idx, sc.pt_idx, 1e-2, orc.LMOptions(solver="pcg", pcg_maxiter=its, pcg_tol=0.0), fixed=fixed)
    with problem(sc, pix, "f64") as prob:
        if frozen:
            prob.set_fixed(torch.from_numpy(fixed))
        (dc, dp, n, rel), launches = _launches(prob, lambda: prob.damped_solve(1e-2, its, 0.0))
        again = prob.damped_solve(1e-2, its, 0.0)[0]
    assert launches < 5 * its  # one launch for the whole PCG, not five an iteration
    assert n == n_ref and abs(rel - rel_ref) <= 1e-7 * abs(rel_ref) + 1e-12
    assert rel_err(np64(dc), dc_ref) < 1e-9 and rel_err(np64(dp), dp_ref) < 1e-9
    assert torch.equal(dc, again)


@pytest.mark.parametrize("solver", ["pcg", "cholesky"])
@pytest.mark.parametrize("precision", ["f64", "f32"])
def test_point_observed_twice_by_a_camera(solver, precision):
    """Both observations' products with each other belong to the camera's own
    block.  The converged step against the oracle's dense Jacobian (FP32 input
    rounded first, so FP32 differs by its linearisation: 1e-3 of the step)."""
    sc = _ragged(6, 60, seed=3, lo=3, hi=5)
    dup = np.arange(0, sc.O, 7)
    sc = scenegen.Scene(sc.cams_gt, sc.points_gt, np.concatenate([sc.cam_idx, sc.cam_idx[dup]]),
                        np.concatenate([sc.pt_idx, sc.pt_idx[dup]]),
                        np.concatenate([sc.noise, sc.noise[dup] + 0.3]), sc.cams_init, sc.points_init)
    pix = orc.pixels_from_scene(sc)
    dc_ref, dp_ref = orc.dense_lm_delta(sc.cams_init, sc.points_init, sc.cam_idx, sc.pt_idx, pix, 1e-1)
    with problem(sc, pix, precision, solver=solver) as prob:
        dc, dp, _, _ = prob.damped_solve(1e-1, 500, 1e-13 if precision == "f64" else 1e-6)
    tol = 1e-8 if precision == "f64" else 1e-3
    assert rel_err(np64(dc), dc_ref) < tol and rel_err(np64(dp), dp_ref) < tol


@pytest.mark.parametrize("C,P,huber", [(24, 2500, 0.0), (97, 4000, 1.0)])
def test_single_precision_trial(C, P, huber):
    """One trial in FP32 against the same in FP64: the trial's cost to 1e-4 of
    the decrease (the step differs by FP32 rounding of the Jacobians)."""
    sc = scenegen.ring_scene(C, P, seed=C, view_p=0.2, huber_delta=huber)
    pix = orc.pixels_from_scene(sc)
    st = []
    for precision in ("f64", "f32"):
        with problem(sc, pix, precision, pcg_maxiter=15, pcg_tol=0.0, lambda0=1e-2) as prob:
            _, launches = _launches(prob, lambda: prob.solve(1))
            assert launches < 60
            st.append(prob.stats()[0])
    a, b = st
    assert b["pcg_iters"] == a["pcg_iters"] == 15
    assert abs(a["cost_trial"] - b["cost_trial"]) < 1e-4 * abs(a["cost"] - a["cost_trial"])
    assert abs(a["model"] - b["model"]) < 1e-4 * abs(a["model"])


def test_unobserved_camera_in_the_direct_solve():
    base = scenegen.arc_scene(5, 60, seed=3, views_lo=2, views_hi=3)
    sc = scenegen.Scene(np.vstack([base.cams_gt, base.cams_gt[:1]]), base.points_gt, base.cam_idx, base.pt_idx,
                        base.noise, np.vstack([base.cams_init, base.cams_init[:1]]), base.points_init)
    pix = orc.pixels_from_scene(sc)
    blk = orc.assemble(sc.cams_init, sc.points_init, sc.cam_idx, sc.pt_idx, pix)
    dc_ref, _, _, _ = orc.solve_damped(blk, sc.cam_idx, sc.pt_idx, 1e-2, orc.LMOptions(solver="cholesky"))
    with problem(sc, pix, "f64", solver="cholesky") as prob:
        dc = np64(prob.damped_solve(1e-2, 0, 0.0)[0])
    assert np.all(dc[5] == 0.0) and rel_err(dc, dc_ref) < 1e-9


def test_solves_on_two_streams_at_once():
    """Two problems solved at the same time, each on a stream and thread of its
    own, give the bits that they give alone."""
    import threading

    scs = [_ragged(160, 2000, seed=5), _ragged(60, 3000, seed=6)]
    pix = [orc.pixels_from_scene(sc) for sc in scs]
    alone = []
    for sc, px in zip(scs, pix):
        with problem(sc, px, "f64", pcg_maxiter=40) as prob:
            prob.solve(6)
            alone.append(prob.params())
    probs = [problem(sc, px, "f64", pcg_maxiter=40) for sc, px in zip(scs, pix)]
    torch.cuda.synchronize()

    def work(prob):
        with torch.cuda.stream(torch.cuda.Stream()):
            for _ in range(6):
                prob.solve(1)

    threads = [threading.Thread(target=work, args=(p,)) for p in probs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    for prob, want in zip(probs, alone):
        got = prob.params()
        torch.cuda.synchronize()
        assert all(torch.equal(a, b) for a, b in zip(got, want))
        prob.close()


@pytest.mark.parametrize("solver", ["pcg", "cholesky"])
@pytest.mark.parametrize("k1", [-3.0, -8.0])
def test_observations_near_the_fold_of_the_distortion(solver, k1):
    """Where 1 + 3 k1 r^2 + 5 k2 r^4 passes through 0 the lean form of an
    observation does not exist: those take their planes.  Two cameras with such
    a distortion, the image radius of their points spread over the fold."""
    sc = _ragged(8, 400, seed=11, lo=3, hi=6)
    cams = sc.cams_init.copy()
    cams[[2, 5], 7] = k1
    pix = orc.pixels_from_scene(sc)
    X = orc.rodrigues(cams[sc.cam_idx, :3]) @ sc.points_init[sc.pt_idx][:, :, None]
    X = X[:, :, 0] + cams[sc.cam_idx, 3:6]
    r2 = ((X[:, :2] / X[:, 2:]) ** 2).sum(1)
    mu, nu = (1 + n * cams[sc.cam_idx, 7] * r2 + m * cams[sc.cam_idx, 8] * r2 * r2 for n, m in ((3, 5), (1, 1)))
    assert np.sum(np.abs(mu) < 0.125 * np.abs(nu)) >= 3
    sc = scenegen.Scene(sc.cams_gt, sc.points_gt, sc.cam_idx, sc.pt_idx, sc.noise, cams, sc.points_init)
    blk = orc.assemble(sc.cams_init, sc.points_init, sc.cam_idx, sc.pt_idx, pix)
    its = 8
    dc_ref, dp_ref, _, _ = orc.solve_damped(blk, sc.cam_idx, sc.pt_idx, 1e-1,
                                            orc.LMOptions(solver=solver, pcg_maxiter=its, pcg_tol=0.0))
    with problem(sc, pix, "f64", solver=solver) as prob:
        dc, dp, _, _ = prob.damped_solve(1e-1, its, 0.0)
    assert rel_err(np64(dc), dc_ref) < 1e-9 and rel_err(np64(dp), dp_ref) < 1e-9


@pytest.mark.parametrize("solver", ["pcg", "cholesky"])
def test_camera_of_focal_length_zero(solver):
    """Its projection's derivative by the point is 0 and so is the lean form's
    factor: those observations take their planes (Jc keeps p q^T, Jp is 0)."""
    sc = _ragged(8, 400, seed=11, lo=3, hi=6)
    cams = sc.cams_init.copy()
    cams[[2, 5], 6] = 0.0
    pix = orc.pixels_from_scene(sc)
    sc = scenegen.Scene(sc.cams_gt, sc.points_gt, sc.cam_idx, sc.pt_idx, sc.noise, cams, sc.points_init)
    blk = orc.assemble(sc.cams_init, sc.points_init, sc.cam_idx, sc.pt_idx, pix)
    its = 8
    dc_ref, dp_ref, n_ref, _ = orc.solve_damped(blk, sc.cam_idx, sc.pt_idx, 1e-1,
                                                orc.LMOptions(solver=solver, pcg_maxiter=its, pcg_tol=0.0))
    assert np.all(np.isfinite(dc_ref)) and np.abs(dc_ref).max() > 0
    with problem(sc, pix, "f64", solver=solver) as prob:
        dc, dp, n, _ = prob.damped_solve(1e-1, its, 0.0)
    if solver == "pcg":
        assert n == n_ref
    assert rel_err(np64(dc), dc_ref) < 1e-9 and rel_err(np64(dp), dp_ref) < 1e-9
