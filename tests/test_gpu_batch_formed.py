"""Windows whose reduced system is formed in their CTA (FP32): observations of
one point by one camera twice (both products belong to the camera's own
block), and frozen parameters.  One trial against the FP64 solve of the same
window: the trial's cost to 1e-4 of the decrease, the bound of the formed
system's other single-precision test."""
import numpy as np
import pytest

import oracle as orc
import paper_2409_12190_gb300 as ba
import scenegen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("huber", [0.0, 1.0])
@pytest.mark.parametrize("C", [2, 6, 20])
def test_point_observed_twice_by_a_camera(C, huber):
    base = scenegen.arc_scene(C, 40 * C, seed=C, views_lo=2, views_hi=min(C, 6))
    dup = np.arange(0, base.O, 7)
    sc = scenegen.Scene(base.cams_gt, base.points_gt, np.concatenate([base.cam_idx, base.cam_idx[dup]]),
                        np.concatenate([base.pt_idx, base.pt_idx[dup]]),
                        np.concatenate([base.noise, base.noise[dup] + 0.3]), base.cams_init, base.points_init)
    inputs = [(s.cams_init, s.points_init, s.cam_idx, s.pt_idx, orc.pixels_from_scene(s)) for s in (sc, base)]
    st = []
    for precision in ("f32", "f64"):
        opts = ba.Options(precision=precision, huber_delta=huber, pcg_maxiter=10, pcg_tol=0.0, lambda0=1e-2)
        with ba.Batch(inputs, opts) as batch:
            batch.solve(1)
            st.append([s[0] for s in batch.stats()])
    for a, b in zip(*st):
        drop = b["cost"] - b["cost_trial"]
        assert drop > 0 and a["pcg_iters"] == b["pcg_iters"] == 10
        assert abs(a["cost_trial"] - b["cost_trial"]) < 1e-4 * drop
        assert abs(a["model"] - b["model"]) < 1e-4 * abs(b["model"])


def test_formed_systems_are_as_accurate_as_the_implicit_product():
    """Three trials of 48 windows from FP32-rounded inputs: the cameras'
    distance from the FP64 batch, formed (recomputed Jacobians) against the
    implicit product (stored ones).  Both round per observation; what the formed
    system adds must stay below that: 1.5 times, over all windows."""
    rng = np.random.default_rng(5)
    inputs = []
    for k in range(48):
        C = int(rng.integers(5, 21))
        sc = scenegen.arc_scene(C, int(rng.integers(200, 900)), seed=100 + k, views_lo=4, views_hi=min(C, 10))
        pix = orc.pixels_from_scene(sc)
        inputs.append([np.asarray(a, np.float32) for a in (sc.cams_init, sc.points_init)] + [sc.cam_idx, sc.pt_idx]
                      + [np.asarray(pix, np.float32)])
    cams = {}
    for precision, jacobian in (("f64", "store"), ("f32", "store"), ("f32", "recompute")):
        opts = ba.Options(precision=precision, jacobian=jacobian, pcg_maxiter=10, pcg_tol=0.0)
        with ba.Batch(inputs, opts) as batch:
            batch.solve(3)
            cams[precision, jacobian] = batch.params(split=False)[0].cpu().double().numpy()
    exact = cams["f64", "store"]
    err = {j: np.linalg.norm(cams["f32", j] - exact) / np.linalg.norm(exact) for j in ("store", "recompute")}
    assert err["recompute"] < 1.5 * err["store"], err
