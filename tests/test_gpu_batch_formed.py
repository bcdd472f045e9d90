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
