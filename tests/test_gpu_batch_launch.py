"""The default launch of a batch: two CTAs an SM only where the batch gives
every SM about the largest window's observations or more (with one CTA an SM
that window bounds the batch, with two it takes longer)."""
import numpy as np
import pytest
import torch

import oracle as orc
import paper_2409_12190_gb300 as ba
import scenegen

pytestmark = pytest.mark.gpu


def _window(P, seed):
    sc = scenegen.arc_scene(4, P, seed=seed, views_lo=3, views_hi=3)
    return sc.cams_init, sc.points_init, sc.cam_idx, sc.pt_idx, orc.pixels_from_scene(sc)


@pytest.mark.parametrize("precision,jacobian,fill", [("f64", "store", 1.0), ("f64", "recompute", 1.3), ("f32", "store", 0.8)])
def test_two_ctas_an_sm_only_where_the_batch_fills_them(precision, jacobian, fill):
    nsm = torch.cuda.get_device_properties(0).multi_processor_count
    opts = ba.Options(precision=precision, jacobian=jacobian, pcg_maxiter=4, pcg_tol=0.0)
    small = _window(10, 1)

    def variant(n, largest):
        with ba.Batch([small] * (n - 1) + [_window(largest, 2)], opts) as b:
            return b.launch()["variant"]

    n = 3 * nsm  # windows of 10 points and one of `largest`: 3 (n - 1) / n x 10 / largest windows' worth an SM
    assert variant(n, 10) == 1
    assert variant(n, int(30 / fill * 0.9)) == 1
    assert variant(n, int(30 / fill * 1.2)) == 0
    assert variant(nsm, 10) == 0
