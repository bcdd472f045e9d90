"""What a problem whose reduced system is formed keeps for its implicit
products (ba_schur_matvec, a part of a partitioned problem)."""
import numpy as np
import pytest
import torch

import oracle as orc
from gpu_helpers import np64, problem, rel_err, small_ring

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("C,P", [(40, 6000), (97, 9000)])
def test_product_keeps_its_long_pieces(C, P):
    """Short pieces fill the chip in a linearisation; every piece more is a
    reduction more in each product, which keeps runs of up to 2,048.  The
    product against the one with recomputed Jacobians (rounding: 1e-11)."""
    sc = small_ring(C, P, seed=C)
    pix = orc.pixels_from_scene(sc)
    x = torch.from_numpy(np.random.default_rng(1).normal(size=(C, 9)))
    with problem(sc, pix, "f64") as prob, problem(sc, pix, "f64", jacobian="recompute") as ref:
        lay = prob.layout()
        per_cam = np.bincount(sc.cam_idx, minlength=C)
        assert lay["product_pieces"] == np.sum(-(-per_cam // 2048)) < lay["pieces"]
        y = prob.schur_matvec(1e-3, x.cuda())
        assert rel_err(np64(y), np64(ref.schur_matvec(1e-3, x.cuda()))) < 1e-11
