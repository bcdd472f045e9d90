"""What a problem whose reduced system is formed keeps for its implicit
products (ba_schur_matvec, a part of a partitioned problem)."""
import numpy as np
import pytest
import torch

import oracle as orc
import paper_2409_12190_gb300 as ba
import scenegen
from gpu_helpers import np64, problem, rel_err, small_ring
from paper_2409_12190_gb300 import _lib
from paper_2409_12190_gb300.partition import PartProblem, exchange_cap

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


def _one_part(C=97, P=9000):
    sc = small_ring(C, P, seed=3)
    pix = orc.pixels_from_scene(sc)
    opts = ba.Options(precision="f64", pcg_maxiter=40, pcg_tol=0.0, huber_delta=sc.huber_delta)
    return sc, (sc.cams_init, sc.points_init, sc.cam_idx, sc.pt_idx, pix), opts


def test_a_part_holds_no_formed_system():
    """Made as a part, or made alone and then given an exchange: the implicit
    product, and the same trials (a sum over one part changes nothing).  Alone
    again: trials to rounding of those of the formed system (1e-9)."""
    sc, arrays, opts = _one_part()
    with ba.Problem(*arrays, opts, device="cuda") as alone:
        assert alone.layout()["formed"] == 1
        alone.solve(3)
        want = alone.stats()
    with PartProblem(*arrays, lambda t: None, opts, device="cuda") as part:
        lay = part.layout()
        assert lay["formed"] == 0 and lay["pieces"] == lay["product_pieces"]
        part.solve(3)
        a = part.stats()
        pa = [t.cpu() for t in part.params()]
    prob = ba.Problem(*arrays, opts, device="cuda")
    prob.solve(1)  # captured with the formed system
    xbuf = torch.zeros(exchange_cap(sc.C), dtype=torch.float64, device="cuda")
    fn = _lib.EXCHANGE_FN(lambda n, stream, ctx: 0)
    _lib.check(_lib.load().ba_set_exchange(prob._h, fn, None, xbuf.data_ptr(), xbuf.numel()))
    assert prob.layout()["formed"] == 0
    prob.set_params(torch.from_numpy(sc.cams_init), torch.from_numpy(sc.points_init))
    prob.set_lambda(opts.lambda0)
    prob.solve(3)
    b = prob.stats()[-3:]
    pb = [t.cpu() for t in prob.params()]
    _lib.check(_lib.load().ba_set_exchange(prob._h, _lib.EXCHANGE_FN(), None, None, 0))
    prob.set_params(torch.from_numpy(sc.cams_init), torch.from_numpy(sc.points_init))
    prob.set_lambda(opts.lambda0)
    prob.solve(3)
    c = prob.stats()[-3:]
    prob.close()
    for got in (a, b, c):
        assert [s["pcg_iters"] for s in got] == [s["pcg_iters"] for s in want]
        assert [s["accepted"] for s in got] == [s["accepted"] for s in want]
        for s, w in zip(got, want):
            assert abs(s["cost_trial"] - w["cost_trial"]) < 1e-9 * w["cost_trial"]
    for x, y in zip(pa, pb):
        assert rel_err(x.numpy(), y.numpy()) < 1e-9


def _large_ring(C, P, views, seed):
    """Points seen by `views` neighbouring cameras of a ring, on the GPU."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    f = dict(dtype=torch.float64, device="cuda")
    cams = torch.zeros(C, 9, **f)
    cams[:, 1] = -2 * np.pi * torch.arange(C, **f) / C
    cams[:, 5], cams[:, 6] = -5.0, 500.0
    pts = 2 * torch.rand(P, 3, generator=g, **f) - 1
    pi = torch.arange(P, device="cuda").repeat_interleave(views)
    ci = (torch.randint(0, C, (P,), generator=g, device="cuda")[:, None] + torch.arange(views, device="cuda")) % C
    ci, pi = ci.reshape(-1).int(), pi.int()
    pix = ba.project(cams, pts, ci, pi)
    pix = pix + torch.randn(pix.shape, generator=g, **f)
    return cams, pts + 0.01 * torch.randn(P, 3, generator=g, **f), ci, pi, pix


def test_a_problem_that_fits_only_unformed_is_made():
    """Memory for the problem with the implicit product, but not for the pairs
    and the lean form that the formed system has instead of the point-major
    planes: made without it."""
    arrays = _large_ring(250, 300000, 12, seed=1)
    opts = ba.Options(precision="f64", pcg_maxiter=30, pcg_tol=0.0)

    class Part(ba.Problem):
        _create = "ba_problem_create_part"

    def run(make):
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        with make(*arrays, opts, device="cuda") as prob:
            took = free - torch.cuda.mem_get_info()[0]
            formed = prob.layout()["formed"]
            prob.solve(1)
            out = [t.clone() for t in prob.params()]
        torch.cuda.synchronize()
        return took, formed, out

    for make in (Part, ba.Problem):
        run(make)  # loads what it needs
    torch.cuda.empty_cache()
    plain, formed_0, want = run(Part)
    formed, formed_1, _ = run(ba.Problem)
    assert (formed_0, formed_1) == (0, 1) and formed - plain > 64 << 20
    torch.cuda.empty_cache()
    filler = torch.empty(torch.cuda.mem_get_info()[0] - (plain + formed) // 2, dtype=torch.uint8, device="cuda")
    try:
        with ba.Problem(*arrays, opts, device="cuda") as prob:
            assert prob.layout()["formed"] == 0
            prob.solve(1)
            got = prob.params()
        assert all(torch.equal(a, b) for a, b in zip(got, want))
    finally:
        del filler
        torch.cuda.empty_cache()


@pytest.mark.parametrize("narrow", [False, True])
def test_single_precision_formed_system_is_as_accurate_as_the_implicit_product(narrow):
    """FP32 trials from FP32-rounded inputs on both routes: their distances from
    the FP64 answer, cameras and points, over 16 problems.  Wide: arcs of 6-36
    cameras, points seen by up to ten of them.  Narrow: rings of 100 whose points
    three neighbours see.  Both routes round per observation; forming S may add
    no more than their spread (15 % of the mean of 16)."""
    class Implicit(ba.Problem):
        _create = "ba_problem_create_part"

    f32 = lambda a: torch.as_tensor(a).float()
    ratios = []
    for seed in range(16):
        if narrow:
            cams, pts, ci, pi, pix = _large_ring(100, 12000, 3, seed=seed + 1)
        else:
            C = 6 + 2 * seed
            sc = scenegen.arc_scene(C, 40 * C, seed=seed, views_lo=4, views_hi=min(C, 10))
            cams, pts, ci, pi, pix = sc.cams_init, sc.points_init, sc.cam_idx, sc.pt_idx, orc.pixels_from_scene(sc)
        out = []
        for make, precision, formed in ((ba.Problem, "f64", None), (Implicit, "f32", 0), (ba.Problem, "f32", 1)):
            opts = ba.Options(precision=precision, pcg_maxiter=20, pcg_tol=0.0)
            with make(f32(cams), f32(pts), ci, pi, f32(pix), opts, device="cuda") as prob:
                assert formed is None or prob.layout()["formed"] == formed
                prob.solve(1)
                out.append([np64(t) for t in prob.params()])
        exact, implicit, form = out
        ratios.append([np.linalg.norm(f - e) / np.linalg.norm(i - e) for e, i, f in zip(exact, implicit, form)])
    mean = np.exp(np.log(ratios).mean(0))
    assert mean[0] < 1.15 and mean[1] < 1.15, mean


@pytest.mark.parametrize("maxiter,formed", [(1, 0), (10, 0), (20, 1), (250, 1)])
def test_the_formed_system_is_chosen_where_it_was_measured_to_pay(maxiter, formed):
    """1,000 cameras, 900,000 observations, 3.5 pairs each, FP64: a trial of 10
    iterations takes 1.05 times as long formed, one of 20 0.76 times."""
    opts = ba.Options(precision="f64", pcg_maxiter=maxiter, pcg_tol=0.0)
    with ba.Problem(*_large_ring(1000, 112500, 8, seed=2), opts, device="cuda") as prob:
        assert prob.layout()["formed"] == formed


@pytest.mark.parametrize("C,P", [(2, 5), (7, 33), (30, 700), (151, 900), (153, 1200), (310, 1500)])
def test_small_problems_take_the_formed_route(C, P):
    """The sizes at which the formed system is compared with the oracle do form
    it, in one launch for the whole PCG; the implicit product takes three an
    iteration."""
    sc = scenegen.arc_scene(C, P, seed=C, views_lo=1, views_hi=9)
    pix = orc.pixels_from_scene(sc)
    for precision in ("f64", "f32"):
        with problem(sc, pix, precision) as prob:
            assert prob.layout()["formed"] == 1
            prob.damped_solve(1e-2, 8, 0.0)
            torch.cuda.synchronize()
            n = ba.kernel_launch_count()
            prob.damped_solve(1e-2, 8, 0.0)
            assert ba.kernel_launch_count() - n < 20
    with problem(sc, pix, "f64", jacobian="recompute") as prob:
        assert prob.layout()["formed"] == 0
    with problem(sc, pix, "f64", solver="cholesky") as prob:
        assert prob.layout()["formed"] == 2


def test_windows_are_formed_in_single_precision():
    inputs = []
    for C in (2, 6, 20):
        sc = scenegen.arc_scene(C, 40 * C, seed=C, views_lo=2, views_hi=min(C, 6))
        inputs.append((sc.cams_init, sc.points_init, sc.cam_idx, sc.pt_idx, orc.pixels_from_scene(sc)))
    for precision, jacobian, formed in (("f32", "auto", True), ("f32", "store", False), ("f64", "auto", False)):
        with ba.Batch(inputs, ba.Options(precision=precision, jacobian=jacobian, pcg_maxiter=10)) as batch:
            assert batch.formed() == formed
