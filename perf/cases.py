"""What a user has this library do, as cases that can be timed and compared.

A case is one pass through the public entry points on a problem that the
user's program keeps: the start values go in, a few Levenberg-Marquardt trials
run, the parameters (or gradients) come out.  The scenes have the shapes of
the repository's seeded workloads (arcs and rings of cameras, sliding windows,
sphere and garage pose graphs), drawn on the GPU from the seed.

Kinds:
  lm       one bundle-adjustment problem, PCG or the direct solver
  adjoint  the differentiable solve: forward trials and the gradients
  steps    linearisation, product and damped solve, for a user with a loop of their own
  batch    many sliding windows in one launch
  pgo      a pose graph, PCG or banded Cholesky
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2409_12190_gb300 as ba

DEV = "cuda"
F64 = torch.float64


# ---------------------------------------------------------------------------
# The cases
# ---------------------------------------------------------------------------

def listed():
    return [
        # a 16-camera window of a tracker, one step per frame with the
        # library's default options: launches and latency count
        dict(name="lm16_f64", kind="lm", scene="arc", C=16, P=1000, views_lo=4, views_hi=12, precision="f64",
             huber=0.0, solver="pcg", maxiter=250, tol=1e-4, trials=1),
        # a small reconstruction in single precision, odd sizes, points of many views
        dict(name="lm97_f32", kind="lm", scene="ring", C=97, P=9001, views_min=3, mean_views=12.0, precision="f32",
             huber=0.0, solver="pcg", maxiter=20, tol=0.0, trials=2),
        # an ordinary reconstruction with outliers under a robust loss, the
        # library's default PCG limits
        dict(name="lm250_huber_f64", kind="lm", scene="ring", C=250, P=60000, views_min=2, mean_views=8.0,
             precision="f64", huber=1.0, solver="pcg", maxiter=250, tol=1e-4, trials=1),
        # the same scale, single precision, a fixed budget of PCG iterations
        dict(name="lm250_huber_f32", kind="lm", scene="ring", C=250, P=60000, views_min=3, mean_views=8.0,
             precision="f32", huber=1.0, solver="pcg", maxiter=20, tol=0.0, trials=1),
        # the explicit reduced camera system and its Cholesky factorisation
        dict(name="direct250_f64", kind="lm", scene="ring", C=250, P=60000, views_min=2, mean_views=8.0,
             precision="f64", huber=1.0, solver="cholesky", maxiter=50, tol=1e-4, trials=1),
        # city scale, double precision: the largest problem
        dict(name="lm4000_f64", kind="lm", scene="ring", C=4000, P=1200000, views_min=2, mean_views=6.7,
             precision="f64", huber=0.0, solver="pcg", maxiter=50, tol=1e-4, trials=2),
        # city scale, single precision
        dict(name="lm4000_f32", kind="lm", scene="ring", C=4000, P=1200000, views_min=3, mean_views=6.7,
             precision="f32", huber=0.0, solver="pcg", maxiter=30, tol=0.0, trials=2),
        # gradients through the solve with respect to the observed pixels (a
        # learned front end): forward trials, then the adjoint to its default tolerance
        dict(name="adjoint64_f64", kind="adjoint", scene="ring", C=64, P=10000, views_min=2, mean_views=8.0,
             precision="f64", huber=0.0, maxiter=30, tol=1e-4, trials=4),
        # a user's own outer loop on a ragged problem: the blocks of one
        # linearisation, one product with the reduced system, one damped solve
        dict(name="steps321_f64", kind="steps", scene="ring", C=321, P=45677, views_min=2, mean_views=9.0,
             precision="f64", huber=0.0, maxiter=30, tol=0.0),
        # 512 sliding windows of uneven size at once, ten PCG iterations a trial
        dict(name="batch512_f32", kind="batch", n=512, c_lo=5, c_hi=20, p_lo=200, p_hi=3000, precision="f32",
             maxiter=10, tol=0.0, trials=3),
        # a loop-closed trajectory, iterative solver
        dict(name="pgo2500_pcg", kind="pgo", graph="sphere", rings=50, per=50, solver="pcg", maxiter=100, tol=1e-4,
             trials=2),
        # a parking-garage drive, direct solver
        dict(name="pgo1661_chol", kind="pgo", graph="garage", rings=11, per=151, solver="cholesky", maxiter=100,
             tol=1e-4, trials=2),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["lm", "lm", "lm", "lm", "direct", "adjoint", "steps", "batch", "pgo", "pgo"])
    if kind == "batch":
        return dict(kind="batch", n=_logint(rng, 40, 512), c_lo=rng.randint(4, 7), c_hi=rng.randint(8, 24),
                    p_lo=_logint(rng, 60, 250), p_hi=_logint(rng, 500, 3000), precision="f32",
                    maxiter=rng.randint(6, 10), tol=0.0, trials=rng.randint(1, 3))
    if kind == "pgo":
        return dict(kind="pgo", graph=rng.choice(["sphere", "garage"]), rings=rng.randint(8, 50),
                    per=rng.randint(10, 50), solver=rng.choice(["pcg", "cholesky"]), maxiter=rng.randint(50, 100),
                    tol=1e-4, trials=rng.randint(1, 3))
    c = dict(kind="lm" if kind == "direct" else kind)
    c["precision"] = rng.choice(["f64", "f64", "f32"]) if kind == "lm" else "f64"
    if kind == "lm" and rng.random() < 0.25:
        lo = rng.randint(3, 5)
        c.update(scene="arc", C=rng.randint(6, 60), P=_logint(rng, 300, 6000), views_lo=lo,
                 views_hi=rng.randint(lo + 1, 14))
    else:
        C = _logint(rng, 24, {"lm": 4000, "direct": 300, "adjoint": 200, "steps": 1500}[kind])
        per = _logint(rng, 100, 300)  # points per camera
        c.update(scene="ring", C=C, P=C * per + rng.randint(0, per), views_min=3 if c["precision"] == "f32" else 2,
                 mean_views=round(rng.uniform(4.5, 6.7 if C > 2000 else 12.0), 1))
    if kind == "steps":
        return dict(c, huber=0.0, maxiter=rng.randint(10, 30), tol=0.0)
    if kind == "adjoint":
        return dict(c, huber=0.0, maxiter=rng.randint(20, 30), tol=1e-4, trials=rng.randint(3, 5))
    c["huber"] = rng.choice([0.0, 1.0])
    c["solver"] = "cholesky" if kind == "direct" else "pcg"
    if c["precision"] == "f32":
        return dict(c, maxiter=rng.randint(10, 25) if c["scene"] == "ring" else rng.randint(6, 10), tol=0.0, trials=1)
    c["trials"] = 1 if kind == "direct" or c["huber"] > 0 else rng.randint(1, 2)
    c.update(maxiter=rng.choice([50, 250]) if c["trials"] == 1 and c["C"] <= 1000 else 50 if c["C"] > 200 else 20,
             tol=1e-4)
    return c


# ---------------------------------------------------------------------------
# Scenes, drawn on the GPU (FP64)
# ---------------------------------------------------------------------------

def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed) * 7919 + 17)


def _randn(g, *shape):
    return torch.randn(*shape, generator=g, device=DEV, dtype=F64)


def _rand(g, *shape):
    return torch.rand(*shape, generator=g, device=DEV, dtype=F64)


def _skew(w):
    z = torch.zeros_like(w[..., 0])
    return torch.stack([z, -w[..., 2], w[..., 1], w[..., 2], z, -w[..., 0], -w[..., 1], w[..., 0], z],
                       -1).reshape(*w.shape[:-1], 3, 3)


def _rotation(w):
    """Rodrigues' formula, batched."""
    t2 = (w * w).sum(-1)
    t = t2.sqrt()
    a = torch.where(t < 1e-4, 1 - t2 / 6, torch.sin(t) / t.clamp_min(1e-300))
    b = torch.where(t < 1e-4, 0.5 - t2 / 24, 2 * torch.sin(0.5 * t) ** 2 / t2.clamp_min(1e-300))
    K = _skew(w)
    return torch.eye(3, dtype=w.dtype, device=w.device) + a[..., None, None] * K + b[..., None, None] * (K @ K)


def _project(cams, pts, ci, pi):
    c = cams[ci]
    X = (_rotation(cams[:, :3])[ci] @ pts[pi][..., None])[..., 0] + c[:, 3:6]
    p = -X[:, :2] / X[:, 2:]
    r2 = (p * p).sum(-1, keepdim=True)
    return c[:, 6:7] * (1 + r2 * (c[:, 7:8] + c[:, 8:9] * r2)) * p


def _ring(C, P, views_min, mean_views, g):
    """Cameras on a full ring facing a cloud of points, each point seen by a
    window of views_min + Geom0 neighbouring cameras (mean mean_views)."""
    phi = 2 * math.pi * torch.arange(C, device=DEV, dtype=F64) / C
    phi = torch.where(phi > math.pi, phi - 2 * math.pi, phi)
    cams = torch.zeros(C, 9, device=DEV, dtype=F64)
    cams[:, 1] = -phi
    cams[:, :3] += 0.02 * _randn(g, C, 3)
    cams[:, 5] = -5.0
    cams[:, 6] = 500.0
    cams[:, 7:] = 1e-3 * _randn(g, C, 2)
    pts = 2 * _rand(g, P, 3) - 1
    q = 1.0 / (mean_views - views_min + 1.0)  # Geom0(q) has the mean (1 - q) / q
    # the same number of points of each count for every seed, in another order
    u = (torch.randperm(P, generator=g, device=DEV).to(F64) + 0.5) / P
    n = (views_min + torch.floor(torch.log(u) / math.log(1 - q)).long()).clamp(max=C)
    start = torch.randint(0, C, (P,), generator=g, device=DEV)
    pi = torch.repeat_interleave(torch.arange(P, device=DEV), n)
    m = torch.arange(pi.shape[0], device=DEV) - (torch.cumsum(n, 0) - n)[pi]
    ci = (start[pi] + m) % C
    return cams, pts, ci, pi


def _arcs(Cs, Ps, views_lo, views_hi, g):
    """Arcs of cameras in front of a point cloud, one per entry of Cs / Ps;
    each point is seen by a random subset of its arc's cameras.  Concatenated,
    with indices local to each arc; prob is the arc of each observation."""
    dev = dict(device=DEV)
    Ct, Pt = torch.tensor(Cs, **dev), torch.tensor(Ps, **dev)
    nc, cmax = int(Ct.sum()), max(Cs)
    coff = torch.cumsum(Ct, 0) - Ct
    cprob = torch.repeat_interleave(torch.arange(len(Cs), **dev), Ct)
    k = (torch.arange(nc, **dev) - coff[cprob]).to(F64)
    cams = torch.zeros(nc, 9, dtype=F64, **dev)
    cams[:, 1] = -0.3 + 0.6 * k / (Ct[cprob] - 1).clamp_min(1).to(F64)
    cams[:, :3] += 0.02 * _randn(g, nc, 3)
    cams[:, 3:5] = _randn(g, nc, 2)
    cams[:, 5] = -5.0
    cams[:, 6] = 500.0
    cams[:, 7:] = 1e-3 * _randn(g, nc, 2)
    npt = int(Pt.sum())
    pprob = torch.repeat_interleave(torch.arange(len(Ps), **dev), Pt)
    pts = 2 * _rand(g, npt, 3) - 1
    hi = Ct[pprob].clamp(max=views_hi)
    lo = hi.clamp(max=views_lo)
    poff = torch.cumsum(Pt, 0) - Pt
    # each arc has every count equally often, whatever the seed
    u = (torch.arange(npt, **dev) - poff[pprob]).to(F64) + 0.5
    n = lo + torch.floor(u / Pt[pprob].to(F64) * (hi - lo + 1).to(F64)).long().clamp(max=hi - lo)
    score = torch.rand(npt, cmax, generator=g, **dev)
    score.masked_fill_(torch.arange(cmax, **dev)[None, :] >= Ct[pprob][:, None], 2.0)
    order = torch.argsort(score, dim=1)
    take = torch.arange(cmax, **dev)[None, :] < n[:, None]
    pid = torch.arange(npt, **dev)[:, None].expand(-1, cmax)[take]
    ci = order[take]
    prob = pprob[pid]
    return cams, pts, ci, pid - poff[prob], prob, coff, poff


def _scene(case, seed):
    """(cams, points, cam_idx, pt_idx, pixels, cams0, points0), observations in
    random order."""
    g = _gen(seed)
    if case["scene"] == "ring":
        cams, pts, ci, pi = _ring(case["C"], case["P"], case["views_min"], case["mean_views"], g)
    else:
        cams, pts, ci, pi = _arcs([case["C"]], [case["P"]], case["views_lo"], case["views_hi"], g)[:4]
    o = torch.randperm(ci.shape[0], generator=g, device=DEV)
    ci, pi = ci[o], pi[o]
    noise = _randn(g, ci.shape[0], 2)
    if case.get("huber", 0.0) > 0:
        out = _rand(g, ci.shape[0]) < 0.02
        psi = 2 * math.pi * _rand(g, ci.shape[0])
        noise += 20.0 * out.to(F64)[:, None] * torch.stack([torch.cos(psi), torch.sin(psi)], -1)
    pix = _project(cams, pts, ci, pi) + noise
    # a start as a front end leaves it: a few pixels off
    cams0, pts0 = cams.clone(), pts + 0.01 * _randn(g, *pts.shape)
    cams0[:, :3] += 0.004 * _randn(g, cams.shape[0], 3)
    cams0[:, 3:6] += 0.01 * _randn(g, cams.shape[0], 3)
    return ci.int(), pi.int(), pix, cams0, pts0, g


def _dtype(case):
    return torch.float32 if case["precision"] == "f32" else F64


# ---------------------------------------------------------------------------
# Pose graphs
# ---------------------------------------------------------------------------

def _qmul(a, b):
    ax, ay, az, aw = a.unbind(-1)
    bx, by, bz, bw = b.unbind(-1)
    return torch.stack([aw * bx + ax * bw + ay * bz - az * by, aw * by - ax * bz + ay * bw + az * bx,
                        aw * bz + ax * by - ay * bx + az * bw, aw * bw - ax * bx - ay * by - az * bz], -1)


def _qrot(q):
    x, y, z, w = q.unbind(-1)
    return torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - z * w), 2 * (x * z + y * w), 2 * (x * y + z * w),
                        1 - 2 * (x * x + z * z), 2 * (y * z - x * w), 2 * (x * z - y * w), 2 * (y * z + x * w),
                        1 - 2 * (x * x + y * y)], -1).reshape(*q.shape[:-1], 3, 3)


def _qconj(q):
    return q * torch.tensor([-1.0, -1, -1, 1], dtype=q.dtype, device=q.device)


def _mv(M, v):
    return (M @ v[..., None])[..., 0]


# coefficients B_2k / (2k)! of x / (e^x - 1) (x/2 handled apart)
_BERN = [1.0 / 12, -1.0 / 720, 1.0 / 30240, -1.0 / 1209600, 1.0 / 47900160, -691.0 / 1307674368000,
         1.0 / 74724249600, -3617.0 / 10670622842880000, 43867.0 / 5109094217170944000]


def _jlinv(ad):
    """Inverse left Jacobian from the adjoint matrix of the tangent vector."""
    I = torch.eye(ad.shape[-1], dtype=ad.dtype, device=ad.device)
    a2 = ad @ ad
    S, pw = I - 0.5 * ad, a2
    for b in _BERN:
        S = S + b * pw
        pw = pw @ a2
    return S


def _jl(ad):
    I = torch.eye(ad.shape[-1], dtype=ad.dtype, device=ad.device).expand_as(ad)
    S, pw = I, I
    for n in range(1, 24):
        pw = pw @ ad / (n + 1)
        S = S + pw
    return S


def _se3_exp(d, P):
    """Exp(d) P for tangents (translation, rotation) and poses (t, q)."""
    t = d[..., 3:].norm(dim=-1, keepdim=True)
    s = torch.where(t < 1e-4, 0.5 - t * t / 48, torch.sin(0.5 * t) / t.clamp_min(1e-300))
    q = _qmul(torch.cat([s * d[..., 3:], torch.cos(0.5 * t)], -1), P[..., 3:])
    q = q / q.norm(dim=-1, keepdim=True)
    q = torch.where(q[..., 3:] < 0, -q, q)
    return torch.cat([_mv(_rotation(d[..., 3:]), P[..., :3]) + _mv(_jl(_skew(d[..., 3:])), d[..., :3]), q], -1)


def _mul_inv(A, B):
    """A^{-1} B of poses."""
    R = _qrot(A[..., 3:]).transpose(-1, -2)
    return torch.cat([_mv(R, B[..., :3] - A[..., :3]), _qmul(_qconj(A[..., 3:]), B[..., 3:])], -1)


def _graph(case, seed):
    """(poses0, ei, ej, meas, info): a sphere of rings or a garage of laps, odometry
    edges and loop closures to the neighbours one ring or lap away."""
    g = _gen(seed)
    R, M = case["rings"], case["per"]
    N = R * M
    k = torch.arange(N, device=DEV)
    r, m = (k // M).to(F64), (k % M).to(F64)
    if case["graph"] == "sphere":
        lat, yaw0 = -0.5 * math.pi + math.pi * (r + 0.5) / R, 2 * math.pi * m / M
        rad = float(R)
        pos = rad * torch.stack([lat.cos() * yaw0.cos(), lat.cos() * yaw0.sin(), lat.sin()], -1)
        yaw, pitch = yaw0 + 0.5 * math.pi, -lat
        offs, st, sr, dt, dr = (-1, 0, 1), 0.05, 0.01, 0.02, 0.004
    else:
        s = 4.0 * m / M
        side = torch.floor(s)
        f = (s - side)[:, None]
        corner = 40.0 * torch.tensor([[0.0, 0], [1, 0], [1, 1], [0, 1], [0, 0]], dtype=F64, device=DEV)
        c0, c1 = corner[side.long()], corner[side.long() + 1]
        pos = torch.cat([c0 + f * (c1 - c0), (3.0 * k / M)[:, None].to(F64)], -1)
        yaw, pitch = 0.5 * math.pi * side, torch.full((N,), -math.atan2(3.0, 160.0), dtype=F64, device=DEV)
        offs, st, sr, dt, dr = (-2, -1, 0, 1, 2), 0.02, 0.005, 0.01, 0.002
    sz, cz, sy, cy = (0.5 * yaw).sin(), (0.5 * yaw).cos(), (0.5 * pitch).sin(), (0.5 * pitch).cos()
    poses = torch.cat([pos, torch.stack([-sz * sy, cz * sy, sz * cy, cz * cy], -1)], -1)
    a = torch.arange(N - M, device=DEV)
    if case["graph"] == "sphere":
        cand = torch.cat([torch.stack([a, (a // M + 1) * M + (a % M + d) % M], -1) for d in offs])
    else:
        cand = torch.cat([torch.stack([a + d, a + M], -1)[(a + d >= 0) & (a + d < a + M - 1)] for d in offs])
    keep = torch.rand(cand.shape[0], generator=g, device=DEV) < 0.99
    e = torch.cat([torch.stack([torch.arange(N - 1, device=DEV), torch.arange(1, N, device=DEV)], -1), cand[keep]])
    sig = torch.tensor([st] * 3 + [sr] * 3, dtype=F64, device=DEV)
    z = _randn(g, e.shape[0], 6) * sig
    meas = _se3_exp(z, _mul_inv(poses[e[:, 0]], poses[e[:, 1]]))
    info = torch.zeros(e.shape[0], 21, dtype=F64, device=DEV)
    info[:, [0, 6, 11, 15, 18, 20]] = 1.0 / (sig * sig)
    step = _randn(g, N, 6) * torch.tensor([dt] * 3 + [dr] * 3, dtype=F64, device=DEV)
    step[0] = 0
    return _se3_exp(torch.cumsum(step, 0), poses), e[:, 0].int(), e[:, 1].int(), meas, info


# ---------------------------------------------------------------------------
# prepare, run
# ---------------------------------------------------------------------------

def _options(case):
    o = ba.Options(precision=case.get("precision", "f64"), huber_delta=case.get("huber", 0.0),
                   pcg_maxiter=case["maxiter"], pcg_tol=case["tol"], solver=case.get("solver", "pcg"))
    return o


def _windows(case, seed):
    # the same windows' sizes for every seed, in another order
    r = np.random.default_rng(9)
    Cs = r.integers(case["c_lo"], case["c_hi"] + 1, case["n"])
    Ps = np.exp(r.uniform(math.log(case["p_lo"]), math.log(case["p_hi"]), case["n"])).round().astype(int)
    o = np.random.default_rng(int(seed)).permutation(case["n"])
    Cs, Ps = Cs[o].tolist(), Ps[o].tolist()
    g = _gen(seed)
    cams, pts, ci, pi, prob, coff, poff = _arcs(Cs, Ps, 4, 10, g)
    pix = _project(cams, pts, ci + coff[prob], pi + poff[prob]) + _randn(g, ci.shape[0], 2)
    c0, p0 = cams.clone(), pts + 0.01 * _randn(g, *pts.shape)
    c0[:, :3] += 0.004 * _randn(g, cams.shape[0], 3)
    c0[:, 3:6] += 0.01 * _randn(g, cams.shape[0], 3)
    return Cs, Ps, ci.int(), pi.int(), pix, c0, p0, prob


def prepare(case, seed):
    kind = case["kind"]
    if kind == "pgo":
        poses0, ei, ej, meas, info = _graph(case, seed)
        return dict(kind=kind, case=case, poses0=poses0,
                    graph=ba.PoseGraph(poses0, ei, ej, meas, info, options=_options(case)))
    if kind == "batch":
        Cs, Ps, ci, pi, pix, c0, p0, prob = _windows(case, seed)
        dt = _dtype(case)
        c0, p0, pix = c0.to(dt), p0.to(dt), pix.to(dt)
        Os = torch.bincount(prob.cpu(), minlength=len(Cs)).tolist()
        parts = [torch.split(t, n) for t, n in ((c0, Cs), (p0, Ps), (ci, Os), (pi, Os), (pix, Os))]
        return dict(kind=kind, case=case, c0=c0, p0=p0, batch=ba.Batch(list(zip(*parts)), _options(case)))
    ci, pi, pix, c0, p0, g = _scene(case, seed)
    dt = _dtype(case)
    c0, p0, pix = c0.to(dt), p0.to(dt), pix.to(dt)
    s = dict(kind=kind, case=case, c0=c0, p0=p0, pix=pix, prob=ba.Problem(c0, p0, ci, pi, pix, _options(case)))
    if kind == "steps":
        s["x"] = _randn(g, case["C"], 9)
    if kind == "adjoint":
        mask = torch.zeros(case["C"], 9, dtype=torch.bool, device=DEV)
        mask[0] = True
        mask[case["C"] // 2, 3:6] = True
        s["prob"].set_fixed(mask)
        s["gc"], s["gp"] = _randn(g, case["C"], 9).to(dt), _randn(g, case["P"], 3).to(dt)
    return s


def run(s):
    case = s["case"]
    if s["kind"] == "lm":
        p = s["prob"]
        p.set_params(s["c0"], s["p0"])
        p.set_lambda(1e-4)
        p.solve(case["trials"])
        return p.params()
    if s["kind"] == "adjoint":
        pix = s["pix"].detach().requires_grad_()
        cams, pts = ba.bundle_adjust(pix, s["c0"], s["p0"], s["prob"], case["trials"], lam=1e-4)
        torch.autograd.backward((cams, pts), (s["gc"], s["gp"]))
        return cams.detach(), pts.detach(), pix.grad
    if s["kind"] == "steps":
        lin = s["prob"].linearize(blocks=True, jacobians=False)
        y = s["prob"].schur_matvec(1e-4, s["x"])
        dc, dp, _, rel = s["prob"].damped_solve(1e-4, case["maxiter"], case["tol"])
        return dict(lin, y=y, dc=dc, dp=dp, rel=rel)
    if s["kind"] == "batch":
        b = s["batch"]
        b.reset()
        b.solve(case["trials"])
        return b.params(split=False)
    gr = s["graph"]
    gr.set_poses(s["poses0"])
    gr.set_lambda(1e-4)
    gr.solve(case["trials"])
    return gr.poses()


# ---------------------------------------------------------------------------
# work: what a pass cannot do without
# ---------------------------------------------------------------------------

def work(case):
    """Bytes: the inputs read once and the outputs written once.  Flops: the
    residuals, Jacobians and normal-equation blocks of each trial (about 500
    per observation, 1,500 per pose-graph edge)."""
    if case["kind"] == "pgo":
        N = case["rings"] * case["per"]
        E = N + (3 if case["graph"] == "sphere" else 5) * (N - case["per"])
        return dict(bytes=E * (8 + 28 * 8) + 2 * N * 56, flops=1500.0 * E * case["trials"])
    b = 4 if case["precision"] == "f32" else 8
    if case["kind"] == "batch":
        C = case["n"] * 0.5 * (case["c_lo"] + case["c_hi"])
        P = case["n"] * (case["p_hi"] - case["p_lo"]) / math.log(case["p_hi"] / case["p_lo"])
        views = 6.5
    else:
        C, P = case["C"], case["P"]
        views = case["mean_views"] if case["scene"] == "ring" else 0.5 * (case["views_lo"] + min(case["views_hi"], C))
    obs = P * views
    out = 2 * (9 * C + 3 * P) * b
    if case["kind"] == "adjoint":
        out += 2 * obs * b
    if case["kind"] == "steps":
        out += (90 * C + 12 * P) * 8
    return dict(bytes=obs * (8 + 2 * b) + out, flops=500.0 * obs * case.get("trials", 1))


# ---------------------------------------------------------------------------
# exact: the same, in 64 bits, with torch alone
# ---------------------------------------------------------------------------

class _Normal:
    """The normal equations of bundle adjustment at (cams, pts)."""

    def __init__(self, cams, pts, ci, pi, pix, huber):
        self.ci, self.pi, self.C, self.P = ci, pi, cams.shape[0], pts.shape[0]
        w = cams[:, :3]
        t2 = (w * w).sum(-1)
        t = t2.sqrt()
        K = _skew(w)
        b = torch.where(t < 1e-4, 0.5 - t2 / 24, 2 * torch.sin(0.5 * t) ** 2 / t2.clamp_min(1e-300))
        c = torch.where(t < 0.1, 1 / 6 - t2 * (1 / 120 - t2 * (1 / 5040 - t2 / 362880)),
                        (t - torch.sin(t)) / (t2 * t).clamp_min(1e-300))
        Jl = torch.eye(3, dtype=F64, device=DEV) + b[:, None, None] * K + c[:, None, None] * (K @ K)
        R = _rotation(w)
        RX = _mv(R[ci], pts[pi])
        X = RX + cams[ci, 3:6]
        f, k1, k2 = (cams[ci, i] for i in (6, 7, 8))
        p = -X[:, :2] / X[:, 2:]
        r2 = (p * p).sum(-1)
        d = 1 + r2 * (k1 + k2 * r2)
        r = (f * d)[:, None] * p - pix
        sq = (r * r).sum(-1)
        n = sq.sqrt()
        self.sw = torch.ones_like(n)
        if huber > 0:
            self.sw = torch.where(n > huber, (huber / n.clamp_min(1e-300)).sqrt(), self.sw)
        dp = torch.zeros(*ci.shape, 2, 3, dtype=F64, device=DEV)
        dp[:, 0, 0] = dp[:, 1, 1] = -1 / X[:, 2]
        dp[:, :, 2] = -p / X[:, 2:]
        M = (f * d)[:, None, None] * torch.eye(2, dtype=F64, device=DEV) + \
            (f * (2 * k1 + 4 * k2 * r2))[:, None, None] * p[:, :, None] * p[:, None, :]
        A = self.sw[:, None, None] * (M @ dp)
        D = self.sw[:, None, None] * p[:, :, None] * torch.stack([d, f * r2, f * r2 * r2], -1)[:, None, :]
        self.Jc = torch.cat([-A @ _skew(RX) @ Jl[ci], A, D], -1)
        self.Jp = A @ R[ci]
        self.r = self.sw[:, None] * r
        self.U = self._cam(self.Jc.transpose(1, 2) @ self.Jc)
        self.V = self._pt(self.Jp.transpose(1, 2) @ self.Jp)
        self.gc = self._cam(_mv(self.Jc.transpose(1, 2), self.r))
        self.gp = self._pt(_mv(self.Jp.transpose(1, 2), self.r))

    def _cam(self, v):
        return torch.zeros(self.C, *v.shape[1:], dtype=F64, device=DEV).index_add_(0, self.ci, v)

    def _pt(self, v):
        return torch.zeros(self.P, *v.shape[1:], dtype=F64, device=DEV).index_add_(0, self.pi, v)

    @staticmethod
    def _damped(B, lam):
        return B + torch.diag_embed(lam[:, None] * torch.diagonal(B, dim1=-2, dim2=-1).clamp(1e-6, 1e32))

    def damp(self, lamc, lamp, fixed=None):
        self.Us, self.Vi = self._damped(self.U, lamc), torch.linalg.inv(self._damped(self.V, lamp))
        self.free = torch.ones(self.C, 9, dtype=F64, device=DEV) if fixed is None else (~fixed).to(F64)
        J = self.Jp @ self.Vi[self.pi] @ self.Jp.transpose(1, 2)
        S = self.Us - self._cam(self.Jc.transpose(1, 2) @ J @ self.Jc)
        f = self.free
        self.M = torch.linalg.inv(S * f[:, :, None] * f[:, None, :] + torch.diag_embed(1 - f))

    def WT(self, x):
        return self._pt(_mv(self.Jp.transpose(1, 2), _mv(self.Jc, x[self.ci])))

    def W(self, y):
        return self._cam(_mv(self.Jc.transpose(1, 2), _mv(self.Jp, y[self.pi])))

    def product(self, x):
        return (_mv(self.Us, x) - self.W(_mv(self.Vi, self.WT(x)))) * self.free

    def rhs(self, gc, gp):
        return (-gc + self.W(_mv(self.Vi, gp))) * self.free

    def back(self, x, gp):
        return -_mv(self.Vi, gp + self.WT(x))

    def pcg(self, b, maxiter, tol, win, nwin):
        """Each window (one for a single problem) with scalars of its own."""
        def dot(u, v):
            return torch.zeros(nwin, dtype=F64, device=DEV).index_add_(0, win, (u * v).sum(-1))

        x, r = torch.zeros_like(b), b.clone()
        z = _mv(self.M, r)
        p, rz, bb = z.clone(), dot(r, z), dot(b, b)
        rel, on = torch.ones_like(bb), torch.ones_like(bb)
        for _ in range(maxiter):
            q = self.product(p)
            pq = dot(p, q)
            on = on * (pq > 0)
            al = torch.where(on > 0, rz / pq, torch.zeros_like(pq))[win][:, None]
            x, r = x + al * p, r - al * q
            rel = torch.where(on > 0, (dot(r, r) / bb).sqrt(), rel)
            on = on * (rel > tol)
            if not float(on.sum()):
                break
            z = _mv(self.M, r)
            rz, old = dot(r, z), rz
            p = z + (rz / old)[win][:, None] * p
        return x, rel

    def dense(self):
        """The reduced system as one matrix, a slice of points at a time."""
        n = 9 * self.C
        S = torch.block_diag(*self.Us) if self.C <= 64 else torch.zeros(n, n, dtype=F64, device=DEV)
        if self.C > 64:
            S.view(self.C, 9, self.C, 9)[torch.arange(self.C), :, torch.arange(self.C), :] = self.Us
        Wk = self.Jc.transpose(1, 2) @ self.Jp
        Lv = torch.linalg.cholesky(self.Vi)
        Yk = Wk @ Lv[self.pi]
        step = 20000
        for a in range(0, self.P, step):
            sel = (self.pi >= a) & (self.pi < a + step)
            E = torch.zeros(n, 3 * step, dtype=F64, device=DEV)
            rows = (9 * self.ci[sel])[:, None, None] + torch.arange(9, device=DEV)[None, :, None]
            cols = (3 * (self.pi[sel] - a))[:, None, None] + torch.arange(3, device=DEV)[None, None, :]
            E[rows.expand(-1, 9, 3), cols.expand(-1, 9, 3)] = Yk[sel]
            S -= E @ E.T
        f = self.free.reshape(-1)
        return S * f[:, None] * f[None, :] + torch.diag(1 - f)


def _lm(cams, pts, ci, pi, pix, case, trials, fixed=None, cwin=None, pwin=None, nwin=1):
    """The LM trials, window by window (one window for a single problem)."""
    huber = case.get("huber", 0.0)
    cwin = torch.zeros(cams.shape[0], dtype=torch.long, device=DEV) if cwin is None else cwin
    pwin = torch.zeros(pts.shape[0], dtype=torch.long, device=DEV) if pwin is None else pwin
    owin = cwin[ci]

    def total(win, v):
        return torch.zeros(nwin, dtype=F64, device=DEV).index_add_(0, win, v)

    def cost(cams, pts):
        n = (_project(cams, pts, ci, pi) - pix).norm(dim=-1)
        h = 0.5 * n * n
        if huber > 0:
            h = torch.where(n > huber, huber * n - 0.5 * huber * huber, h)
        return total(owin, h)

    F, lam = cost(cams, pts), torch.full((nwin,), 1e-4, dtype=F64, device=DEV)
    for _ in range(trials):
        lin = _Normal(cams, pts, ci, pi, pix, huber)
        lin.damp(lam[cwin], lam[pwin], fixed)
        b = lin.rhs(lin.gc, lin.gp)
        if case.get("solver") == "cholesky":
            L = torch.linalg.cholesky(lin.dense())
            x = torch.cholesky_solve(b.reshape(-1, 1), L).reshape(-1, 9)
        else:
            x, _ = lin.pcg(b, case["maxiter"], case["tol"], cwin, nwin)
        dp = lin.back(x, lin.gp)
        e = _mv(lin.Jc, x[ci]) + _mv(lin.Jp, dp[pi])
        model = -total(cwin, (lin.gc * x).sum(-1)) - total(pwin, (lin.gp * dp).sum(-1)) \
            - 0.5 * total(owin, (e * e).sum(-1))
        Ft = cost(cams + x, pts + dp)
        rho = (F - Ft) / model
        ok = torch.isfinite(Ft) & (model > 0) & (Ft < F)
        cams = torch.where(ok[cwin][:, None], cams + x, cams)
        pts = torch.where(ok[pwin][:, None], pts + dp, pts)
        F = torch.where(ok, Ft, F)
        lam = torch.where(~ok | (rho < 0.25), (lam / 0.0625).clamp(max=1e32),
                          torch.where(rho > 0.75, (lam / 2.0).clamp(min=1e-16), lam))
    return cams, pts


def _se3_ad(xi):
    ad = torch.zeros(*xi.shape[:-1], 6, 6, dtype=F64, device=DEV)
    ad[..., :3, :3] = ad[..., 3:, 3:] = _skew(xi[..., 3:])
    ad[..., :3, 3:] = _skew(xi[..., :3])
    return ad


def _residual(Z, ei, ej, meas):
    T = _mul_inv(Z[ei], Z[ej])
    qm = _qconj(meas[:, 3:])
    q = _qmul(T[:, 3:], qm)
    t = T[:, :3] - _mv(_qrot(q), meas[:, :3])
    q = torch.where(q[:, 3:] < 0, -q, q)
    s = q[:, :3].norm(dim=-1, keepdim=True)
    phi = torch.where(s < 1e-9, 2.0 / q[:, 3:], 2 * torch.atan2(s, q[:, 3:]) / s.clamp_min(1e-300)) * q[:, :3]
    return torch.cat([_mv(_jlinv(_skew(phi)), t), phi], -1)


def _pgo_exact(case, seed):
    Z, ei, ej, meas, info = _graph(case, seed)
    ei, ej = ei.long(), ej.long()
    N, lam = Z.shape[0], 1e-4
    Om = torch.zeros(len(ei), 6, 6, dtype=F64, device=DEV)
    iu = np.triu_indices(6)
    Om[:, iu[0], iu[1]] = info
    Om[:, iu[1], iu[0]] = info
    free = torch.ones(N, 1, dtype=F64, device=DEV)
    free[0] = 0

    def scatter(vj, vi):
        z = torch.zeros(N, *vj.shape[1:], dtype=F64, device=DEV)
        return z.index_add_(0, ej, vj).index_add_(0, ei, vi)

    def cost(Z):
        r = _residual(Z, ei, ej, meas)
        return 0.5 * float((r * _mv(Om, r)).sum())

    F, lin = cost(Z), None
    for _ in range(case["trials"]):
        if lin is None:
            r = _residual(Z, ei, ej, meas)
            Rt = _qrot(Z[ei, 3:]).transpose(1, 2)
            Ad = torch.zeros(len(ei), 6, 6, dtype=F64, device=DEV)
            Ad[:, :3, :3] = Ad[:, 3:, 3:] = Rt
            Ad[:, :3, 3:] = -Rt @ _skew(Z[ei, :3])
            A = _jlinv(_se3_ad(r)) @ Ad
            B = A.transpose(1, 2) @ Om @ A
            gq = _mv(A.transpose(1, 2), _mv(Om, r))
            lin = B, scatter(B, B), scatter(gq, -gq)
        B, H, gr = lin
        D = lam * torch.diagonal(H, dim1=1, dim2=2).clamp(1e-6, 1e32)
        b = -gr * free

        def product(x):
            u = _mv(B, x[ej] - x[ei])
            return (scatter(u, -u) + D * x) * free

        if case["solver"] == "cholesky":
            S = torch.zeros(N, 6, N, 6, dtype=F64, device=DEV)
            S[torch.arange(N), :, torch.arange(N), :] = H + torch.diag_embed(D)
            S.permute(0, 2, 1, 3).reshape(N * N, 6, 6)
            M2 = torch.zeros(N * N, 6, 6, dtype=F64, device=DEV)
            M2.index_add_(0, ei * N + ej, -B).index_add_(0, ej * N + ei, -B)
            S += M2.reshape(N, N, 6, 6).permute(0, 2, 1, 3)
            f = free.expand(-1, 6).reshape(-1)
            S = S.reshape(6 * N, 6 * N) * f[:, None] * f[None, :] + torch.diag(1 - f)
            x = torch.cholesky_solve(b.reshape(-1, 1), torch.linalg.cholesky(S)).reshape(N, 6)
        else:
            Mi = torch.linalg.inv(H + torch.diag_embed(D)) * free[:, :, None]
            x, rr = torch.zeros_like(b), b.clone()
            z = _mv(Mi, rr)
            p, rz, bb = z.clone(), float((rr * z).sum()), float((b * b).sum())
            for _k in range(case["maxiter"]):
                q = product(p)
                pq = float((p * q).sum())
                if not pq > 0:
                    break
                x, rr = x + rz / pq * p, rr - rz / pq * q
                if float((rr * rr).sum()) <= case["tol"] ** 2 * bb:
                    break
                z = _mv(Mi, rr)
                rz, old = float((rr * z).sum()), rz
                p = z + rz / old * p
        u = x[ej] - x[ei]
        model = -float((gr * x).sum()) - 0.5 * float((u * _mv(B, u)).sum())
        Zt = torch.where(free > 0, _se3_exp(x, Z), Z)
        Ft = cost(Zt)
        rho = (F - Ft) / model if model else float("nan")
        if math.isfinite(Ft) and model > 0 and Ft < F:
            Z, F, lin = Zt, Ft, None
            lam = max(lam / 2.0, 1e-16) if rho > 0.75 else min(lam / 0.0625, 1e32) if rho < 0.25 else lam
        else:
            lam = min(lam / 0.0625, 1e32)
    return Z


def exact(case, seed):
    kind = case["kind"]
    if kind == "pgo":
        return _pgo_exact(case, seed)
    dt = _dtype(case)
    if kind == "batch":
        Cs, Ps, ci, pi, pix, c0, p0, prob = _windows(case, seed)
        c0, p0, pix = (t.to(dt).to(F64) for t in (c0, p0, pix))
        off = [torch.tensor(np.cumsum(v) - v, device=DEV) for v in (np.array(Cs), np.array(Ps))]
        cw, pw = (torch.repeat_interleave(torch.arange(len(v), device=DEV), torch.tensor(v, device=DEV))
                  for v in (Cs, Ps))
        return _lm(c0, p0, ci.long() + off[0][prob], pi.long() + off[1][prob], pix, case, case["trials"], None, cw, pw,
                   len(Cs))
    ci, pi, pix, c0, p0, g = _scene(case, seed)
    c0, p0, pix = (t.to(dt).to(F64) for t in (c0, p0, pix))
    ci, pi = ci.long(), pi.long()
    if kind == "lm":
        return _lm(c0, p0, ci, pi, pix, case, case["trials"])
    lam = [torch.full((n,), 1e-4, dtype=F64, device=DEV) for n in (case["C"], case["P"])]
    win = torch.zeros(case["C"], dtype=torch.long, device=DEV)
    if kind == "steps":
        x = _randn(g, case["C"], 9)
        n = _Normal(c0, p0, ci, pi, pix, 0.0)
        n.damp(*lam)
        dc, rel = n.pcg(n.rhs(n.gc, n.gp), case["maxiter"], case["tol"], win, 1)
        return dict(U=n.U, V=n.V, gc=n.gc, gp=n.gp, y=n.product(x), dc=dc, dp=n.back(dc, n.gp), rel=float(rel))
    fixed = torch.zeros(case["C"], 9, dtype=torch.bool, device=DEV)
    fixed[0] = True
    fixed[case["C"] // 2, 3:6] = True
    gc, gp = _randn(g, case["C"], 9), _randn(g, case["P"], 3)
    cams, pts = _lm(c0, p0, ci, pi, pix, case, case["trials"], fixed)
    n = _Normal(cams, pts, ci, pi, pix, 0.0)
    n.damp(*lam, fixed)
    v = torch.linalg.solve(n.dense(), n.rhs(-gc, -gp).reshape(-1)).reshape(-1, 9)
    e = _mv(n.Jc, v[ci]) + _mv(n.Jp, n.back(v, -gp)[pi])
    return cams, pts, n.sw[:, None] * e
