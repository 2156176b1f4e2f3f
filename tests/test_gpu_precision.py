"""What is computed beyond FP32 keeps its bits: double-float residuals, FP64 camera records."""
import numpy as np
import pytest

from oracle import ba_oracle as O
from paper_2605_30583_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_2605_30583_gb300 import binding, build
    build.build()
    binding.lib()
    return binding


@pytest.mark.parametrize("scene,n_cams,n_pts,kw", [("cloud", 200, 50_000, {}),
                                                   ("band", 3000, 100_000, dict(ring_radius=65.0, scene="band"))])
def test_residual_error(B, scene, n_cams, n_pts, kw):
    """Pixels are the exact projections rounded to FP32, so residuals below 1e-6 px show the
    arithmetic's error and not their own rounding.  The bound is the error of the same formula with
    every double-float operation renormalised and a correctly rounded FP32 reciprocal, taken in
    the same operations on the host, plus 4 % for the choice of observations and for operations
    that round differently."""
    prob = synth.make_problem(n_cams, n_pts, ("poisson", 3.0), "nearest", seed=200, **kw)
    args = prob.cams_gt, prob.pts_gt, prob.cam_idx, prob.pt_idx
    exact = O.residuals(*args, np.zeros((prob.n_obs, 2)))
    px = exact.astype(np.float32).astype(np.float64)
    p = B.Problem(prob.n_cams, prob.n_pts, prob.cam_idx, prob.pt_idx, px)
    p.set_params(prob.cams_gt, prob.pts_gt)
    _, r, _ = p.evaluate(residuals=True)
    pick = np.abs(exact - px) < 1e-6
    err = (r.double().cpu().numpy() - (exact - px))[pick]
    ref = (_renormalised(prob, px) - (exact - px))[pick]
    assert np.sqrt(np.mean(err**2)) <= 1.04 * np.sqrt(np.mean(ref**2))


@pytest.mark.parametrize("n_cams,n_pts,kw", [(200, 5000, {}), (3000, 20_000, dict(ring_radius=65.0, scene="band"))])
def test_camera_record_error(B, n_cams, n_pts, kw):
    """The FP64 form's residuals against extended precision: no further off than the formula with
    sin th / th, 2 sin^2(th / 2) / th^2 in FP64 on the host, plus 6 % for operations that round
    differently (FMA)."""
    prob = synth.make_problem(n_cams, n_pts, ("poisson", 3.0), "nearest", seed=1, **kw)
    p = B.Problem(prob.n_cams, prob.n_pts, prob.cam_idx, prob.pt_idx, prob.pixels, precision="fp64")
    p.set_params(prob.cams_gt, prob.pts_gt)
    _, r, _ = p.evaluate(residuals=True)
    exact = _residuals(prob, np.longdouble)

    def rms(x):
        return float(np.sqrt(np.mean((x - exact) ** 2)))

    assert rms(r.cpu().numpy()) <= 1.06 * rms(_residuals(prob, np.float64))


def test_reciprocal_is_the_rounded_quotient(B):
    """Two Newton-Raphson steps from the hardware's ~20 bits leave 2^-70 before the last rounding, so
    a result differs from the rounded quotient only where that lies within 2^-17 ulp of the middle
    between two numbers: 2^-16 of the arguments at most."""
    import torch
    x = np.concatenate([1.0 + np.random.default_rng(3).random(1_000_000), np.logspace(-299, 299, 200_001)])
    y = B.selftest_rcp64(torch.from_numpy(x).cuda()).cpu().numpy()
    assert np.mean(y != 1.0 / x) <= 2.0**-16


@pytest.mark.parametrize("iters", [2, 4])
def test_camera_blocks_with_tiny_pivots(B, iters):
    """A camera that sees points on its axis only: no observation moves with w_z, t_z, f, k1 or k2,
    and with min_diag = 1e-305 their pivots are ~1e-307.  The block is positive definite all the same,
    and the preconditioner is its inverse: FP64 form against the oracle."""
    prob = synth.make_problem(12, 200, ("poisson", 3.0), "uniform", seed=9)
    k = 6
    cams, pts, ci, pi = prob.cams_init.copy(), prob.pts_init.copy(), prob.cam_idx.copy(), prob.pt_idx
    ci[ci == 0] = 1 + pi[ci == 0] % 11
    cams[0, :6] = 0.0
    pts[:k, :2], pts[:k, 2] = 0.0, -np.linspace(2.0, 3.0, k)
    ci = np.concatenate([ci, np.zeros(k, ci.dtype)])
    pi = np.concatenate([pi, np.arange(k, dtype=pi.dtype)])
    px = np.concatenate([prob.pixels, np.random.default_rng(8).standard_normal((k, 2))])
    opts = dict(max_lm_iters=1, max_pcg_iters=iters, pcg_rel_tol=0.0, min_diag=1e-305)
    p = B.Problem(prob.n_cams, prob.n_pts, ci, pi, px, precision="fp64")
    p.set_params(cams, pts)
    h = p.solve(**opts).history[0]
    o = O.ba_solve(cams, pts, ci, pi, px, O.LMOptions(**opts)).history[0]
    assert h["pcg_iters"] == o["pcg_iters"] == iters
    assert abs(h["model_decrease"] - o["model_decrease"]) <= 1e-9 * o["model_decrease"]


@pytest.mark.parametrize("pcg_kernel", [0, 1])
def test_gradients_whose_squares_leave_the_fp32_range(B, pcg_kernel):
    """A point that grazes a camera's plane (|p| ~ 1000) has a derivative of ~1e15 in k2: g there is
    ~1e20, representable in FP32, its square is not.  |r_0|^2 and r^T z are summed in FP64, so the
    first step is the oracle's (the FP32 residual after it may still be too long to go on)."""
    prob = synth.make_problem(12, 200, ("poisson", 3.0), "uniform", seed=12)
    cams, pts = prob.cams_init.copy(), prob.pts_init.copy()
    cams[0], pts[0] = 0.0, (1.0, 0.3, -1e-3)
    cams[0, 6] = 1000.0
    ci, pi = prob.cam_idx.copy(), prob.pt_idx
    ci[ci == 0] = 1 + pi[ci == 0] % 11
    ci = np.concatenate([ci, np.zeros(1, ci.dtype)])
    pi = np.concatenate([pi, np.zeros(1, pi.dtype)])
    cams, pts = cams.astype(np.float32).astype(np.float64), pts.astype(np.float32).astype(np.float64)
    px = np.concatenate([prob.pixels, O.residuals(cams, pts, ci[-1:], pi[-1:], np.zeros((1, 2))) + 60.0])
    px = px.astype(np.float32).astype(np.float64)
    opts = dict(max_lm_iters=1, max_pcg_iters=1)
    g = O.linearize(cams, pts, ci, pi, px).g
    assert 2e19 < np.abs(g).max() < 1e38
    p = B.Problem(prob.n_cams, prob.n_pts, ci, pi, px)
    p.set_params(cams, pts)
    res = p.solve(pcg_kernel=pcg_kernel, **opts)
    o = O.ba_solve(cams, pts, ci, pi, px, O.LMOptions(**opts)).history[0]
    assert res.accepted == 1 and o["accepted"]
    assert abs(res.history[0]["model_decrease"] - o["model_decrease"]) <= 1e-3 * abs(o["model_decrease"])


@pytest.mark.parametrize("pcg_kernel", [0, 2])
def test_residuals_whose_squares_add_up_beyond_fp32(B, pcg_kernel):
    """Sixty cameras with g ~ 3e18 in k2 (a grazing point each, as above): every square is an FP32 number,
    their sum over the grid's CTAs is not.  The exchanged totals carry it."""
    k = 60
    base = synth.make_problem(12, 200, ("poisson", 3.0), "uniform", seed=13)
    centre = np.zeros((k, 3))
    centre[:, 0] = 10.0 * np.arange(k)
    far = np.array([300.0, 0.0, 700.0])
    cams = np.zeros((k + 1, 9))
    cams[:k, 3:6], cams[k, 3:6], cams[:, 6] = -centre, -far, 1000.0
    cams = np.concatenate([base.cams_init, cams]).astype(np.float32).astype(np.float64)
    pts = np.concatenate([base.pts_init, centre + (1.0, 0.3, -1e-3)]).astype(np.float32).astype(np.float64)
    i = np.arange(k)
    ci = np.concatenate([base.cam_idx, 12 + i, np.full(k, 12 + k)]).astype(np.uint32)
    pi = np.concatenate([base.pt_idx, 200 + i, 200 + i]).astype(np.uint32)
    px = np.concatenate([base.pixels, O.residuals(cams, pts, ci, pi, np.zeros((len(ci), 2)))[len(base.pixels):]])
    px[len(base.pixels):len(base.pixels) + k, 0] += 2.5
    px = px.astype(np.float32).astype(np.float64)
    g = O.linearize(cams, pts, ci, pi, px).g
    assert np.abs(g).max() < 1e19 and np.sum(g**2) > 3.5e38
    opts = dict(max_lm_iters=1, max_pcg_iters=1)
    p = B.Problem(len(cams), len(pts), ci, pi, px)
    p.set_params(cams, pts)
    res = p.solve(pcg_kernel=pcg_kernel, **opts)
    o = O.ba_solve(cams, pts, ci, pi, px, O.LMOptions(**opts)).history[0]
    assert res.accepted == 1 and o["accepted"] and res.history[0]["pcg_iters"] == 1
    assert abs(res.history[0]["model_decrease"] - o["model_decrease"]) <= 1e-3 * abs(o["model_decrease"])


def test_batch_costs_beyond_the_fp32_range(B):
    """Squared residuals of ~1e37 each are FP32 numbers; their sum is not, and the cost is an FP64
    sum.  Terms round to FP32: 1e-6 relative."""
    import dataclasses
    prob = synth.round_to_f32(synth.make_problem(8, 100, ("poisson", 3.0), "uniform", seed=14))
    scaled = synth.round_to_f32(dataclasses.replace(prob, pixels=prob.pixels * 1e16))
    ref = [0.5 * np.sum(O.residuals(p.cams_init, p.pts_init, p.cam_idx, p.pt_idx, p.pixels) ** 2) for p in (prob, scaled)]
    assert ref[1] > 3.5e38
    b = B.Batch([prob, scaled])
    b.set_params(np.concatenate([prob.cams_init] * 2), np.concatenate([prob.pts_init] * 2))
    res = b.solve(max_lm_iters=0)
    for r, want in zip(res, ref):
        assert abs(r.initial_cost - want) <= 1e-6 * want


def _residuals(prob, dtype):
    c, X = prob.cams_gt.astype(dtype), prob.pts_gt.astype(dtype)[prob.pt_idx]
    w, th2 = c[:, :3], (c[:, :3] ** 2).sum(1)
    th = np.sqrt(th2)
    K = np.zeros((len(c), 3, 3), dtype)
    K[:, 2, 1], K[:, 0, 2], K[:, 1, 0] = w.T
    K -= K.transpose(0, 2, 1)
    eye = np.eye(3, dtype=dtype)
    K2 = w[:, :, None] * w[:, None, :] - th2[:, None, None] * eye
    R = eye + (np.sin(th) / th)[:, None, None] * K + (2 * np.sin(th / 2) ** 2 / th2)[:, None, None] * K2
    R, c = R[prob.cam_idx], c[prob.cam_idx]
    P = sum(R[:, :, j] * X[:, j, None] for j in range(3)) + c[:, 3:6]
    q = -P[:, :2] / P[:, 2:]
    n2 = (q * q).sum(1)
    return (c[:, 6] * (1 + n2 * (c[:, 7] + c[:, 8] * n2)))[:, None] * q - prob.pixels


# ---- double-float arithmetic on the host: float32 pairs, FMA through float64 (a product of two
# float32 values is exact there)
F = np.float32


def _fma(a, b, c):
    return (a.astype(np.float64) * b + c).astype(F)


def _norm(h, l):
    s = h + l
    return s, l - (s - h)


def _add(a, b):
    s = a[0] + b[0]
    t = s - a[0]
    return _norm(s, ((a[0] - (s - t)) + (b[0] - t)) + (a[1] + b[1]))


def _mul(a, b):
    p = a[0] * b[0]
    e = _fma(a[0], b[0], -p)
    return _norm(p, _fma(a[1], b[0], _fma(a[0], b[1], e)))


def _rcp(b):
    x = (1.0 / b[0].astype(np.float64)).astype(F)
    bx = _mul(b, (x, np.zeros_like(x)))
    return _norm(x, x * ((F(1) - bx[0]) - bx[1]))


def _pair(x):
    h = x.astype(F)
    return h, (x - h).astype(F)


def _renormalised(prob, px):
    from scipy.spatial.transform import Rotation
    c, X = prob.cams_gt[prob.cam_idx], prob.pts_gt[prob.pt_idx]
    R = Rotation.from_rotvec(prob.cams_gt[:, :3]).as_matrix()[prob.cam_idx]
    X = [_pair(X[:, j]) for j in range(3)]
    P = []
    for i in range(3):
        a = _mul(_pair(R[:, i, 0]), X[0])
        for j in (1, 2):
            a = _add(a, _mul(_pair(R[:, i, j]), X[j]))
        P.append(_add(a, _pair(c[:, 3 + i])))
    iz = _rcp(P[2])
    q = [_mul(P[0], iz), _mul(P[1], iz)]
    one = (np.ones_like(iz[0]), np.zeros_like(iz[0]))
    n2 = _add(_mul(q[0], q[0]), _mul(q[1], q[1]))
    s = _add(_mul(n2, _add(_pair(c[:, 7]), _mul(_pair(c[:, 8]), n2))), one)
    fs = _mul(_pair(c[:, 6]), s)
    out = []
    for k in range(2):
        h, l = _add(_mul(fs, q[k]), (px[:, k].astype(F), np.zeros_like(iz[0])))
        out.append(-(h + l))
    return np.stack(out, 1).astype(np.float64)
