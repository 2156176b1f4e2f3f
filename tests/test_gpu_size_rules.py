"""GPU parity at the sizes where the kernels' rules change: ends of tiles, few and many
tiles, cameras that see a point twice, weights and a depth guard, unaligned outputs.

Tolerances as derived in test_gpu_parity.py (FP32 arithmetic on FP32-rounded inputs):
operator entries 1e-4 of the sum of their terms' magnitudes, Jacobian blocks 1e-5,
final costs 1e-4, the first step's model decrease 1e-5; FP64 form 1e-10.
"""
import ctypes
import dataclasses

import numpy as np
import pytest

from oracle import ba_oracle as O
from paper_2605_30583_gb300 import synth

pytestmark = pytest.mark.gpu
TILE = 256


@pytest.fixture(scope="module")
def B():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_2605_30583_gb300 import binding, build
    build.build()
    binding.lib()
    return binding


def _scene(n_cams, n_pts, seed, repeats=0):
    prob = synth.make_problem(n_cams, n_pts, ("poisson", 3.0), "uniform", seed=seed)
    if repeats:
        rng = np.random.default_rng(seed)
        pick = rng.choice(prob.n_obs, size=repeats, replace=False)
        px = prob.pixels[pick] + rng.uniform(-1.0, 1.0, size=(repeats, 2))
        prob = dataclasses.replace(prob, cam_idx=np.concatenate([prob.cam_idx, prob.cam_idx[pick]]),
                                   pt_idx=np.concatenate([prob.pt_idx, prob.pt_idx[pick]]),
                                   pixels=np.concatenate([prob.pixels, px]))
    return synth.round_to_f32(prob)


def _bind(B, prob, precision="mixed"):
    p = B.Problem(prob.n_cams, prob.n_pts, prob.cam_idx, prob.pt_idx, prob.pixels, precision=precision)
    p.set_params(prob.cams_init, prob.pts_init)
    return p


def _args(prob):
    return prob.cams_init, prob.pts_init, prob.cam_idx, prob.pt_idx, prob.pixels


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
@pytest.mark.parametrize("n_cams,n_pts,repeats", [(3, 1, 0), (5, 3, 2), (8, TILE - 1, 0), (8, TILE, 40), (9, TILE + 1, 0),
                                                  (40, 3 * TILE + 2, 60)])
def test_tile_ends(B, n_cams, n_pts, repeats, precision):
    import torch
    prob = _scene(n_cams, n_pts, 100 + n_pts, repeats)
    p = _bind(B, prob, precision)
    op_tol, j_tol = (1e-4, 1e-5) if precision == "mixed" else (1e-10, 1e-10)
    _, r, J = p.evaluate(residuals=True, jacobian=True)
    ref = O.residuals(*_args(prob))
    assert np.all(np.abs(r.double().cpu().numpy() - ref) <= (2e-4 if precision == "mixed" else 1e-9) + j_tol * np.abs(ref))
    _, Jc, Jp = O.jacobian_blocks(*_args(prob))
    J = J.double().cpu().numpy()
    for got, want in ((J[:, :, :9], Jc), (J[:, :, 9:], Jp)):
        assert np.all(np.linalg.norm(got - want, axis=(1, 2)) <= j_tol * np.linalg.norm(want, axis=(1, 2)))
    lin = O.linearize(*_args(prob))
    D = O.damping_diag(lin.J)
    v = np.random.default_rng(1).standard_normal(9 * n_cams + 3 * n_pts).astype(np.float32).astype(np.float64)
    out, _ = p.apply_normal(0.01, torch.from_numpy(v))
    Ja = abs(lin.J)
    scale = Ja.T @ (Ja @ np.abs(v)) + 0.01 * D * np.abs(v)
    err = np.abs(out.double().cpu().numpy() - O.normal_matvec(lin, D, 0.01, v))
    assert np.all(err <= op_tol * scale), np.max(err / scale)


@pytest.mark.parametrize("more", [0, 1])
def test_few_and_many_tiles(B, more):
    """At most two tiles per SM: 512 threads a tile, residuals and |J h|^2 in one launch."""
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    prob = _scene(30, 2 * sms * TILE + more, 7)
    opts = dict(max_lm_iters=2, max_pcg_iters=8)
    res = _bind(B, prob).solve(**opts)
    ref = O.ba_solve(*_args(prob), O.LMOptions(**opts))
    assert abs(res.final_cost - ref.final_cost) <= 1e-4 * ref.final_cost
    h, o = res.history[0], ref.history[0]
    assert abs(h["model_decrease"] - o["model_decrease"]) <= 1e-5 * o["model_decrease"]


@pytest.mark.parametrize("solver,pcg_kernel", [(0, 0), (0, 1), (0, 2), (0, 3), (1, 0)])
@pytest.mark.parametrize("repeats,eps,loss", [(0, 0.1, 0), (50, 0.0, 0), (50, 0.1, 1)])
def test_solvers_with_guard_weights_and_repeats(B, solver, pcg_kernel, repeats, eps, loss):
    prob = _scene(20, 3 * TILE + 5, 11, repeats)
    opts = dict(max_lm_iters=3, max_pcg_iters=12, eps_depth=eps)
    res = _bind(B, prob).solve(solver=solver, pcg_kernel=pcg_kernel, loss=loss, loss_scale=2.0, **opts)
    ref = O.ba_solve(*_args(prob), O.LMOptions(solver="schur" if solver else "pcgnr", loss="huber" if loss else "squared",
                                               loss_scale=2.0, **opts))
    assert res.status == 0
    assert abs(res.final_cost - ref.final_cost) <= 1e-4 * ref.final_cost
    for h, o in zip(res.history, ref.history):
        assert abs(h["pcg_iters"] - o["pcg_iters"]) <= 2 and h["accepted"] == o["accepted"]


@pytest.mark.parametrize("iters", [1, 2, 3])
def test_points_step_of_the_last_iteration(B, iters):
    """Separate kernels: the points' step of an iteration is taken by the next operator, that
    of the last one by the candidate."""
    prob = _scene(12, 2 * TILE + 3, 21)
    opts = dict(max_lm_iters=1, max_pcg_iters=iters)
    h = _bind(B, prob).solve(pcg_kernel=1, **opts).history[0]
    o = O.ba_solve(*_args(prob), O.LMOptions(**opts)).history[0]
    assert h["pcg_iters"] == o["pcg_iters"] == iters
    assert abs(h["model_decrease"] - o["model_decrease"]) <= 1e-5 * o["model_decrease"]
    assert abs(h["cost_new"] - o["cost_new"]) <= 1e-5 * o["cost_new"]


@pytest.mark.parametrize("n_cams,n_pts", [(20, 3 * TILE), (200, 20 * TILE + 7)])
def test_a_persistent_solve_stops_on_a_true_residual(B, n_cams, n_pts):
    """The step of one LM iteration meets the tolerance in FP64: |b - (J^T J + mu D) h| <= tol |b|.
    h is the difference of the parameters; FP32 rounding of h and of the residual that the kernel
    forms adds at most ~1e-5 |b| at tol 1e-3."""
    prob = _scene(n_cams, n_pts, 31)
    p = _bind(B, prob)
    tol = 1e-3
    res = p.solve(max_lm_iters=1, max_pcg_iters=300, pcg_rel_tol=tol)
    assert res.history[0]["accepted"] and res.history[0]["pcg_iters"] < 300
    c, q = p.get_params()
    h = np.concatenate([(np.asarray(c) - prob.cams_init).ravel(), (np.asarray(q) - prob.pts_init).ravel()])
    lin = O.linearize(*_args(prob))
    D = O.damping_diag(lin.J)
    b = -(lin.J.T @ np.asarray(lin.r).ravel())
    left = b - O.normal_matvec(lin, D, 1.0 / O.LMOptions().initial_trust_region, h)
    assert np.linalg.norm(left) <= (1.01 * tol + 1e-5) * np.linalg.norm(b)


def test_unaligned_evaluation_outputs(B):
    """Outputs that are not 16-byte (Jacobian) or 8-byte (residual) aligned hold the same values."""
    import torch
    prob = _scene(10, TILE + 9, 41)
    p = _bind(B, prob)
    _, r, J = p.evaluate(residuals=True, jacobian=True)
    for shift in (1, 2, 3):
        r2 = torch.empty(2 * prob.n_obs + shift, device="cuda")[shift:]
        J2 = torch.empty(24 * prob.n_obs + shift, device="cuda")[shift:]
        cost = ctypes.c_double()
        B.check(B.lib().ba_evaluate(p._h, ctypes.byref(cost), r2.data_ptr(), J2.data_ptr()))
        assert torch.equal(r2.view_as(r), r) and torch.equal(J2.view_as(J), J)


@pytest.mark.parametrize("n_pts", [63, 64, 65, 2 * 64 + 1, 152 * 64, 152 * 64 + 1])
def test_tile_size_rule(B, n_pts):
    """Small problems are cut into tiles of 64 to 256 points, a multiple of four."""
    import torch
    prob = _scene(24, n_pts, 300 + n_pts)
    p = _bind(B, prob)
    p.evaluate()
    lin = O.linearize(*_args(prob))
    D = O.damping_diag(lin.J)
    v = np.random.default_rng(2).standard_normal(9 * 24 + 3 * n_pts).astype(np.float32).astype(np.float64)
    out, _ = p.apply_normal(0.01, torch.from_numpy(v))
    Ja = abs(lin.J)
    scale = Ja.T @ (Ja @ np.abs(v)) + 0.01 * D * np.abs(v)
    err = np.abs(out.double().cpu().numpy() - O.normal_matvec(lin, D, 0.01, v))
    assert np.all(err <= 1e-4 * scale), np.max(err / scale)
    opts = dict(max_lm_iters=2, max_pcg_iters=8)
    res = p.solve(**opts)
    ref = O.ba_solve(*_args(prob), O.LMOptions(**opts))
    assert abs(res.final_cost - ref.final_cost) <= 1e-4 * ref.final_cost


def test_the_operator_and_the_gradient_share_their_jacobian(B):
    """A point 0.5 to 1 in front of a camera that is 1000 from the origin has ~5 digits left in
    P = R X + t.  g = J^T r and J^T J use the same rounded P: with r = J d in the linearisation's
    arithmetic, J^T J d and J^T r agree to FP32 rounding of the sums, 2e-6 of their norm, where
    Jacobians that round P differently disagree by ~1e-4."""
    import torch
    rng = np.random.default_rng(5)
    n_cams, n_pts = 4, 300
    cams = np.zeros((n_cams, 9))
    cams[:, :3] = 0.3 * rng.standard_normal((n_cams, 3))
    cams[:, 6] = 700.0
    from scipy.spatial.transform import Rotation
    R = Rotation.from_rotvec(cams[:, :3]).as_matrix()
    pts = 1000.0 * np.array([0.6, -0.5, 0.62]) + rng.uniform(-0.2, 0.2, size=(n_pts, 3))
    centre = 1000.0 * np.array([0.6, -0.5, 0.62])
    P0 = np.array([0.0, 0.0, -0.75])   # the centre of the points in each camera
    cams[:, 3:6] = P0 - R @ centre
    cams, pts = cams.astype(np.float32).astype(np.float64), pts.astype(np.float32).astype(np.float64)
    ci, pi = np.tile(np.arange(n_cams), n_pts), np.repeat(np.arange(n_pts), n_cams)
    p = B.Problem(n_cams, n_pts, ci.astype(np.uint32), pi.astype(np.uint32), np.zeros((len(ci), 2)))
    p.set_params(cams, pts)
    _, _, J = p.evaluate(jacobian=True)
    J = J.double().cpu().numpy()
    d = np.concatenate([np.zeros(9 * n_cams), rng.standard_normal(3 * n_pts)]).astype(np.float32).astype(np.float64)
    dp = d[9 * n_cams:].reshape(-1, 3)
    r = np.einsum("oij,oj->oi", J[:, :, 9:], dp[pi])
    want = np.zeros((n_pts, 3))
    np.add.at(want, pi, np.einsum("oij,oi->oj", J[:, :, 9:], r))
    out, _ = p.apply_normal(0.0, torch.from_numpy(d))
    got = out.double().cpu().numpy()[9 * n_cams:].reshape(-1, 3)
    assert np.linalg.norm(got - want) <= 2e-6 * np.linalg.norm(want)
