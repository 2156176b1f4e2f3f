"""GPU parity where tiles are extreme: more observations in one tile than the shared-memory sort
or the tile kernels' tables hold, full tiles with a ragged end, many light tiles in one CTA.

Tolerances as derived in test_gpu_parity.py (FP32 arithmetic on FP32-rounded inputs): operator
entries 1e-4 of the sum of their terms' magnitudes, first step's model decrease and candidate cost
1e-5, final costs 1e-4; FP64 form 1e-8.
"""
import numpy as np
import pytest

from oracle import ba_oracle as O
from paper_2605_30583_gb300 import synth

pytestmark = pytest.mark.gpu

SORT_MAX = 16384        # observations of a tile that are sorted in shared memory
TABLE_MAX = 160 * 1024  # bytes of a tile's observation table in shared memory
SMS = 152


@pytest.fixture(scope="module")
def B():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_2605_30583_gb300 import binding, build
    build.build()
    binding.lib()
    return binding


def _tile_points(n_pts):
    """Points per tile (layout.h)."""
    full = -(-n_pts // 256)
    if full > 16 * SMS:
        return 256
    tiles = -(-full // SMS) * SMS
    return min(256, max(64, -(--(-n_pts // tiles) // 4) * 4))


def _bind(B, prob, precision="mixed"):
    p = B.Problem(prob.n_cams, prob.n_pts, prob.cam_idx, prob.pt_idx, prob.pixels, precision=precision)
    p.set_params(prob.cams_init, prob.pts_init)
    return p


def _args(prob):
    return prob.cams_init, prob.pts_init, prob.cam_idx, prob.pt_idx, prob.pixels


def _check_operator(B, p, prob, lin, tol):
    import torch
    p.evaluate()
    D = O.damping_diag(lin.J)
    v = np.random.default_rng(4).standard_normal(9 * prob.n_cams + 3 * prob.n_pts).astype(np.float32).astype(np.float64)
    out, _ = p.apply_normal(0.01, torch.from_numpy(v))
    Ja = abs(lin.J)
    scale = Ja.T @ (Ja @ np.abs(v)) + 0.01 * D * np.abs(v)
    err = np.abs(out.double().cpu().numpy() - O.normal_matvec(lin, D, 0.01, v))
    assert np.all(err <= tol * scale), np.max(err / scale)


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
def test_a_tile_beyond_the_shared_memory_sort(B, precision):
    """One tile of more observations than the bind sorts per tile: the global sort."""
    prob = synth.round_to_f32(synth.make_problem(300, 64, ("poisson", 2000.0), "uniform", seed=61))
    assert _tile_points(prob.n_pts) >= prob.n_pts and SORT_MAX < prob.n_obs and 5 * prob.n_obs < TABLE_MAX
    p = _bind(B, prob, precision)
    _check_operator(B, p, prob, O.linearize(*_args(prob)), 1e-4 if precision == "mixed" else 1e-10)
    opts = dict(max_lm_iters=4, max_pcg_iters=20)
    res = p.solve(**opts)
    ref = O.ba_solve(*_args(prob), O.LMOptions(**opts))
    assert res.status == 0
    tol = 1e-4 if precision == "mixed" else 1e-8
    assert abs(res.final_cost - ref.final_cost) <= tol * ref.final_cost


def test_a_tile_beyond_the_observation_table(B):
    """One tile whose table does not fit: the kernels that read the observations from memory.
    The step of 1 to 3 PCG iterations (the points' part of the last one is taken by the candidate)."""
    prob = synth.round_to_f32(synth.make_problem(2700, 64, ("poisson", 20000.0), "uniform", seed=62))
    assert _tile_points(prob.n_pts) >= prob.n_pts and prob.n_obs > TABLE_MAX
    p = _bind(B, prob)
    _check_operator(B, p, prob, O.linearize(*_args(prob)), 1e-4)
    for iters in (1, 2, 3):
        p.set_params(prob.cams_init, prob.pts_init)
        opts = dict(max_lm_iters=1, max_pcg_iters=iters, pcg_rel_tol=0.0)
        h = p.solve(pcg_kernel=1, **opts).history[0]
        o = O.ba_solve(*_args(prob), O.LMOptions(**opts)).history[0]
        assert h["pcg_iters"] == o["pcg_iters"] == iters
        assert abs(h["model_decrease"] - o["model_decrease"]) <= 1e-5 * o["model_decrease"]
        assert abs(h["cost_new"] - o["cost_new"]) <= 1e-5 * o["cost_new"]


@pytest.mark.parametrize("n_pts", [SMS * 256 - 1, SMS * 256 - 3])
def test_full_tiles_with_a_ragged_end(B, n_pts):
    """Tiles of 256 points (slots up to 255), the last one short and not a multiple of four."""
    assert _tile_points(n_pts) == 256 and n_pts % 4 != 0
    prob = synth.round_to_f32(synth.make_problem(60, n_pts, ("poisson", 3.0), "nearest", seed=63))
    p = _bind(B, prob)
    _check_operator(B, p, prob, O.linearize(*_args(prob)), 1e-4)
    for kernel in (1, 3):
        p.set_params(prob.cams_init, prob.pts_init)
        opts = dict(max_lm_iters=1, max_pcg_iters=3, pcg_rel_tol=0.0)
        h = p.solve(pcg_kernel=kernel, **opts).history[0]
        o = O.ba_solve(*_args(prob), O.LMOptions(**opts)).history[0]
        assert abs(h["model_decrease"] - o["model_decrease"]) <= 1e-5 * o["model_decrease"]


def uneven_problem():
    """152 tiles of 64 points: 20 whose points every one of 300 cameras sees, 132 whose points two
    of 100 other cameras see.  A CTA's share of the observations is one part in 152, so one that
    starts after the heavy tiles takes some twenty light ones."""
    heavy, n_pts, seen, others = 20 * 64, SMS * 64, 300, 100
    prob = synth.make_problem(seen + others, n_pts, ("poisson", 3.0), "uniform", seed=64)
    ci, pi = [np.tile(np.arange(seen), heavy)], [np.repeat(np.arange(heavy), seen)]
    light = np.arange(heavy, n_pts)
    for step in (0, 7):
        ci.append(seen + (light + step) % others)
        pi.append(light)
    import dataclasses
    ci, pi = np.concatenate(ci).astype(np.uint32), np.concatenate(pi).astype(np.uint32)
    exact = O.residuals(prob.cams_gt, prob.pts_gt, ci, pi, np.zeros((len(ci), 2)))
    noise = np.random.default_rng(65).standard_normal(exact.shape)
    return synth.round_to_f32(dataclasses.replace(prob, cam_idx=ci, pt_idx=pi, pixels=exact + noise))


def test_many_light_tiles_in_one_cta(B):
    """The persistent PCG takes every plan that its shared memory holds, also CTAs of twenty tiles."""
    prob = uneven_problem()
    assert _tile_points(prob.n_pts) == 64
    share = prob.n_obs / SMS
    assert 17 * 64 * 2 < share < 22 * 64 * 2
    p = _bind(B, prob)
    opts = dict(max_lm_iters=2, max_pcg_iters=10)
    ref = O.ba_solve(*_args(prob), O.LMOptions(**opts))
    for kernel in (2, 0):
        p.set_params(prob.cams_init, prob.pts_init)
        res = p.solve(pcg_kernel=kernel, **opts)
        assert res.status == 0
        assert abs(res.final_cost - ref.final_cost) <= 1e-4 * ref.final_cost
        h, o = res.history[0], ref.history[0]
        assert abs(h["model_decrease"] - o["model_decrease"]) <= 1e-5 * o["model_decrease"]
        assert p.profile_kernels(reps=1)["pcg_persistent"] > 0.0
