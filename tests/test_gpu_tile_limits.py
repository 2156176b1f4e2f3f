"""GPU parity where tiles are extreme: many light tiles in one CTA of the persistent PCG.

Tolerances as derived in test_gpu_parity.py (FP32 arithmetic on FP32-rounded inputs): first step's
model decrease 1e-5, final costs 1e-4.
"""
import numpy as np
import pytest

from oracle import ba_oracle as O
from paper_2605_30583_gb300 import synth

pytestmark = pytest.mark.gpu

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
