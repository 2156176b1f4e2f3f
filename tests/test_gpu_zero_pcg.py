"""A solve that runs no PCG iteration takes a zero step, whatever was solved before."""
import numpy as np
import pytest

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


@pytest.mark.parametrize("use_graph", [0, 1, 2])
@pytest.mark.parametrize("pcg_kernel", [0, 1, 2, 3])
def test_no_pcg_iterations_means_no_step(B, pcg_kernel, use_graph):
    """The first solve takes a good step; with the parameters set back, the same step would be
    accepted again.  Without PCG iterations h = 0: the model decrease is 0 and every step is
    rejected, so the parameters stay exactly as set."""
    prob = synth.round_to_f32(synth.make_config("tiny", seed=5))
    p = B.Problem(prob.n_cams, prob.n_pts, prob.cam_idx, prob.pt_idx, prob.pixels)
    p.set_params(prob.cams_init, prob.pts_init)
    first = p.solve(max_lm_iters=1, pcg_kernel=pcg_kernel, use_graph=use_graph)
    assert first.accepted == 1
    p.set_params(prob.cams_init, prob.pts_init)
    res = p.solve(max_lm_iters=2, max_pcg_iters=0, pcg_kernel=pcg_kernel, use_graph=use_graph)
    assert res.accepted == 0 and res.final_cost == res.initial_cost == first.initial_cost
    assert all(h["model_decrease"] == 0.0 for h in res.history)
    cams, pts = p.get_params()
    assert np.array_equal(cams, prob.cams_init) and np.array_equal(pts, prob.pts_init)
