"""The PCG iteration's byte model as the kernels move the data: the points' step h += alpha p is taken
by the next operator, not by the update."""
import os
import sys
from types import SimpleNamespace

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
import bench  # noqa: E402


def test_tile_pcg_iteration_bytes_with_the_deferred_step():
    # per point 96 (operator: z, p, D, X, h in, p, q, h out) + 48 (update: r, q in, r, z out) + 24 (M^-1)
    for sizes, want in (((0, 1, 0), 168), ((1, 0, 0), 1048), ((0, 0, 1), 4)):
        prob = SimpleNamespace(n_cams=sizes[0], n_pts=sizes[1], n_obs=sizes[2])
        assert bench.pcg_iter_tile_model(prob, deferred_h=True) == want
