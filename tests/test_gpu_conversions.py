"""The kernels' FP32 / FP64 conversions on the integer units against the conversion instructions."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _bits(lo, hi, n, dtype, rng):
    return rng.integers(lo, hi, size=n, dtype=np.uint64).astype(np.uint32 if dtype == np.float32 else np.uint64).view(dtype)


def test_conversions_equal_the_casts():
    """Every class of number, bit for bit (a NaN has to stay one): random bit patterns, zeros of both
    signs, subnormals, the ends of the normal range, infinities and NaN; and for the rounding, ties to
    even and odd, their neighbours, carries into the exponent and from the largest float to infinity."""
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_2605_30583_gb300 import binding, build
    build.build()
    rng = np.random.default_rng(0)
    n = 1 << 20
    f = _bits(0, 1 << 32, n, np.float32, rng).copy()
    edges = np.array([0, 1, 0x7fffff, 0x800000, 0x800001, 0x3f800000, 0x7f7fffff, 0x7f800000, 0x7f800001, 0x7fc00000],
                     np.uint32)
    f[: 2 * len(edges)] = np.concatenate([edges, edges | 0x80000000]).astype(np.uint32).view(np.float32)
    d = _bits(0, (1 << 64) - 1, n, np.float64, rng).copy()
    # exponents within and around the floats' range, where the integer path and its limits are
    near = rng.integers(890 - 30, 1160, size=n // 2, dtype=np.uint64) << 52 | rng.integers(0, 1 << 52, size=n // 2,
                                                                                          dtype=np.uint64)
    d[: n // 2] = (near | rng.integers(0, 2, size=n // 2, dtype=np.uint64) << 63).view(np.float64)
    # ties and their neighbours: the 29 bits that are cut off at 0, 1, half - 1, half, half + 1 and all set
    cut = np.array([0, 1, (1 << 28) - 1, 1 << 28, (1 << 28) + 1, (1 << 29) - 1], np.uint64)
    top = np.array([0, 1, 2, (1 << 23) - 2, (1 << 23) - 1], np.uint64)
    exp = np.array([0, 1, 871, 872, 873, 896, 897, 898, 1023, 1149, 1150, 1151, 2046, 2047], np.uint64)
    grid = (exp[:, None, None] << np.uint64(52) | top[None, :, None] << np.uint64(29) | cut[None, None, :]).ravel()
    grid = np.concatenate([grid, grid | np.uint64(1 << 63)]).view(np.float64)
    d[-len(grid):] = grid
    wide, narrowed = binding.selftest_conversions(torch.from_numpy(f).cuda(), torch.from_numpy(d).cuda())
    wide, narrowed = wide.cpu().numpy(), narrowed.cpu().numpy()
    with np.errstate(over="ignore", under="ignore", invalid="ignore"):
        for got, want, bits in ((wide, f.astype(np.float64), np.uint64), (narrowed, d.astype(np.float32), np.uint32)):
            nan = np.isnan(want)
            assert np.array_equal(np.isnan(got), nan)
            assert np.array_equal(got[~nan].view(bits), want[~nan].view(bits))
