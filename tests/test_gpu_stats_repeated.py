"""GPU checks of the statistics on repeated values -- flat image pairs, one motion per object, stripes -- where every
thread's sum meets the same roundings, so that an error of theirs does not average out.

The reference is exact (rationals).  Bars: a kernel's sum is exact to some 2^-70 until the words of a warp meet in FP64;
from there on two additions to join the words, four to add a block's warps, nine to add the blocks and one division
round by at most 2^-53 each, 16 in all.  The variance subtracts the square of a mean so obtained (35 roundings)."""
from fractions import Fraction

import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

U = 2.0 ** -53
SIZES = [(128, 128), (641, 363), (1920, 1080)]  # 2^14 vectors, the shortest summed as floats; a remainder; the benchmark's


@pytest.fixture(scope="module")
def b():
    if not torch.cuda.is_available():
        pytest.fail("a CUDA GPU is required for the gpu-marked tests")
    from paper_2307_12607_gb300 import build, binding
    build.build()
    return binding


def stripes(values, n):
    """values[0], values[1], ... in turn, n of them, on the GPU."""
    v = torch.from_numpy(values).cuda()
    return v.repeat(-(-n // len(values)))[:n].contiguous()


def counts(period, n):
    return [n // period + (1 if j < n % period else 0) for j in range(period)]


@pytest.mark.parametrize("period", [1, 4])
@pytest.mark.parametrize("W,H", SIZES)
def test_color_mse_of_repeated_values(b, W, H, period):
    rng = np.random.default_rng(period)
    n = 3 * W * H
    for _ in range(8):
        x = rng.uniform(size=period).astype(np.float32)
        y = (rng.uniform(size=period) * 2.0 ** -rng.integers(0, 16, size=period)).astype(np.float32)
        want = sum(c * (Fraction(float(p)) - Fraction(float(q))) ** 2 for c, p, q in zip(counts(period, n), x, y)) / n
        got = b.exw_color_mse(stripes(x, n).view(3, H, W), stripes(y, n).view(3, H, W))
        assert abs(Fraction(got) - want) <= 16 * U * want


@pytest.mark.parametrize("period", [2, 4])
@pytest.mark.parametrize("W,H", SIZES)
def test_mv_variance_of_repeated_values(b, W, H, period):
    rng = np.random.default_rng(10 + period)
    n = W * H
    for _ in range(8):
        v = [(rng.normal(size=period) * 2.0 ** rng.integers(-12, 12, size=period)).astype(np.float32) for _ in range(2)]
        got = b.exw_mv_variance(torch.stack([stripes(a, n).view(H, W) for a in v]))
        assert got[0] == n
        for axis in (0, 1):
            off = [Fraction(float(a)) - Fraction(float(v[axis][0])) for a in v[axis]]
            mean = sum(c * d for c, d in zip(counts(period, n), off)) / n
            square = sum(c * d * d for c, d in zip(counts(period, n), off)) / n
            assert abs(Fraction(got[1 + axis]) - (square - mean * mean)) <= U * (17 * square + 36 * mean * mean)
