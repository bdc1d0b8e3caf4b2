"""GPU checks of the statistics' summation paths at the sizes where they change: below and above the length from which
values are added as float pairs, lengths that leave a remainder of a 16-byte load, addresses that are not multiples of
16 bytes, and values that leave the float path (tiny, huge and non-finite differences).

Bars: a chain of n FP64 additions of positive terms is within n 2^-53 of the exact sum, relative; the kernels' trees of
n values are held to that (and to 16 of them for short inputs).  The variance subtracts the square of the mean offset
from the mean square, so its bar is multiplied by their ratio to the variance."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def b():
    if not torch.cuda.is_available():
        pytest.fail("a CUDA GPU is required for the gpu-marked tests")
    from paper_2307_12607_gb300 import build, binding
    build.build()
    return binding


def on_gpu(x, offset):
    """x on the GPU, its first element ``offset`` elements past a 256-byte boundary."""
    buf = torch.zeros(x.size + offset, dtype=torch.from_numpy(x).dtype, device="cuda")
    t = buf[offset:].view(x.shape)
    t.copy_(torch.from_numpy(x))
    return t


def exact_square_sum(d):
    """Sum of squares of float64 values, exact up to one rounding (Veltkamp split, math.fsum)."""
    c = 134217729.0 * d
    hi = c - (c - d)
    lo = d - hi
    return math.fsum(np.concatenate([hi * hi, 2 * hi * lo, lo * lo]).ravel().tolist())


SIZES = [(1, 1), (5, 1), (73, 74), (74, 74), (127, 129), (129, 127), (641, 363)]


@pytest.mark.parametrize("dtype", [np.float32, np.float16])
@pytest.mark.parametrize("offset", [0, 1])
@pytest.mark.parametrize("W,H", SIZES)
def test_color_mse(b, W, H, offset, dtype):
    rng = np.random.default_rng(W * 1000 + H)
    x = rng.uniform(size=(3, H, W)).astype(dtype)
    y = np.clip(x + rng.normal(scale=0.05, size=x.shape), 0, 1).astype(dtype)
    want = exact_square_sum(x.astype(np.float64) - y.astype(np.float64)) / x.size
    got = b.exw_color_mse(on_gpu(x, offset), on_gpu(y, offset))
    assert got == pytest.approx(want, rel=max(16, x.size) * 2.0 ** -53, abs=0)


@pytest.mark.parametrize("offset", [0, 1])
@pytest.mark.parametrize("W,H", SIZES)
def test_mv_variance(b, W, H, offset):
    rng = np.random.default_rng(W * 1000 + H)
    mv = (rng.uniform(-9, 9, size=(2, H, W)) + 2.5).astype(np.float32)
    mv[0][rng.uniform(size=(H, W)) < 0.05] = np.nan
    ok = np.isfinite(mv).all(0)
    got = b.exw_mv_variance(on_gpu(mv, offset))
    assert got[0] == ok.sum()
    if ok.sum() == 0:
        return
    for axis in (0, 1):
        m = mv[axis][ok].astype(np.float64)
        off = m - m[0]
        mean = math.fsum(off.tolist()) / m.size
        sq = exact_square_sum(off) / m.size
        want = sq - mean * mean
        assert got[1 + axis] == pytest.approx(want, rel=0, abs=max(16, m.size) * 2.0 ** -53 * (sq + mean * mean))


@pytest.mark.parametrize("kind", ["tiny", "huge", "mixed"])
def test_values_outside_the_float_path(b, kind):
    rng = np.random.default_rng(7)
    x = rng.uniform(size=(3, 97, 128)).astype(np.float32)
    y = x.copy()
    if kind in ("tiny", "mixed"):  # differences whose squares are subnormal in float32
        x[:, ::3] = (rng.uniform(1, 2, size=x[:, ::3].shape) * 1e-22).astype(np.float32)
        y[:, ::3] = 0.0
    if kind in ("huge", "mixed"):
        x[:, 1::3] = (rng.uniform(1, 2, size=x[:, 1::3].shape) * 1e30).astype(np.float32)
    want = exact_square_sum(x.astype(np.float64) - y.astype(np.float64)) / x.size
    got = b.exw_color_mse(on_gpu(x, 0), on_gpu(y, 0))
    assert got == pytest.approx(want, rel=x.size * 2.0 ** -53, abs=0)
    mv = np.stack([x[0], y[0]])
    off = mv.astype(np.float64) - mv[:, :1, :1].astype(np.float64)
    got = b.exw_mv_variance(on_gpu(mv, 0))
    for axis in (0, 1):
        mean = math.fsum(off[axis].ravel().tolist()) / off[axis].size
        sq = exact_square_sum(off[axis]) / off[axis].size
        assert got[1 + axis] == pytest.approx(max(sq - mean * mean, 0.0), rel=0,
                                              abs=off[axis].size * 2.0 ** -53 * (sq + mean * mean))


def test_non_finite_colours_reach_the_result(b):
    x = np.full((3, 80, 90), 0.5, np.float32)
    y = x.copy()
    y[1, 40, 45] = np.inf
    assert b.exw_color_mse(on_gpu(x, 0), on_gpu(y, 0)) == math.inf
    y[1, 40, 45] = np.nan
    assert math.isnan(b.exw_color_mse(on_gpu(x, 0), on_gpu(y, 0)))


@pytest.mark.parametrize("dtype", [np.float32, np.float16])
@pytest.mark.parametrize("W,H", [(11, 11), (12, 19), (74, 18), (75, 21), (138, 97), (139, 40)])
def test_ssim_strips_and_chunks(b, W, H, dtype):
    # one output, and the edges of a warp's 64 columns and of its rows.  The bar is that of the oracle test: window
    # moments within about 1e-7, and an error e in a variance moves a window's SSIM by at most e / C2 (C2 = 9e-4)
    rng = np.random.default_rng(W + 100 * H)
    x = rng.uniform(size=(3, H, W)).astype(dtype)
    y = np.clip(x + rng.normal(scale=0.08, size=x.shape), 0, 1).astype(dtype)
    g = np.exp(-(np.arange(11) - 5.0) ** 2 / 4.5)
    g /= g.sum()

    def mean(v):
        v = sum(g[i] * v[:, :, i:W - 10 + i] for i in range(11))
        return sum(g[i] * v[:, i:H - 10 + i, :] for i in range(11))

    p, q = x.astype(np.float64), y.astype(np.float64)
    mp, mq = mean(p), mean(q)
    vp, vq, c = mean(p * p) - mp * mp, mean(q * q) - mq * mq, mean(p * q) - mp * mq
    want = (((2 * mp * mq + 1e-4) * (2 * c + 9e-4)) / ((mp * mp + mq * mq + 1e-4) * (vp + vq + 9e-4))).mean()
    for offset in (0, 1):
        assert abs(b.exw_ssim(on_gpu(x, offset), on_gpu(y, offset)) - want) <= 2e-4
