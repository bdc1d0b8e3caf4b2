"""GPU check of the target offset floor(1/2 + k mv / denom) against exact rational arithmetic, at the values where a
rounding could go wrong: every half-integer boundary of k mv / denom and its float neighbours, subnormal and tiny
motions, the largest that can land and the smallest that cannot, for every denominator and its smallest and largest
fractions.  One row of pixels far apart in a wide frame; each lands where the exact offset says, or nowhere."""
import math
from fractions import Fraction

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


def motions(k, denom):
    vals = [0.0, -0.0, 1e-45, -1e-45, 1e-38, -1e-30, 2.0 ** -26, -(2.0 ** -25), 65535.97, -65536.0, 1048575.9, -1048576.0,
            1048576.0, 3e9, -3e9, 1e30, math.inf, -math.inf, math.nan]
    for i in list(range(-40, 41)) + [-8191, -1000, 777, 4095, 8190]:
        x = np.float32((i + 0.5) * denom / max(k, 1))
        vals += [x, np.nextafter(x, np.float32(np.inf)), np.nextafter(x, np.float32(-np.inf)), np.float32(i)]
    return np.array(vals, np.float32)


@pytest.mark.parametrize("axis", [0, 1])
@pytest.mark.parametrize("denom", [1, 2, 4, 8, 64])
def test_offsets_are_exact(b, denom, axis):
    n = 16384
    W, H = (n, 1) if axis == 0 else (1, n)
    for k in sorted({0, 1, denom // 2, denom - 1, denom}):
        vals = motions(k, denom)
        for start in range(0, len(vals), 4):
            for at, v in zip((5, 8191, 8192, 16380), vals[start:start + 4]):
                depth = torch.full((H, W), float("nan"), device="cuda")
                mv = torch.zeros((2, H, W), device="cuda")
                depth.view(-1)[at] = 1.0
                mv[axis].view(-1)[at] = float(v)
                keys = b.exw_splat_motion(depth, mv, k, denom).view(-1)
                got = torch.nonzero(keys != b.KEY_EMPTY).view(-1).tolist()
                want = []
                # (k = 0 leaves a pixel where it is for motions below 2^23 denom, the range of the definition)
                if np.isfinite(v) and (k > 0 or abs(float(v)) < 2.0 ** 23 * denom):
                    t = at + math.floor(Fraction(1, 2) + Fraction(k, denom) * Fraction(float(v)))
                    want = [t] if 0 <= t < n else []
                assert got == want, (k, denom, float(v), at)
