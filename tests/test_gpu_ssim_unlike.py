"""GPU check of SSIM on images that share nothing, where every position's distance from 1 is near 1: roundings of it must
not lean to one side, or they move the mean of millions of positions.

Bar: a position's distance is within some 2^-23 of its exact value either way, and the 121 positions that share a pixel
may err together, so a mean of N positions is within 2^-23 sqrt(121 / N) unless the errors lean."""
import math

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


def exact(a, c):
    g = torch.exp(-((torch.arange(11, dtype=torch.float64, device="cuda") - 5) ** 2) / 4.5)
    g /= g.sum()

    def mean(v):
        v = sum(g[i] * v[:, :, i:v.shape[2] - 10 + i] for i in range(11))
        return sum(g[i] * v[:, i:v.shape[1] - 10 + i, :] for i in range(11))

    a, c = a.double(), c.double()
    p, q = mean(a), mean(c)
    va, vc, cov = mean(a * a) - p * p, mean(c * c) - q * q, mean(a * c) - p * q
    s = (2 * p * q + 1e-4) * (2 * cov + 9e-4) / ((p * p + q * q + 1e-4) * (va + vc + 9e-4))
    return float(s.mean()), s.numel()


@pytest.mark.parametrize("seed", [1, 2, 3])
@pytest.mark.parametrize("W,H", [(640, 360), (1280, 720), (1919, 1079)])
def test_unrelated_noise(b, W, H, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    a, c = (torch.rand((3, H, W), device="cuda", generator=gen) for _ in range(2))
    want, n = exact(a, c)
    assert abs(b.exw_ssim(a, c) - want) <= 2.0 ** -23 * math.sqrt(121 / n)
