"""GPU check of the SSIM of images that are alike: exactly 1 for equal images, and elsewhere the index's distance from 1
within the rounding of its moments -- second moments of at most 1 through two passes of 11 multiply-adds and the squares
(46 roundings of 2^-24) against a variance term of at least 9e-4, so 46 * 2^-24 / 9e-4 < 3.1e-3 of the distance."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def b():
    if not torch.cuda.is_available():
        pytest.fail("a CUDA GPU is required for the gpu-marked tests")
    from paper_2307_12607_gb300 import build, binding
    build.build()
    return binding


@pytest.mark.parametrize("dtype", [np.float32, np.float16])
@pytest.mark.parametrize("W,H", [(11, 11), (74, 12), (75, 40), (333, 97)])
@pytest.mark.parametrize("noise", [0.0, 1e-4, 0.02])
def test_ssim_of_like_images(b, W, H, dtype, noise):
    rng = np.random.default_rng(W + H)
    x = np.clip(np.cumsum(rng.normal(scale=0.02, size=(3, H, W)), axis=2) + 0.8, 0.0, 1.0).astype(dtype)
    y = np.clip(x + rng.normal(scale=noise, size=x.shape) if noise else x, 0.0, 1.0).astype(dtype)
    got = b.exw_ssim(torch.from_numpy(x).cuda(), torch.from_numpy(y).cuda())
    if noise == 0.0:
        assert got == 1.0
        return
    want = oracle.ssim(x.astype(np.float64), y.astype(np.float64))
    assert abs(got - want) <= 3.1e-3 * (1.0 - want)
