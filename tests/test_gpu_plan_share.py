"""GPU check of the plans that several warps make together (frames of up to 608 tiles): every tile's outputs equal the
staged ones bit for bit, at one tile, at ragged edges, at the last size planned this way and the first planned by one
warp a tile; with one motion everywhere, a motion per object, motions that reach from far (more regions than lanes, more
candidates than a plan stores) and a frame where nothing can land."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2307_12607_gb300 import scenes  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def b():
    if not torch.cuda.is_available():
        pytest.fail("a CUDA GPU is required for the gpu-marked tests")
    from paper_2307_12607_gb300 import build, binding
    build.build()
    return binding


def bits(t):
    return t.view(torch.int16 if t.dtype == torch.float16 else torch.int32)


@pytest.mark.parametrize("dtype", [np.float32, np.float16])
@pytest.mark.parametrize("W,H", [(20, 9), (33, 65), (250, 131), (1024, 608), (1024, 616)])
@pytest.mark.parametrize("motion", ["one", "objects", "far", "none"])
def test_shared_plans_equal_staged(b, W, H, dtype, motion):
    color, depth, mv = scenes.random_frame(W, H, 31 + W, mv_scale={"objects": 9.0, "far": 300.0}.get(motion, 0.0))
    if motion == "one":
        mv[0], mv[1] = 5.75, -3.25
        depth[:] = 40.0 + 0.001 * np.arange(W, dtype=np.float32)
    elif motion == "none":
        mv[:] = np.nan
    c, d, m = (torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in (color.astype(dtype), depth, mv))
    out, mask = b.exw_extrapolate(c, d, m)
    for j in range(3):
        keys = b.exw_splat_motion(d, m, j + 1, 4)
        want, wmask = b.exw_warp(c, d, m, keys, j + 1, 4)
        b.exw_fill_holes(want, wmask)
        assert torch.equal(mask[j], wmask) and torch.equal(bits(out[j]), bits(want))
