"""GPU checks of the fused fill's two paths and of the nodes it leaves to the coarse pass: holes that the 2 x 2 block can
fill (no pyramid, a lazy node), deeper ones, and tiles without a valid pixel whose value comes from lazy nodes of tiles
with scattered holes.  The fused fill equals the staged one bit for bit."""
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
@pytest.mark.parametrize("W,H", [(256, 160), (264, 168), (250, 131), (1000, 320)])
@pytest.mark.parametrize("scattered", [0.0, 0.03, 0.5])
def test_fused_fill_equals_staged(b, W, H, dtype, scattered):
    rng = np.random.default_rng(W + H)
    color, depth, mv = scenes.random_frame(W, H, 9, mv_scale=0.0)
    depth[:] = 40.0 + 0.001 * np.arange(W, dtype=np.float32)
    yy, xx = np.mgrid[0:H, 0:W]
    mv[0], mv[1] = 1.3 + 0.002 * xx, -0.7 + 0.001 * yy  # a motion that varies: no uniform tiles
    depth[rng.uniform(size=(H, W)) < scattered] = np.nan  # scattered holes
    depth[40:136, 64:170] = np.nan                        # whole tiles without a valid pixel
    c, d, m = (torch.from_numpy(x).cuda() for x in (color.astype(dtype), depth, mv))
    ws = b.workspace(b.exw_workspace_bytes(b.OP_EXTRAPOLATE, W, H, b.F16 if dtype == np.float16 else b.F32, 1, 3),
                     c.device)
    out, mask = b.exw_extrapolate(c, d, m, ws=ws)
    st = b.frame_stats(ws)
    assert min(st["tiles_without_valid_pixel"]) > 0
    if scattered < 0.1:  # (at 0.5 most tiles have a hole that level 1 cannot fill)
        assert st["lazy_nodes_computed"]["from_outputs"] > 0
    for j in range(3):
        keys = b.exw_splat_motion(d, m, j + 1, 4)
        want, wmask = b.exw_warp(c, d, m, keys, j + 1, 4)
        b.exw_fill_holes(want, wmask)
        assert torch.equal(mask[j], wmask) and torch.equal(bits(out[j]), bits(want))
