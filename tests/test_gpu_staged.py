"""GPU checks of the staged kernels' fused form: exw_warp_recursive gathers, fills and carries in one kernel, so its
frames equal the staged entry points called one after the other (splat, warp, fill, carry), bit for bit -- at the edges
of the 32 x 32 tiles, with holes that reach every level of the pyramid, with and without the fill."""
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


@pytest.mark.parametrize("fill", [True, False])
@pytest.mark.parametrize("dtype", [np.float32, np.float16])
@pytest.mark.parametrize("W,H", [(1, 1), (1, 70), (2, 33), (31, 32), (33, 31), (64, 64), (97, 95), (257, 130)])
def test_recursive_equals_the_staged_calls(b, W, H, dtype, fill):
    color, depth, mv = scenes.random_frame(W, H, 3 * W + H, depth_levels=5, mv_scale=5.0, invalid_fraction=0.05)
    depth[H // 3:H // 3 + 40, W // 4:W // 4 + 70] = np.nan  # whole tiles, and parts of tiles, without a valid pixel
    c, d, m = (torch.from_numpy(x).cuda() for x in (color.astype(dtype), depth, mv))
    got = b.exw_warp_recursive(c, d, m, 3, fill=fill)
    for out, mask in got:
        keys = b.exw_splat_motion(d, m, 1, 4)
        want, wmask = b.exw_warp(c, d, m, keys, 1, 4)
        if fill:
            b.exw_fill_holes(want, wmask)
        assert torch.equal(mask, wmask) and torch.equal(bits(out), bits(want))
        d, m = b.exw_carry_motion(keys, wmask, d, m)
        c = want


def test_clearing_keys_at_any_address(b):
    # the keys are cleared in 16-byte stores: an odd first or last key stands alone
    for W, H, offset in ((1, 1, 0), (1, 1, 1), (3, 5, 1), (3, 5, 0), (64, 33, 1), (641, 363, 1)):
        buf = torch.full((W * H + offset + 1,), 77, dtype=torch.int64, device="cuda")
        keys = buf[offset:offset + W * H].view(H, W)
        depth = torch.full((H, W), float("nan"), device="cuda")
        b.exw_splat_motion(depth, torch.zeros((2, H, W), device="cuda"), 1, 4, keys)
        assert (keys == b.KEY_EMPTY).all() and buf[-1].item() == 77 and (offset == 0 or buf[0].item() == 77)
