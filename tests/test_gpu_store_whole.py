"""GPU check that the storing entry points write every element of their gradients and read none: buffers full of NaN end
with the bits that accumulating into zeros gives, at sizes below and above one CTA's tile and a megabyte."""
import struct

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2307_12607_gb300 import scenes  # noqa: E402

pytestmark = pytest.mark.gpu

SIZES = [(1, 1), (33, 31), (97, 95), (641, 363)]


@pytest.fixture(scope="module")
def b():
    if not torch.cuda.is_available():
        pytest.fail("a CUDA GPU is required for the gpu-marked tests")
    from paper_2307_12607_gb300 import build, binding
    build.build()
    return binding


def frames(F, W, H, dtype):
    f = [scenes.random_frame(W, H, 5 * W + H + i, depth_levels=2, mv_scale=3.0, invalid_fraction=0.05) for i in range(F)]
    c, d, m = (torch.from_numpy(np.stack([x[j] for x in f])).cuda() for j in range(3))
    return c.to(dtype), d, m


def nan(*shape):
    return torch.full(shape, float("nan"), device="cuda")


def same(x, y):
    return torch.equal(x.view(torch.int32), y.view(torch.int32))


@pytest.mark.parametrize("dtype", [torch.float32, torch.float16])
@pytest.mark.parametrize("W,H", SIZES)
def test_backward(b, W, H, dtype):
    c, d, m = (t[0] for t in frames(1, W, H, dtype))
    g = torch.randn((3, H, W), device="cuda")
    keys = b.exw_splat_motion(d, m, 2, 4)
    want = b.exw_warp_backward(g, c, d, m, keys, 2, 4, torch.zeros((3, H, W), device="cuda"),
                               torch.zeros((2, H, W), device="cuda"))
    gc, gm = nan(3, H, W), nan(2, H, W)
    b._check(b.lib().exw_warp_backward_store(g.data_ptr(), c.data_ptr(), b._cdt(c), d.data_ptr(), m.data_ptr(),
                                             keys.data_ptr(), W, H, 2, 4, gc.data_ptr(), gm.data_ptr(), None, 0,
                                             torch.cuda.current_stream().cuda_stream))
    assert same(gc, want[0]) and same(gm, want[1])


@pytest.mark.parametrize("dtype", [torch.float32, torch.float16])
@pytest.mark.parametrize("W,H", SIZES)
def test_training_pass(b, W, H, dtype):
    F, nfrac = 2, 3
    c, d, m = frames(F, W, H, dtype)
    t = torch.rand((F, nfrac, 3, H, W), device="cuda").to(dtype)
    want = b.exw_warp_l2_grad(c, d, m, t, nfrac, grad_color=torch.zeros((F, 3, H, W), device="cuda"),
                              grad_mv=torch.zeros((F, 2, H, W), device="cuda"))
    gc, gm, loss = nan(F, 3, H, W), nan(F, 2, H, W), torch.full((F,), float("nan"), dtype=torch.float64, device="cuda")
    ws = b.workspace(b.exw_workspace_bytes(b.OP_WARP_L2_GRAD, W, H, b._cdt(c), 1, nfrac), "cuda")
    desc = struct.pack("@" + b._TRAIN * F, *[
        v for f in range(F)
        for v in (c[f].data_ptr(), d[f].data_ptr(), m[f].data_ptr(), W, H, b._cdt(c),
                  *(t[f, j].data_ptr() for j in range(nfrac)), gc[f].data_ptr(), gm[f].data_ptr())])
    b._check(b.lib().exw_warp_l2_grad_store(desc, F, nfrac, loss.data_ptr(), ws.data_ptr(), ws.numel(),
                                            torch.cuda.current_stream().cuda_stream))
    assert torch.equal(loss, want[0]) and same(gc, want[1]) and same(gm, want[2])
