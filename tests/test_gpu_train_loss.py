"""GPU check of the training pass's losses over several frames: a frame's loss is summed with the next frame's clear, the
last one's by itself, so the losses and gradients of a call over n frames equal those of n calls over one frame bit for
bit -- at one pixel, one tile, ragged edges and more tiles than the sum has threads, in a workspace full of garbage."""
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


@pytest.mark.parametrize("dtype", [np.float32, np.float16])
@pytest.mark.parametrize("W,H", [(1, 1), (32, 32), (33, 65), (643, 517)])
@pytest.mark.parametrize("n", [1, 2, 5])
def test_losses_equal_one_frame_calls(b, W, H, dtype, n):
    rng = np.random.default_rng(W + H + n)
    frames = [scenes.random_frame(W, H, 7 * i + W, mv_scale=4.0, invalid_fraction=0.02) for i in range(n)]
    c, d, m = (torch.from_numpy(np.stack([f[j] for f in frames]).astype(dtype if j == 0 else np.float32)).cuda()
               for j in range(3))
    target = torch.from_numpy(rng.uniform(size=(n, 3, 3, H, W)).astype(dtype)).cuda()
    ws = b.workspace(b.exw_workspace_bytes(b.OP_WARP_L2_GRAD, W, H, b.F16 if dtype == np.float16 else b.F32, 1, 3),
                     c.device)
    ws.fill_(0xA5)
    got = b.exw_warp_l2_grad(c, d, m, target, 3, ws=ws)
    for i in range(n):
        ws.fill_(0x5A)
        want = b.exw_warp_l2_grad(c[i:i + 1], d[i:i + 1], m[i:i + 1], target[i:i + 1], 3, ws=ws)
        for g, w in zip(got, want):
            assert torch.equal(g[i:i + 1], w)
