"""GPU check of the tiles without a valid pixel in a recursive chain, whose coarse values and fix-up go with the next
step's clear and splat: more such tiles than blocks take at once, values from several levels up, one, two and five steps
(the counters change places at every step) in a workspace full of garbage, alone and replayed from a captured graph."""
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
@pytest.mark.parametrize("W,H", [(1280, 736), (1001, 467)])
@pytest.mark.parametrize("steps", [1, 2, 5])
def test_chain_equals_the_staged_calls(b, W, H, dtype, steps):
    color, depth, mv = scenes.random_frame(W, H, W + steps, mv_scale=2.0)
    depth[:, W // 3:] = np.nan  # two thirds of the tiles
    depth[:64, :] = np.nan
    c, d, m = (torch.from_numpy(x).cuda() for x in (color.astype(dtype), depth, mv))
    ws = b.workspace(b.exw_workspace_bytes(b.OP_WARP_RECURSIVE, W, H, b.F16 if dtype == np.float16 else b.F32, 1, 1),
                     c.device)
    out = torch.empty((steps, 3, H, W), dtype=c.dtype, device="cuda")
    mask = torch.empty((steps, H, W), dtype=torch.uint8, device="cuda")

    def run():
        ws.fill_(0xA5)
        out.fill_(0.5)
        b.exw_warp_recursive(c, d, m, steps, True, out, mask, ws)

    run()
    first = out.clone()
    sc, sd, sm = c, d, m
    for i in range(steps):
        keys = b.exw_splat_motion(sd, sm, 1, 4)
        want, wmask = b.exw_warp(sc, sd, sm, keys, 1, 4)
        b.exw_fill_holes(want, wmask)
        assert torch.equal(mask[i], wmask) and torch.equal(bits(out[i]), bits(want))
        sd, sm = b.exw_carry_motion(keys, wmask, sd, sm)
        sc = want
    side = torch.cuda.Stream()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=side):
        run()
    for _ in range(2):
        graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(bits(out), bits(first))
