"""GPU check of the rule that gives a launch loader warps only where the streams TMA cannot stage hold 5% of its tiles: on
both sides of the line every stream's outputs are those of its own call, and the unaligned stream's tiles have windows
on one side only."""
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


def stream(W, H, dtype, seed):
    color, depth, mv = scenes.render(scenes.make_scene(W, H, seed, 6, vmax=9.0, pan_max=3.0), 0.0)
    return tuple(torch.from_numpy(x).cuda() for x in (color.astype(dtype), depth, mv))


# the unaligned stream holds 28 tiles; 532 aligned ones make 5.0%, one tile more makes less
@pytest.mark.parametrize("fill", [True, False])
@pytest.mark.parametrize("dtype", [np.float32, np.float16])
@pytest.mark.parametrize("aligned,loaders", [((19 * 32, 28 * 32), True), ((13 * 32, 41 * 32), False)])
def test_both_sides_of_the_line(b, aligned, loaders, dtype, fill):
    streams = [stream(*aligned, dtype, 1), stream(222, 122, dtype, 2)]
    ws = b.workspace(b.exw_batched_workspace_bytes(streams, 3), streams[0][0].device)
    outs = b.exw_extrapolate_batched(streams, fill=fill, ws=ws)
    st = b.frame_stats(ws, 1)
    assert (st["tiles_window_all"] + st["tiles_smooth"] + st["tiles_uniform"] > 0) == loaders
    for (c, d, m), (out, mask) in zip(streams, outs):
        want, wmask = b.exw_extrapolate(c, d, m, fill=fill, tma=False)
        assert torch.equal(mask, wmask) and torch.equal(out, want)
    assert b.exw_device_status(ws) == 0
