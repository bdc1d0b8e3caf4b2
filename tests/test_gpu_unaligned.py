"""GPU checks of the engine's loader warps: frames whose rows or base addresses are not multiples of 16 bytes are staged
into the same shared-memory windows as TMA's (half colour of odd width excepted), so their results equal the
global-memory reads (tma=False) bit for bit -- at every remainder of a row modulo 16 bytes, for both colour types, at
bases off by one element, in frames smaller than a window and in batches that mix both kinds of streams."""
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


def on_gpu(x, offset=0):
    """x on the GPU, its first element ``offset`` elements past a 256-byte boundary."""
    buf = torch.zeros(x.size + offset, dtype=torch.from_numpy(x).dtype, device="cuda")
    t = buf[offset:].view(x.shape)
    t.copy_(torch.from_numpy(x))
    return t


def frame(W, H, dtype, kind):
    if kind == "scene":  # smooth, uniform and splat tiles
        color, depth, mv = scenes.render(scenes.make_scene(W, H, W * 7 + H, 6, vmax=9.0, pan_max=3.0), 0.0)
    else:                # splat tiles throughout, invalid sources, ties
        color, depth, mv = scenes.random_frame(W, H, W + H, depth_levels=3, mv_scale=5.0, invalid_fraction=0.05)
    return color.astype(dtype), depth, mv


def bits(t):
    return t.view(torch.int16 if t.dtype == torch.float16 else torch.int32)


@pytest.mark.parametrize("kind", ["scene", "random"])
@pytest.mark.parametrize("dtype", [np.float32, np.float16])
@pytest.mark.parametrize("W,H", [(1, 1), (3, 70), (33, 31), (62, 65), (190, 97), (257, 130), (258, 129), (259, 128),
                                 (260, 127), (261, 126), (262, 125), (263, 124)])
def test_every_row_remainder(b, W, H, dtype, kind):
    color, depth, mv = frame(W, H, dtype, kind)
    c, d, m = on_gpu(color), on_gpu(depth), on_gpu(mv)
    ws = b.workspace(b.exw_workspace_bytes(b.OP_EXTRAPOLATE, W, H, b.F16 if dtype == np.float16 else b.F32, 1, 3),
                     c.device)
    for fill in (True, False):
        out, mask = b.exw_extrapolate(c, d, m, fill=fill, ws=ws)
        st = b.frame_stats(ws)
        if W > 200 and (dtype == np.float32 or W % 2 == 0):
            assert st["tiles_window_all"] > 0
            assert kind != "scene" or st["tiles_smooth"] > 0
        want, wmask = b.exw_extrapolate(c, d, m, fill=fill, tma=False)
        assert torch.equal(mask, wmask) and torch.equal(bits(out), bits(want))
        assert b.exw_device_status(ws) == 0


@pytest.mark.parametrize("dtype", [np.float32, np.float16])
@pytest.mark.parametrize("offsets", [(1, 0, 0), (0, 1, 0), (0, 0, 3), (3, 1, 2), (4, 2, 2)])
def test_bases_off_a_16_byte_boundary(b, dtype, offsets):
    color, depth, mv = frame(320, 160, dtype, "scene")
    c, d, m = (on_gpu(x, o) for x, o in zip((color, depth, mv), offsets))
    out, mask = b.exw_extrapolate(c, d, m)
    want, wmask = b.exw_extrapolate(on_gpu(color), on_gpu(depth), on_gpu(mv))
    assert torch.equal(mask, wmask) and torch.equal(bits(out), bits(want))


def test_mixed_streams(b):
    sizes = [(320, 180, np.float32), (321, 180, np.float32), (256, 144, np.float16), (250, 141, np.float16),
             (135, 77, np.float16), (64, 64, np.float32), (66, 63, np.float32)]
    frames = [frame(W, H, t, "scene" if i % 3 else "random") for i, (W, H, t) in enumerate(sizes)]
    streams = [tuple(on_gpu(x) for x in f) for f in frames]
    for _ in range(3):
        outs = b.exw_extrapolate_batched(streams)
        for (c, d, m), (out, mask) in zip(streams, outs):
            want, wmask = b.exw_extrapolate(c, d, m, tma=False)
            assert torch.equal(mask, wmask) and torch.equal(bits(out), bits(want))
