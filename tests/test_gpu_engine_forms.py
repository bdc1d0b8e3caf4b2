"""GPU checks of both forms of the engine kernel -- the common one, which every launch of aligned frames takes, and the one
with loader warps -- over one to three fractions: each call against the staged kernels (splat, warp, fill), which have
neither plans nor windows, and the host-injected wait that runs out, which each form has to leave by its own barriers."""
import os

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2307_12607_gb300 import scenes  # noqa: E402

pytestmark = pytest.mark.gpu

FORMS = {"common": [(256, 144, torch.float16), (320, 180, torch.float32), (200, 120, torch.float16)],
         "loaders": [(254, 144, torch.float16), (321, 180, torch.float32), (198, 121, torch.float16)]}


@pytest.fixture(scope="module")
def b():
    if not torch.cuda.is_available():
        pytest.fail("a CUDA GPU is required for the gpu-marked tests")
    from paper_2307_12607_gb300 import build, binding
    build.build()
    return binding


def streams_of(form, seed=0):
    streams = []
    for i, (W, H, dt) in enumerate(FORMS[form]):
        if i % 2:  # splat tiles throughout, invalid sources, ties
            c, d, m = scenes.random_frame(W, H, seed + i, depth_levels=3, mv_scale=5.0, invalid_fraction=0.05)
        else:      # smooth, uniform and splat tiles
            c, d, m = scenes.render(scenes.make_scene(W, H, seed + i, 6, vmax=9.0, pan_max=3.0), 0.0)
        streams.append((torch.from_numpy(np.ascontiguousarray(c)).to(dt).cuda(), torch.from_numpy(d).cuda(),
                        torch.from_numpy(m).cuda()))
    return streams


def staged(b, c, d, m, k, fill):
    keys = b.exw_splat_motion(d, m, k, 4)
    out, mask = b.exw_warp(c, d, m, keys, k, 4)
    return (b.exw_fill_holes(out, mask) if fill else out), mask


def assert_staged(b, stream, out, mask, nfrac, fill):
    for j in range(nfrac):
        want, wmask = staged(b, *stream, j + 1, fill)
        assert torch.equal(mask[j], wmask) and torch.equal(out[j], want)


@pytest.mark.parametrize("fill", [True, False])
@pytest.mark.parametrize("nfrac", [1, 2, 3])
@pytest.mark.parametrize("form", list(FORMS))
def test_every_number_of_fractions(b, form, nfrac, fill):
    streams = streams_of(form)
    for stream in streams:  # one frame: its plans by four warps a tile
        out, mask = b.exw_extrapolate(*stream, nfrac=nfrac, fill=fill)
        assert_staged(b, stream, out, mask, nfrac, fill)
    outs = b.exw_extrapolate_batched(streams, nfrac=nfrac, fill=fill)  # the others' plans in the engine
    for stream, (out, mask) in zip(streams, outs):
        assert_staged(b, stream, out, mask, nfrac, fill)


@pytest.mark.parametrize("form", list(FORMS))
def test_a_wait_that_runs_out_leaves_the_context_usable(b, form):
    streams = streams_of(form, seed=3)
    ws = b.workspace(b.exw_batched_workspace_bytes(streams, 3), "cuda")
    os.environ["EXW_FAULT"] = "timeout"
    try:
        b.exw_extrapolate_batched(streams, 3, ws=ws)
        torch.cuda.synchronize()
        assert b.exw_device_status(ws) == 4          # EXW_ERR_TIMEOUT
    finally:
        del os.environ["EXW_FAULT"]
    outs = b.exw_extrapolate_batched(streams, 3, ws=ws)
    torch.cuda.synchronize()
    assert b.exw_device_status(ws) == 0
    for stream, (out, mask) in zip(streams, outs):
        assert_staged(b, stream, out, mask, 3, True)
