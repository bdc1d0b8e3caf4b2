"""GPU check that the masks of the fused calls are outputs only: a caller with no use for them may hand the same plane to
every fraction, frame and stream, and the colours -- the coarse values of tiles without a valid pixel among them, which
are computed from what the other tiles held -- are those of the call with a plane each."""
import struct

import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

NF = 3
CASES = [(256, 192, torch.float32, True), (256, 192, torch.float16, True), (256, 192, torch.float32, False),
         (250, 170, torch.float32, True), (250, 171, torch.float16, True), (231, 173, torch.float16, True)]


@pytest.fixture(scope="module")
def b():
    if not torch.cuda.is_available():
        pytest.fail("a CUDA GPU is required for the gpu-marked tests")
    from paper_2307_12607_gb300 import build, binding
    build.build()
    return binding


def scene(W, H, dtype, seed):
    """A moving plane whose upper left corner carries no source (the 64 x 64 pixels there, a whole node of the first coarse
    level, stay without a valid pixel) and with lone source pixels missing everywhere: their holes lie at other places in
    each fraction, nearly all with a valid pixel in their 2 x 2 block, in the tiles the corner's coarse value is made of."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    color = torch.rand(3, H, W, device="cuda", generator=g).to(dtype)
    depth = 10.0 + 0.1 * torch.rand(H, W, device="cuda", generator=g)
    depth[torch.rand(H, W, device="cuda", generator=g) < 0.02] = float("nan")
    depth[:80, :80] = float("nan")
    mv = torch.empty(2, H, W, device="cuda")
    mv[0], mv[1] = 9.0 + seed, -6.0
    mv[:, :, W // 2 + 40:] += torch.rand(2, H, W - W // 2 - 40, device="cuda", generator=g)
    return color, depth, mv


@pytest.mark.parametrize("W,H,dtype,tma", CASES)
def test_one_mask_plane_for_every_output(b, W, H, dtype, tma):
    frames = [scene(W, H, dtype, s) for s in range(2)]
    color, depth, mv = (torch.stack(t) for t in zip(*frames))
    want, mask = b.exw_extrapolate(color, depth, mv, nfrac=NF, tma=tma)
    tiles = mask[:, :, :H // 32 * 32, :W // 32 * 32].unflatten(3, (-1, 32)).unflatten(2, (-1, 32))
    assert bool((tiles != 0).all(5).all(3).any()), "no tile without a valid pixel"
    out, scratch = torch.empty_like(want), torch.empty(H, W, dtype=torch.uint8, device="cuda")
    step = 3 * W * H * out.element_size()
    outs = struct.pack(f"@{4 * NF}P", *[p for q in range(2 * NF) for p in (out.data_ptr() + q * step, scratch.data_ptr())])
    ws = b.workspace(b.exw_workspace_bytes(b.OP_EXTRAPOLATE, W, H, b._cdt(color), 2, NF), color.device)
    for _ in range(3):
        out.fill_(float("nan"))
        b._check(b.lib().exw_extrapolate(b._frames(color, depth, mv, 2, W, H, b._cdt(color)), 2, NF,
                                         0 if tma else b.FLAG_NO_TMA, outs, ws.data_ptr(), ws.numel(),
                                         torch.cuda.current_stream().cuda_stream))
        assert torch.equal(out, want)


def test_one_mask_plane_for_every_stream(b):
    streams = [scene(W, H, dtype, s) for s, (W, H, dtype, _) in enumerate(CASES)]
    want = b.exw_extrapolate_batched(streams, nfrac=NF)
    outs = [(torch.empty_like(o), m) for o, m in want]
    scratch = torch.empty(max(d.numel() for _, d, _ in streams), dtype=torch.uint8, device="cuda")
    vals = []
    for (c, d, m), (o, _) in zip(streams, outs):
        H, W = d.shape
        vals += (c.data_ptr(), d.data_ptr(), m.data_ptr(), W, H, b._cdt(c))
        for j in range(NF):
            vals += (o[j].data_ptr(), scratch.data_ptr())
    ws = b.workspace(b.exw_batched_workspace_bytes(streams, NF), streams[0][0].device)
    descs = struct.pack("@" + b._STREAM * len(streams), *vals)
    for _ in range(3):
        for o, _ in outs:
            o.fill_(float("nan"))
        b._check(b.lib().exw_extrapolate_batched(descs, len(streams), NF, 0, ws.data_ptr(), ws.numel(), None,
                                                 torch.cuda.current_stream().cuda_stream))
        for (o, _), (w, _) in zip(outs, want):
            assert torch.equal(o, w)
