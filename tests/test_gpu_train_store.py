"""GPU checks of the gradients that are stored instead of accumulated (the binding's case of no gradient passed in): the
same bits as accumulating into zeros, whatever the buffers held, at the edges of the 32 x 32 source tiles, for residuals
of every sign (the taps' directions) and for one to three fractions."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2307_12607_gb300 import scenes  # noqa: E402

pytestmark = pytest.mark.gpu

SIZES = [(1, 1), (2, 40), (31, 33), (33, 31), (64, 64), (97, 95), (200, 70)]


@pytest.fixture(scope="module")
def b():
    if not torch.cuda.is_available():
        pytest.fail("a CUDA GPU is required for the gpu-marked tests")
    from paper_2307_12607_gb300 import build, binding
    build.build()
    return binding


def frames(F, W, H, dtype):
    f = [scenes.random_frame(W, H, 5 * W + H + i, depth_levels=2, mv_scale=3.0, quarter_grid=bool(i % 2),
                             invalid_fraction=0.05) for i in range(F)]
    c, d, m = (torch.from_numpy(np.stack([x[j] for x in f])).cuda() for j in range(3))
    return c.to(dtype), d, m


def poison(b):
    """Fill torch's free memory with NaN, so that a value read before it is written shows."""
    torch.full((1 << 22,), float("nan"), device="cuda")


@pytest.mark.parametrize("dtype", [torch.float32, torch.float16])
@pytest.mark.parametrize("W,H", SIZES)
def test_backward_stores_what_it_would_add_to_zeros(b, W, H, dtype):
    c, d, m = (t[0] for t in frames(1, W, H, dtype))
    g = torch.randn((3, H, W), device="cuda")
    for k in (1, 3):
        want = b.exw_warp_backward(g, c, d, m, None, k, 4, torch.zeros((3, H, W), device="cuda"),
                                   torch.zeros((2, H, W), device="cuda"))
        poison(b)
        got = b.exw_warp_backward(g, c, d, m, None, k, 4)
        for x, y in zip(got, want):
            assert torch.equal(x.view(torch.int32), y.view(torch.int32))


@pytest.mark.parametrize("nfrac", [1, 3])
@pytest.mark.parametrize("dtype", [torch.float32, torch.float16])
@pytest.mark.parametrize("W,H", SIZES)
def test_training_pass_stores_what_it_would_add_to_zeros(b, W, H, dtype, nfrac):
    F = 2
    c, d, m = frames(F, W, H, dtype)
    t = torch.rand((F, nfrac, 3, H, W), device="cuda").to(dtype)
    gc, gm = torch.zeros((F, 3, H, W), device="cuda"), torch.zeros((F, 2, H, W), device="cuda")
    want = b.exw_warp_l2_grad(c, d, m, t, nfrac, grad_color=gc, grad_mv=gm)
    poison(b)
    got = b.exw_warp_l2_grad(c, d, m, t, nfrac)
    assert torch.equal(got[0], want[0])
    for x, y in zip(got[1:], want[1:]):
        assert torch.equal(x.view(torch.int32), y.view(torch.int32))
