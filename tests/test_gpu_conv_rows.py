"""What the row forms of the convolution and of the weight gradient owe to the per-tap forms
they replaced: as short FP32 sums, and the same reach of infinities and NaN."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2109_07929_gb300 as mca  # noqa: E402

DEV = "cuda:0"
C = 32


def _weight_gradient(x, gz, K, d):
    """(gw, gb, scratch) of the weight gradient, the scratch filled with a mark before."""
    lib = mca.load()
    N, H, W, _ = x.shape
    gw = torch.empty(C, C, K, K, device=DEV)
    gb = torch.empty(C, device=DEV)
    scratch = torch.full((int(lib.mca_cnn_wgrad_scratch(N, H, W, K)),), -7.0, device=DEV)
    assert lib.mca_cnn_conv_wgrad(x.data_ptr(), gz.data_ptr(), N, H, W, K, d, C, C,
                                  scratch.data_ptr(), gw.data_ptr(), gb.data_ptr(), None) == 0
    assert lib.mca_cnn_check(None) == 0
    return gw, gb, scratch


@pytest.mark.parametrize("K,d,N,H,W", [(11, 8, 11, 187, 187), (11, 4, 16, 100, 100),
                                       (5, 1, 40, 130, 60), (13, 2, 9, 256, 256)])
def test_weight_gradient_partial_sums_are_short(K, d, N, H, W):
    """A partial sum of the row form takes at most as many MMA steps (16 pixels of a row each)
    as one of the per-tap form, 16 image rows of ceil(W / 64) chunks of 64 pixels, and at most
    256: FP32 accumulation on the tensor cores loses about a rounding per step.  The sets
    written in the scratch count the partial sums."""
    g = torch.Generator(device=DEV).manual_seed(K + W)
    x, gz = (torch.rand((N, H, W, C), generator=g, device=DEV).to(torch.bfloat16)
             for _ in range(2))
    _, _, scratch = _weight_gradient(x, gz, K, d)
    size = K * K * C * C
    sets = scratch[:scratch.numel() // size * size].view(-1, size)
    written = int((sets != -7.0).all(dim=1).sum())
    chunks = -(-W // 64)
    whole, rest = divmod(H, 4 * d)
    blocks = whole * d + min(rest, d)            # blocks of four gradient rows per image
    steps = 4 * -(-N * blocks * chunks // written)
    assert steps <= 4 * min(64, 16 * chunks)
