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


def _reach(t):
    """0 finite, 1 infinity, 2 minus infinity, 3 NaN."""
    t = t.double().cpu()
    return (torch.isposinf(t).int() + 2 * torch.isneginf(t).int() + 3 * torch.isnan(t).int())


@pytest.mark.parametrize("value", [float("inf"), float("nan")])
@pytest.mark.parametrize("K,d,H,W", [(5, 1, 9, 64), (7, 2, 30, 128), (11, 4, 70, 64),
                                     (13, 1, 21, 64), (11, 32, 50, 64)])
def test_weight_gradient_reach_of_infinities(K, d, H, W, value):
    """An infinity or a NaN in x reaches the taps that multiply it with a pixel of the gradient,
    and no others: rows of the images past the last gradient row have none (widths are whole
    chunks of 64 pixels, so that no pixel past the row's end takes part).  gz > 0, so the
    reached taps are the value itself."""
    N = 2
    g = torch.Generator(device=DEV).manual_seed(K * H)
    x, gz = ((torch.rand((N, H, W, C), generator=g, device=DEV) + 0.5).to(torch.bfloat16)
             for _ in range(2))
    spots = [(0, 0, 0, 3), (0, H - 1, W - 1, 5), (1, H // 2, W // 3, 7)]
    for n, y, xx, ci in spots:
        x[n, y, xx, ci] = value
    gw, gb, _ = _weight_gradient(x, gz, K, d)
    want = torch.zeros(C, C, K, K, dtype=torch.int32)
    kind = 3 if value != value else 1
    r = K // 2
    for n, y, xx, ci in spots:
        for ky in range(K):
            for kx in range(K):
                py, px = y - (ky - r) * d, xx - (kx - r) * d
                if 0 <= py < H and 0 <= px < W:
                    want[:, ci, ky, kx] = kind
    assert torch.equal(_reach(gw), want)
    assert int(_reach(gb).sum()) == 0


def _convolve(x, w, d, bias=None, backward_of=None):
    """The layer's forward convolution, or with backward_of = its input the backward data one
    of the output gradient x."""
    lib = mca.load()
    N, H, W, _ = x.shape
    K = w.shape[-1]
    wf = torch.empty(K * K, C, C, dtype=torch.int16, device=DEV)
    wb = torch.empty_like(wf)
    assert lib.mca_cnn_prep_weights(w.data_ptr(), C, C, K, C, wf.data_ptr(), wb.data_ptr(),
                                    None) == 0
    out = torch.empty_like(x)
    if backward_of is None:
        rc = lib.mca_cnn_conv(x.data_ptr(), N, H, W, wf.data_ptr(), K, d, C, C, bias.data_ptr(), 0,
                              0, None, out.data_ptr(), None, None)
    else:
        rc = lib.mca_cnn_conv(x.data_ptr(), N, H, W, wb.data_ptr(), K, d, C, C, None, 1, 1,
                              backward_of.data_ptr(), out.data_ptr(), None, None)
    assert rc == 0 and lib.mca_cnn_check(None) == 0
    return out


@pytest.mark.parametrize("value", [float("inf"), float("nan")])
@pytest.mark.parametrize("K,d,H,W", [(5, 1, 9, 70), (7, 2, 30, 50), (9, 1, 17, 64), (11, 4, 70, 90),
                                     (11, 32, 70, 150), (13, 1, 20, 65), (15, 1, 18, 64)])
def test_convolution_reach_of_infinities(K, d, H, W, value):
    """An infinity or a NaN in a pixel reaches the outputs whose window holds it, and no others,
    forward and backward (weights > 0: the reached outputs are the value itself)."""
    N = 2
    g = torch.Generator(device=DEV).manual_seed(K * H)
    x = (torch.rand((N, H, W, C), generator=g, device=DEV) + 0.5).to(torch.bfloat16)
    below = x.clone()
    w = torch.rand((C, C, K, K), generator=g, device=DEV) + 0.5
    spots = [(0, 0, 0, 3), (0, H - 1, W - 1, 5), (1, H // 2, W // 3, 7)]
    for n, y, xx, ci in spots:
        x[n, y, xx, ci] = value
    want = torch.zeros(N, H, W, C, dtype=torch.int32)
    reach = [(i - K // 2) * d for i in range(K)]
    for n, y, xx, _ in spots:
        rows = [y + i for i in reach if 0 <= y + i < H]
        cols = [xx + i for i in reach if 0 <= xx + i < W]
        for yy in rows:
            want[n, yy, cols] = 3 if value != value else 1
    bias = torch.zeros(C, device=DEV)
    assert torch.equal(_reach(_convolve(x, w, d, bias)), want)
    assert torch.equal(_reach(_convolve(x, w, d, backward_of=below)), want)


@pytest.mark.parametrize("value", [float("inf"), float("nan")])
@pytest.mark.parametrize("K,d,H,W", [(5, 1, 9, 70), (7, 2, 30, 50), (11, 4, 70, 90), (11, 4, 5, 40),
                                     (13, 1, 20, 65), (15, 1, 18, 64)])
def test_convolution_reach_of_weights_without_numbers(K, d, H, W, value):
    """An infinite or NaN weight makes its channel's outputs that value where its tap lies inside
    the image, and NaN where the tap's pixel is padding: zero times it (x > 0, weights > 0)."""
    N = 2
    g = torch.Generator(device=DEV).manual_seed(K * H)
    x = (torch.rand((N, H, W, C), generator=g, device=DEV) + 0.5).to(torch.bfloat16)
    w = torch.rand((C, C, K, K), generator=g, device=DEV) + 0.5
    w[3, 5, 0, 1] = value
    w[31, 0, K - 1, K // 2] = value
    want = torch.zeros(N, H, W, C, dtype=torch.int32)
    for co, ky, kx in ((3, 0, 1), (31, K - 1, K // 2)):
        y, xx = torch.meshgrid(torch.arange(H) + (ky - K // 2) * d,
                               torch.arange(W) + (kx - K // 2) * d, indexing="ij")
        inside = (y >= 0) & (y < H) & (xx >= 0) & (xx < W)
        want[..., co] = torch.where(inside, 1 if value == value else 3, 3).int()
    bias = torch.zeros(C, device=DEV)
    assert torch.equal(_reach(_convolve(x, w, d, bias)), want)


@pytest.mark.parametrize("K", [3, 5, 11, 13, 15])
@pytest.mark.parametrize("d", [70, 2 ** 29, 2 ** 30, 2 ** 30 + 1, 2 ** 31 - 1])
def test_dilations_beyond_the_image(K, d):
    """The weight gradient of a dilation beyond the image is that of its centre tap, whatever the
    dilation (four times it no longer fits 32 bits); the convolution refuses a row segment that
    does not fit, whatever its 32-bit products wrap to."""
    N, H, W = 2, 9, 70
    g = torch.Generator(device=DEV).manual_seed(K)
    x, gz = (torch.randn((N, H, W, C), generator=g, device=DEV).to(torch.bfloat16)
             for _ in range(2))
    gw, _, _ = _weight_gradient(x, gz, K, d)
    centre = gz.double().reshape(-1, C).T @ x.double().reshape(-1, C)
    size = gz.double().abs().reshape(-1, C).T @ x.double().abs().reshape(-1, C)
    r = K // 2
    assert bool(((gw[:, :, r, r].double() - centre).abs() <= 1e-5 * size).all())
    gw[:, :, r, r] = 0
    assert int(torch.count_nonzero(gw)) == 0
    if d > 70:
        out, wt = torch.empty_like(x), torch.zeros(K * K, C, C, device=DEV).to(torch.bfloat16)
        for dd in (d, 1431655721, 1431655722, 1431655766):
            assert mca.load().mca_cnn_conv(x.data_ptr(), N, H, W, wt.data_ptr(), K, dd, C, C, None, 0, 0,
                                           None, out.data_ptr(), None, None) == mca.ERR_INVALID_ARG


@pytest.mark.parametrize("K,most", [(3, 224), (5, 112), (7, 70), (9, 53), (11, 40), (13, 33), (15, 28)])
def test_dilations_that_a_layer_may_ask_for(K, most):
    """A convolution takes the dilations whose row segment k_conv_tc's stages hold, and refuses the
    next one, whichever form runs."""
    N, H, W = 1, 3, 20
    x = torch.zeros(N, H, W, C, device=DEV).to(torch.bfloat16)
    out, wt = torch.empty_like(x), torch.zeros(K * K, C, C, device=DEV).to(torch.bfloat16)
    for d, rc in ((most, 0), (most + 1, mca.ERR_INVALID_ARG)):
        assert mca.load().mca_cnn_conv(x.data_ptr(), N, H, W, wt.data_ptr(), K, d, C, C, None, 0, 0,
                                       None, out.data_ptr(), None, None) == rc
    assert mca.load().mca_cnn_check(None) == 0


@pytest.mark.parametrize("K,d,N,H,W", [(5, 1, 2, 17, 500), (5, 20, 1, 33, 47), (5, 60, 1, 96, 130),
                                       (7, 48, 2, 70, 60), (9, 53, 1, 64, 300), (15, 28, 1, 120, 70),
                                       (11, 40, 3, 30, 41), (13, 20, 6, 21, 65), (5, 53, 9, 21, 70),
                                       (11, 4, 2, 40, 150)])
def test_layer_at_the_sizes_where_forms_change(K, d, N, H, W):
    """Forward, backward data and weight gradient on both sides of the rules that choose a form:
    dilations that leave few pixels of a tile, single waves, images of fewer rows than four
    dilations.  FP32 sums of exact BF16 products: 1e-5 of the summed term magnitudes, BF16
    outputs within 2^-8 of the value besides."""
    g = torch.Generator(device=DEV).manual_seed(K * H + d)
    x, gz = (torch.randn((N, H, W, C), generator=g, device=DEV).to(torch.bfloat16)
             for _ in range(2))
    w = (torch.randn((C, C, K, K), generator=g, device=DEV) / (C * K * K) ** 0.5)
    w = w.to(torch.bfloat16).float()
    got = [_convolve(x, w, d, torch.zeros(C, device=DEV)), _convolve(gz, w, d, backward_of=x),
           _weight_gradient(x, gz, K, d)[0]]

    def ref(xv, wv, gzv):
        xv = xv.double().permute(0, 3, 1, 2).cpu().requires_grad_(True)
        wv = wv.double().cpu().requires_grad_(True)
        y = torch.nn.functional.conv2d(xv, wv, padding=d * (K // 2), dilation=d)
        y.backward(gzv.double().permute(0, 3, 1, 2).cpu())
        return [y.detach().permute(0, 2, 3, 1), xv.grad.permute(0, 2, 3, 1), wv.grad]

    want, size = ref(x, w, gz), ref(x.abs(), w.abs(), gz.abs())
    want[1] = torch.where(x.double().cpu() > 0, want[1], 0.1 * want[1])
    for k in range(3):
        half = 2.0 ** -8 * want[k].abs() if k < 2 else 0.0
        assert bool(((got[k].double().cpu() - want[k]).abs() <= half + 1e-5 * size[k]).all())
