"""The Krylov vector kernels at the sizes where their pairs of entries, half-block sums and
per-length instantiations can go wrong: odd and even rows and columns, a pair across a row
and across the two layers, one, two and three entries per accumulator, one to 30 basis
vectors, buffers off the 16-byte boundary."""
import numpy as np
import pytest

import mca_inputs as mi
from oracle import mca_oracle as O

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2109_07929_gb300 as mca  # noqa: E402

DEV = "cuda:0"


def _off(shape, off, dtype=torch.float64):
    """A contiguous tensor whose data starts `off` entries into its allocation."""
    n = int(np.prod(shape))
    return torch.empty(n + 2, dtype=dtype, device=DEV)[off:off + n].view(shape)


@pytest.mark.parametrize("off", [0, 1])
@pytest.mark.parametrize("m,n", [(1, 2), (3, 5), (5, 4), (2, 256), (31, 130), (33, 47),
                                 (700, 300), (3, 1025)])
def test_apply_does_not_depend_on_alignment(m, n, off):
    """w = J z of the paired kernel (even n, 16-byte boundaries) and of the single-cell one:
    the same operations per cell, so the same bits; against the oracle's FP64 product within
    1e-14 of 8 |z|_max (the bound of the FP64 apply)."""
    cb = mi.make_crossbar(m, n, 3, nvec=2)
    rng = np.random.default_rng(m * n)
    D = np.abs(rng.standard_normal((2, m * n))) * 1e-5
    z = rng.standard_normal((2, 2 * m * n))
    p = cb.params
    with mca.Solver(mca.default_params(m, n, max_batch=2, flags=0), cb.gmap) as s:
        Dd, zd, w = _off(D.shape, off), _off(z.shape, off), _off(z.shape, off)
        Dd.copy_(torch.as_tensor(D))
        zd.copy_(torch.as_tensor(z))
        s.jacobian_apply(Dd, zd, w)
        z32, w32 = _off(z.shape, off, torch.float32), _off(z.shape, off)
        z32.copy_(zd.float())
        s.jacobian_apply_f32(Dd, z32, w32)
        ref, ref32 = _off(z.shape, 1), _off(z.shape, 1)
        s.jacobian_apply(Dd, zd, ref)
        s.jacobian_apply_f32(Dd, z32, ref32)
    assert torch.equal(w, ref) and torch.equal(w32, ref32)
    zero = np.zeros(m * n)
    for v in range(2):
        J = O.jacobian(p, D[v].reshape(m, n), zero, zero)
        assert np.abs(w[v].cpu().numpy() - J @ z[v]).max() <= 1e-14 * 8 * np.abs(z[v]).max()


@pytest.mark.parametrize("off", [0, 1])
@pytest.mark.parametrize("m,n,nvec", [(1, 3, 1), (5, 7, 2), (16, 130, 3), (64, 64, 1),
                                      (640, 255, 1), (300, 512, 2), (768, 700, 1)])
def test_gmres_reaches_its_tolerance(m, n, nvec, off):
    """Restarted GMRES on J dx = rhs with the Jacobi preconditioner (long cycles, all basis
    lengths; dx on and off a 16-byte boundary): the cycle's own residual estimate equals the
    true residual of dx to 1e-6 (CGS with selective reorthogonalisation keeps the estimate
    exact to about 30 * 1e-8)."""
    cb = mi.make_crossbar(m, n, 5, nvec=nvec, gdist="uniform_paper", g_src=1.0,
                          g_term_top_right=1.0, g_term_bot_top=1.0, g_sense=1.0, b=0.0)
    p = cb.params
    prm = mca.default_params(m, n, g_src=1.0, g_term_top_right=1.0, g_term_bot_top=1.0,
                             g_sense=1.0, b=0.0, precision=mca.PREC_JACOBI, max_batch=nvec)
    D = np.tile(cb.gmap.reshape(1, -1), (nvec, 1))
    rhs = np.random.default_rng(7).standard_normal((nvec, 2 * m * n))
    with mca.Solver(prm, cb.gmap) as s:
        dx = _off(rhs.shape, off)
        Dd, rd = torch.as_tensor(D, device=DEV), torch.as_tensor(rhs, device=DEV)
        its, est = s.gmres_solve(Dd, D.mean(axis=1), rd, dx, 1e-9)
    x = dx.cpu().numpy()
    zero = np.zeros(m * n)
    for v in range(nvec):
        r = np.linalg.norm(rhs[v] - O.jacobian(p, cb.gmap, zero, zero) @ x[v])
        scale = np.linalg.norm(rhs[v])
        assert its[v] >= 1 and abs(r - est[v]) <= 1e-6 * r + 1e-13 * scale


@pytest.mark.parametrize("m,n", [(2, 2), (1, 31), (32, 33), (31, 64), (65, 2), (100, 1025),
                                 (2049, 3), (3, 2049), (1057, 40)])
def test_mhat_line_solves_in_chunks(m, n):
    """The paper's M_hat with every line cut into 32 chunks: lines shorter than 32 nodes, whole
    and partly filled chunks, empty ones.  Each of the two solves is backward stable, so z_t
    is within about 16 eps kappa of exact per solve (kappa <= (4 + a) / a: 7e-10 in all), and
    z_b follows it; the oracle forms z_b from z_t with an error of its own of a few eps times
    the operator's terms, 4 |z_t| / a."""
    cb = mi.make_crossbar(m, n, 4, g_wire_bot=0.5)
    p = cb.params
    r = np.random.default_rng(7).standard_normal((3, 2 * m * n))
    a = np.array([2.1e-5, 7.0e-4, 0.2])
    prm = mca.default_params(m, n, g_wire_bot=0.5, precision=mca.PREC_MHAT, max_batch=3)
    with mca.Solver(prm, cb.gmap) as s:
        z = torch.empty(3, 2 * m * n, dtype=torch.float64, device=DEV)
        s.precond_apply(a, torch.as_tensor(r, device=DEV), z)
        z = z.cpu().numpy()
    for v in range(3):
        z1, z2 = O.precond_apply_block(p, None, a[v], a[v], r[v, :m * n], r[v, m * n:],
                                       minv=lambda w: O.mhat_apply_inverse(p, a[v], a[v], w))
        n1, n2 = np.linalg.norm(z1), np.linalg.norm(z2)
        assert np.linalg.norm(z[v, :m * n] - z1) <= 1e-9 * n1
        assert (np.linalg.norm(z[v, m * n:] - z2) <=
                1e-9 * n2 + 16 * 1.1e-16 * 4 / a[v] * n1)


@pytest.mark.parametrize("m,n", [(1, 1), (1, 33), (5, 130), (129, 65), (64, 257), (2, 4100)])
def test_fp64_preconditioner_in_slices(m, n):
    """The FP64 transforms on BF16 slices: ragged tiles and K, and (4100) a K beyond one FP32
    accumulator.  P z = r within the eigenvectors' own accuracy (1e-9, the bar of their parity
    test) of |P| |z|; scaling r by 2^-980 scales z exactly (every row's slices are relative to
    its exponent); a NaN reaches the output."""
    cb = mi.make_crossbar(m, n, 4)
    p = cb.params
    rng = np.random.default_rng(7)
    r = rng.uniform(0.5, 1.0, (2, 2 * m * n)) * rng.choice([-1.0, 1.0], (2, 2 * m * n))
    r[1, : m * n] *= 10.0 ** rng.uniform(-8, 0, m * n)
    a = np.array([2.1e-5, 0.2])
    with mca.Solver(mca.default_params(m, n, precision=mca.PREC_FP64, max_batch=2), cb.gmap) as s:
        rd = torch.as_tensor(r, device=DEV)
        z, zs, zn = (torch.empty_like(rd) for _ in range(3))
        s.precond_apply(a, rd, z)
        s.precond_apply(a, rd * 2.0 ** -980, zs)
        rd[0, 0] = float("nan")
        s.precond_apply(a, rd, zn)
    assert torch.equal(zs, z * 2.0 ** -980)
    assert bool(torch.isnan(zn[0]).any()) and torch.equal(zn[1], z[1])
    z = z.cpu().numpy()
    for v in range(2):
        P = O.precond_matrix(p, a[v], a[v])
        size = 5.0 + 2 * a[v]                      # |P| <= 4 g + 2 a, plus the terminations
        assert np.linalg.norm(P @ z[v] - r[v]) <= 1e-9 * size * np.linalg.norm(z[v])


@pytest.mark.parametrize("n", [512, 4000])
def test_fp64_slices_of_coherent_rows(n):
    """A constant right-hand side against the nearly constant lowest mode: the slice products of
    a weight all have one sign and sum beyond 2^24 unless K is cut.  Extended-precision sums
    with the handle's own eigenpairs; rounding stays within 4 transforms x n ulps."""
    cb = mi.make_crossbar(1, n, 4)
    weak = dict(g_src=1e-12, g_term_top_right=1e-12)
    with mca.Solver(mca.default_params(1, n, precision=mca.PREC_FP64, max_batch=1, **weak),
                    cb.gmap) as s:
        mu, qr, nu, _ = s.eigenpairs()
        a = 2.1e-5
        z = torch.empty(1, 2 * n, dtype=torch.float64, device=DEV)
        s.precond_apply(np.array([a]), torch.full_like(z, 63.4921875 / 32), z)
    ld = np.longdouble
    x = qr.astype(ld).T @ np.full(n, 63.4921875 / 32, ld)
    mu, nu0, a = mu.astype(ld), ld(nu[0]), ld(a)
    det = mu * nu0 + mu * a + nu0 * a
    ref = np.concatenate([qr.astype(ld) @ ((nu0 + a + a) * x / det),
                          qr.astype(ld) @ ((mu + a + a) * x / det)])
    err = np.abs(z.cpu().numpy()[0] - ref).max() / np.abs(ref).max()
    assert err <= 4 * n * 2.0 ** -53


@pytest.mark.parametrize("m,n,nvec", [(5, 130, 1), (129, 65, 2)])
def test_fp64_preconditioner_of_part_of_a_batch(m, n, nvec):
    """Fewer vectors than the handle holds: the same values as in a handle made for them."""
    cb = mi.make_crossbar(m, n, 4)
    r = np.random.default_rng(8).uniform(-1.0, 1.0, (nvec, 2 * m * n))
    zs = []
    for mb in (nvec, 3):
        pr = mca.default_params(m, n, precision=mca.PREC_FP64, max_batch=mb)
        with mca.Solver(pr, cb.gmap) as s:
            rd = torch.as_tensor(r, device=DEV)
            zs.append(torch.empty_like(rd))
            s.precond_apply(np.full(nvec, 2.1e-5), rd, zs[-1])
    assert torch.equal(zs[0], zs[1])


@pytest.mark.parametrize("K,d,H,W", [(5, 1, 3, 70), (11, 1, 13, 130), (11, 2, 5, 40),
                                     (11, 8, 40, 260), (11, 32, 70, 150), (7, 3, 9, 16),
                                     (13, 1, 20, 65), (15, 1, 18, 64), (9, 43, 50, 100)])
def test_convolution_forms(K, d, H, W):
    """The convolutions' and the weight gradient's row forms and the forms they fall back to
    (kernels of 15, dilations whose four taps do not fit): odd rows, rows without a partner, tiles
    cut by the image, taps beyond the kernel row.  FP32 accumulation of exact BF16 products:
    1e-5 of the summed term magnitudes (forward, backward data, weights), BF16 outputs within
    2^-8 of the value besides."""
    lib = mca.load()
    N, C = 2, 32
    g = torch.Generator(device=DEV).manual_seed(K * H + d)

    def rnd(*shape):
        return torch.randn(*shape, generator=g, device=DEV).to(torch.bfloat16)

    x, gz = rnd(N, H, W, C), rnd(N, H, W, C)
    w = (rnd(C, C, K, K).float() / (C * K * K) ** 0.5).to(torch.bfloat16).float()
    bias = torch.randn(C, generator=g, device=DEV)
    wf = torch.empty(K * K, C, C, dtype=torch.int16, device=DEV)
    wb = torch.empty_like(wf)
    out, gx = torch.empty_like(x), torch.empty_like(x)
    gw, gb = torch.empty_like(w), torch.empty_like(bias)
    scratch = torch.empty(int(lib.mca_cnn_wgrad_scratch(N, H, W, K)), device=DEV)
    p = [t.data_ptr() for t in (x, gz, wf, wb, bias, out, gx, gw, gb, scratch)]
    assert lib.mca_cnn_prep_weights(w.data_ptr(), C, C, K, C, p[2], p[3], None) == 0
    assert lib.mca_cnn_conv(p[0], N, H, W, p[2], K, d, C, C, p[4], 1, 0, None, p[5], None, None) == 0
    assert lib.mca_cnn_conv(p[1], N, H, W, p[3], K, d, C, C, None, 1, 1, p[0], p[6], None, None) == 0
    assert lib.mca_cnn_conv_wgrad(p[0], p[1], N, H, W, K, d, C, C, p[9], p[7], p[8], None) == 0
    assert lib.mca_cnn_check(None) == 0

    def ref(xv, wv, gzv):
        xv = xv.double().permute(0, 3, 1, 2).cpu().requires_grad_(True)
        wv = wv.double().cpu().requires_grad_(True)
        y = torch.nn.functional.conv2d(xv, wv, padding=d * (K // 2), dilation=d)
        y.backward(gzv.double().permute(0, 3, 1, 2).cpu())
        return [t.detach() for t in (y, xv.grad, wv.grad)]

    y, dx, dw = ref(x, w, gz)
    ys, dxs, dws = ref(x.abs(), w.abs(), gz.abs())
    z = y + bias.double().cpu()[None, :, None, None]
    zs = ys + bias.double().cpu().abs()[None, :, None, None]
    z = torch.where(z > 0, z, 0.1 * z)
    got = out.double().permute(0, 3, 1, 2).cpu()
    assert bool(((got - z).abs() <= 2.0 ** -8 * z.abs() + 1e-5 * zs).all())
    xc = x.double().permute(0, 3, 1, 2).cpu()
    dx = torch.where(xc > 0, dx, 0.1 * dx)
    got = gx.double().permute(0, 3, 1, 2).cpu()
    assert bool(((got - dx).abs() <= 2.0 ** -8 * dx.abs() + 1e-5 * dxs).all())
    assert bool(((gw.double().cpu() - dw).abs() <= 1e-5 * dws).all())
    gs = gz.double().sum(dim=(0, 1, 2)).cpu()
    assert bool(((gb.double().cpu() - gs).abs() <= 1e-5 * gz.double().abs().sum(dim=(0, 1, 2)).cpu()).all())
