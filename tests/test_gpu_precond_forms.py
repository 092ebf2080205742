"""What the sliced FP64 transforms and the chunked line solves of the paper's M_hat owe to the
plain FP64 forms they replaced: the same infinities and NaN, and their accuracy."""
import numpy as np
import pytest

import mca_inputs as mi
import slice_model as S

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2109_07929_gb300 as mca  # noqa: E402

DEV = "cuda:0"


def _reach(t):
    """0 finite, 1 infinity, 2 minus infinity, 3 NaN."""
    return np.isposinf(t) * 1 + np.isneginf(t) * 2 + np.isnan(t) * 3


def _chain(rows, q):
    """out[c][r] = sum_k rows[r][k] q[c][k], one product after the other."""
    out = np.zeros((q.shape[0], rows.shape[0]))
    for k in range(q.shape[1]):
        out = out + np.outer(q[:, k], rows[:, k])
    return out


@pytest.mark.parametrize("value", [float("inf"), float("-inf"), float("nan")])
@pytest.mark.parametrize("m,n", [(1, 1), (1, 7), (7, 1), (5, 40), (33, 70), (2, 600)])
def test_fp64_preconditioner_reach_of_infinities(m, n, value):
    """An infinite or NaN entry of r gives the infinities and NaN of the plain FP64 sums (with the
    handle's own eigenvectors); the other vector of the batch is not touched."""
    cb = mi.make_crossbar(m, n, 4)
    rng = np.random.default_rng(1)
    a = np.array([2e-5, 0.2])
    with mca.Solver(mca.default_params(m, n, precision=mca.PREC_FP64, max_batch=2),
                    cb.gmap) as s:
        mu, qr, nu, qc = s.eigenpairs()
        for pos in (0, m * n - 1, m * n + m * n // 2):
            r = rng.standard_normal((2, 2 * m * n))
            rd = torch.as_tensor(r, device=DEV)
            clean, z = torch.empty_like(rd), torch.empty_like(rd)
            s.precond_apply(a, rd, clean)
            rd[0, pos] = value
            s.precond_apply(a, rd, z)
            assert torch.equal(z[1], clean[1])
            with np.errstate(invalid="ignore"):
                h = [_chain(_chain(x.reshape(m, n), qr.T), qc.T)
                     for x in rd[0].cpu().numpy().reshape(2, m * n)]
                det = nu[:, None] * mu + a[0] * (nu[:, None] + mu)
                t = ((nu[:, None] + a[0]) * h[0] + a[0] * h[1]) / det
                b = (a[0] * h[0] + (mu + a[0]) * h[1]) / det
                ref = [_chain(_chain(y, qr), qc) for y in (t, b)]
            assert np.array_equal(_reach(z[0].cpu().numpy()),
                                  _reach(np.concatenate([x.ravel() for x in ref])))


@pytest.mark.parametrize("value", [float("inf"), float("-inf"), float("nan")])
@pytest.mark.parametrize("m,n", [(1, 1), (1, 7), (7, 1), (5, 40), (33, 70), (300, 33)])
def test_mhat_reach_of_infinities(m, n, value):
    """z_b = G_2^-1 r_b along columns and z_t = (r_t + a z_b) G_1^-1 along rows, with inverses
    whose entries are all positive: an entry of r_t reaches its row of z_t as it is, one of r_b
    its column of z_b and with it every entry of z_t."""
    cb = mi.make_crossbar(m, n, 4)
    kind = 3 if value != value else (1 if value > 0 else 2)
    r = np.random.default_rng(1).standard_normal((1, 2, m, n))
    with mca.Solver(mca.default_params(m, n, precision=mca.PREC_MHAT, max_batch=1),
                    cb.gmap) as s:
        for layer in (0, 1):
            for i, j in {(0, 0), (m // 2, n // 2), (m - 1, n - 1)}:
                rd = torch.as_tensor(r, device=DEV)
                rd[0, layer, i, j] = value
                z = torch.empty_like(rd)
                s.precond_apply(np.array([2e-4]), rd.view(1, -1), z.view(1, -1))
                want = np.zeros((2, m, n), int)
                if layer == 0:
                    want[0, i] = kind
                else:
                    want[0] = kind
                    want[1, :, j] = kind
                assert np.array_equal(_reach(z[0].cpu().numpy()), want)


@pytest.mark.parametrize("m,n", [(33, 70), (64, 128), (129, 65), (9, 600), (600, 9)])
def test_fp64_preconditioner_loses_no_weight(m, n):
    """The apply's error within 3 expected errors of its slices, against extended precision with
    the handle's own eigenpairs (on the host model a lost weight 7 exceeds that bar 19 times)."""
    cb = mi.make_crossbar(m, n, 4)
    r = np.random.default_rng(m).uniform(-1, 1, (2, 2, m, n))
    a = np.array([2e-5, 0.2])
    with mca.Solver(mca.default_params(m, n, precision=mca.PREC_FP64, max_batch=2),
                    cb.gmap) as s:
        mu, qr, nu, qc = s.eigenpairs()
        rd = torch.as_tensor(r.reshape(2, -1), device=DEV)
        z = torch.empty_like(rd)
        s.precond_apply(a, rd, z)
    z = z.cpu().numpy().reshape(r.shape)
    for v in range(2):
        ref = S.exact(r[v], qr, qc, mu, nu, a[v])
        err = float(np.sqrt(((z[v] - ref) ** 2).sum()))
        assert err <= 3 * S.expected_error(r[v], qr, qc, mu, nu, a[v])


def _line(n, g, first, last, a):
    """Diagonal of tridiag(-g, d + a, -g) over a line of n nodes between two terminations."""
    d = np.full(n, 2.0 * g)
    if n == 1:
        d[0] = first + last
    else:
        d[0], d[-1] = first + g, g + last
    return d + a


def _times(d, g, x, sign=-1.0):
    """The line operator along axis 0, in extended precision; sign = 1: its absolute values."""
    x = x.astype(np.longdouble)
    y = d.astype(np.longdouble)[:, None] * x
    y[1:] += sign * g * x[:-1]
    y[:-1] += sign * g * x[1:]
    return y


def _solve_line(d, g, w):
    """Thomas sweeps along axis 0 (all terms of one sign for w >= 0)."""
    piv, y = d.copy(), w.copy()
    for j in range(1, len(d)):
        q = g / piv[j - 1]
        piv[j] -= q * g
        y[j] += q * y[j - 1]
    y[-1] /= piv[-1]
    for j in range(len(d) - 2, -1, -1):
        y[j] = (y[j] + g * y[j + 1]) / piv[j]
    return y


@pytest.mark.parametrize("m,n", [(2, 2), (8, 9), (9, 8), (1, 31), (32, 33), (65, 2), (100, 1025),
                                 (2049, 3), (1057, 40)])
def test_mhat_solves_are_backward_stable(m, n):
    """G_2 z_b = r_b and z_t G_1 = r_t + a z_b to rounding, for a / g on both sides of the closed
    form's two branches and at both ends.  A chunk of L nodes forms its carries' factors as
    products of up to L terms, in both sweeps, so the residual is within (8 + 2 L) 2^-53 of
    |G| |z|, with |z| the solution for |r| (an M-matrix: all its terms are positive)."""
    cb = mi.make_crossbar(m, n, 4, g_wire_bot=0.5)
    p = cb.params
    a = np.array([1e-9, 2.1e-5, 0.2, 3.0, 1e6])
    r = np.random.default_rng(7).standard_normal((len(a), 2, m, n))
    prm = mca.default_params(m, n, g_wire_bot=0.5, precision=mca.PREC_MHAT, max_batch=len(a))
    with mca.Solver(prm, cb.gmap) as s:
        rd = torch.as_tensor(r.reshape(len(a), -1), device=DEV)
        z = torch.empty_like(rd)
        s.precond_apply(a, rd, z)
    z = z.cpu().numpy().reshape(r.shape)
    for v, av in enumerate(a):
        for g, first, last, x, rhs, extra in (
                (p.g_wire_bot, p.g_term_bot_top, p.g_sense, z[v, 1], r[v, 1], 0.0),
                (p.g_wire_top, p.g_src, p.g_term_top_right, z[v, 0].T, r[v, 0].T, z[v, 1].T)):
            d = _line(x.shape[0], g, first, last, av)
            w = rhs + np.longdouble(av) * extra
            size = np.abs(rhs) + av * np.abs(extra)
            bound = (8 + 2 * -(-x.shape[0] // 32)) * 2.0 ** -53 * _times(
                d, g, _solve_line(d, g, size), 1.0)
            assert bool((np.abs(_times(d, g, x) - w) <= bound).all()), (av, g)
