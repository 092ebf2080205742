"""Host model of the FP64 transforms on BF16 slices (csrc/k_precond64.cu) and of their error.

A row x of an operand is held as x = 2^(e - 5) sum_s a_s 128^-s, s = 0 .. 7, |a_s| <= 64, 2^e <=
max |x| < 2^(e + 1), each entry rounded to a multiple of 2^(e - 54).  A product of two entries is
then 2^(ea + eb - 10) sum_st a_s b_t 128^-(s + t), and the terms of weight s + t >= 8 are left out.
In units of 2^(ea + eb):
* the seven terms of weight 8 are at most 2^-54 each, those behind them less by 128 and more, and
  the two roundings at most 2^-55 x 2 each: DROPPED = 9.1 x 2^-54 in all;
* over data whose digits are evenly spread in [-64, 63] (rms 37), the seven terms have an rms of
  sqrt(7) (37 / 64)^2 x 2^-54 = 0.88 x 2^-54, and with the roundings' 2 x 2^-54 / sqrt(12) =
  0.58 x 2^-54 of the mean square entries below 1.1 x 2^-54: RMS_DROPPED.
"""
import numpy as np

DROPPED = 9.1 * 2.0 ** -54
RMS_DROPPED = 1.1 * 2.0 ** -54
KMAX = 512                 # K of one range, joined to FP64


def exponents(x):
    return np.frexp(np.abs(x).max(axis=1))[1] - 1


def digits(x):
    """(8, rows, K) digits of a matrix's rows, as integers."""
    e = exponents(x)
    f = np.floor(np.ldexp(np.abs(x).astype(np.longdouble), (54 - e)[:, None]) + 0.5).astype(np.int64)
    out = np.empty((8,) + x.shape, np.int64)
    for s in range(7, 0, -1):
        out[s] = ((f + 64) & 127) - 64
        f = (f - out[s]) >> 7
    out[0] = f
    return out * np.sign(x).astype(np.int64)


def transform(a, b, weights=8):
    """out[c][r] = sum_k a[r][k] b[c][k] as the kernel forms it, from the first `weights` weights
    (products of digits and their sums over a range are exact in FP64 matrix products)."""
    da, db = digits(a).astype(float), digits(b).astype(float)
    scale = exponents(a)[None, :] + exponents(b)[:, None] - 10
    out = np.zeros((b.shape[0], a.shape[0]))
    for k in range(0, a.shape[1], KMAX):
        w = slice(k, k + KMAX)
        s = np.zeros(out.shape, np.longdouble)
        for d in range(weights):
            part = sum(da[i][:, w] @ db[d - i][:, w].T for i in range(d + 1)).T
            s += np.ldexp(part.astype(np.longdouble), -7 * d)
        out = out + np.ldexp(s.astype(float), scale)
    return out


def modes(h, mu, nu, a):
    """The per-mode 2 x 2 inverse of the two layers' coefficients h[layer][i'][k']."""
    n = nu[:, None]
    det = n * mu + a * (n + mu)
    return (((n + a) * h[0] + a * h[1]) / det, (a * h[0] + (mu + a) * h[1]) / det)


def apply(r, qr, qc, mu, nu, a, gemm):
    """z = P^-1 r, r[layer][i][j], by four transforms of each layer."""
    h = [gemm(gemm(x, qr.T), qc.T) for x in r]
    return np.stack([gemm(gemm(y, qr), qc) for y in modes(h, mu, nu, a)])


def exact(r, qr, qc, mu, nu, a):
    ld = [np.asarray(x).astype(np.longdouble) for x in (r, qr, qc, mu, nu, a)]
    return apply(*ld, lambda x, q: q @ x.T)


def expected_error(r, qr, qc, mu, nu, a):
    """Root of the expected square norm of apply()'s error on evenly spread digits: variances of
    the entries carried through the four transforms, each of which adds what its slices leave out
    and the rounding of its sums (2^-53 of the result per addition, taken whole)."""
    def step(x, var, q):
        out = q @ x.T
        k = x.shape[1]
        own = RMS_DROPPED ** 2 * k * 4.0 ** (exponents(x)[None, :] + exponents(q)[:, None])
        rounded = (2 * -(-k // KMAX) - 1) * (2.0 ** -53 * out) ** 2
        return out, (q ** 2) @ var.T + own + rounded

    h, hv = zip(*(step(*step(x, np.zeros(x.shape), qr.T), qc.T) for x in r))
    n = nu[:, None]
    det = n * mu + a * (n + mu)
    total = 0.0
    for y, c in zip(modes(h, mu, nu, a), ((n + a, a), (a, mu + a))):
        var = sum((ci / det) ** 2 * v for ci, v in zip(c, hv))
        size = sum(np.abs(ci * x) for ci, x in zip(c, h)) / np.abs(det)
        var = var + (4 * 2.0 ** -53 * size) ** 2
        total += step(*step(y, var, qr), qc)[1].sum()
    return np.sqrt(total)
