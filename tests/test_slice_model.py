"""The error of the FP64 transforms' slices, on the host model: the bound that the kernel states,
and that the bar of its GPU test would show a lost weight."""
from fractions import Fraction

import numpy as np
import pytest

import slice_model as S


def _chain(n, first, last):
    d = np.full(n, 2.0)
    d[0], d[-1] = first + 1.0, 1.0 + last
    t = np.diag(d) - np.eye(n, k=1) - np.eye(n, k=-1)
    return np.linalg.eigh(t)


def test_what_a_product_leaves_out():
    """In exact arithmetic: DROPPED holds for the digits {33, -64 x 7} that drop the most, for
    entries far below their rows' maxima and for random ones, and is no more than a third too
    large."""
    worst = np.ldexp(float(sum(d * 128 ** (7 - s) for s, d in enumerate([33] + [-64] * 7))), -54)
    rng = np.random.default_rng(0)
    pairs = [(worst, worst)] + [tuple(rng.uniform(1, 2, 2)) for _ in range(300)]
    pairs += [tuple(rng.uniform(1, 2, 2) * 2.0 ** -rng.integers(0, 60, 2)) for _ in range(300)]
    most = 0
    for x, y in pairs:
        # the row's maximum beside the entry, 1 for the entries that are not it
        a, b = np.array([[x, 1.0]]), np.array([[y, 1.0]])
        scale = Fraction(2) ** int(S.exponents(a)[0] + S.exponents(b)[0])
        da, db = S.digits(a)[:, 0, 0], S.digits(b)[:, 0, 0]
        kept = sum(Fraction(int(da[s]) * int(db[t]), 128 ** (s + t))
                   for s in range(8) for t in range(8 - s)) * scale / 2 ** 10
        most = max(most, abs(kept - Fraction(x) * Fraction(y)) / scale)
    assert Fraction(S.DROPPED) * 2 / 3 <= most <= Fraction(S.DROPPED)


@pytest.mark.parametrize("m,n", [(33, 70), (9, 600), (65, 129)])
@pytest.mark.parametrize("a", [2e-5, 0.2])
def test_lost_weights_show(m, n, a):
    """The modelled apply lies within 3 expected errors, and without weight 7 far outside."""
    mu, qr = _chain(n, 0.1, 1e-3)
    nu, qc = _chain(m, 1e-3, 0.1)
    r = np.random.default_rng(m).uniform(-1, 1, (2, m, n))
    args = (r, qr, qc, mu, nu, a)
    ref, bar = S.exact(*args), 3 * S.expected_error(*args)
    err = [float(np.sqrt(((S.apply(*args, lambda x, q: S.transform(x, q, w)) - ref) ** 2).sum()))
           for w in (8, 7)]
    assert err[0] <= bar and err[1] >= 4 * bar
