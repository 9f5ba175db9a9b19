"""The FP64 operator's integer neighbour sum at the edges of its exponent range.

y = D x - c S with S the six-neighbour sum.  S carries at most six truncations
of 2^-59 2^E (2^E the binade of the largest neighbour) and one rounding, y one
rounding of c S, one of the product or the sum, and D one of its own two
additions: |y - exact| <= 2^-53 (2 |c S| + 2 |y| + 4 |D x|) + 2^-56 |c| max|nbr|.
"""
from fractions import Fraction

import numpy as np
import pytest

from gpu_common import dev, host
from paper_2605_25149_gb300 import hq, inputs

pytestmark = pytest.mark.gpu


def neighbours(X, m):
    """The six neighbour values of every point (zero outside), 6 x n x N."""
    P = np.zeros((m + 2, m + 2, m + 2, X.shape[1]))
    P[1:-1, 1:-1, 1:-1] = X.reshape(m, m, m, -1)
    s = [slice(0, -2), slice(2, None)]
    c = slice(1, -1)
    out = [P[c, c, a] for a in s] + [P[c, a, c] for a in s] + [P[a, c, c] for a in s]
    return [o.reshape(m ** 3, -1) for o in out]


def block(kind, m, N):
    rng = np.random.default_rng(17)
    x = rng.standard_normal((m ** 3, N))
    if kind == "wide":          # exponents apart by up to 80 binades, some zeros
        x = np.ldexp(x, rng.integers(-40, 41, x.shape)) * (rng.random(x.shape) > 0.1)
    elif kind == "cancel":      # neighbours that nearly cancel, both signs of a power of two
        x = np.where(rng.random(x.shape) > 0.5, 1.0, -1.0) * (1.0 + np.ldexp(rng.integers(0, 3, x.shape).astype(float), -52))
    elif kind == "small":       # across the lower end of the integer sum's range, subnormals among them
        x = np.ldexp(x, rng.integers(-1060, -930, x.shape))
    elif kind == "large":       # across its upper end, sums that stay finite
        x = np.ldexp(x, rng.integers(1000, 1013, x.shape))
    return x


@pytest.mark.parametrize("zmarch", ["0", "1"])
@pytest.mark.parametrize("m,N", [(5, 1), (7, 3), (9, 8)])
@pytest.mark.parametrize("kind", ["plain", "wide", "cancel", "small", "large"])
def test_operator_error_bound(kind, m, N, zmarch, monkeypatch):
    monkeypatch.setenv("HQ_ZMARCH", zmarch)
    V = inputs.wells(m, 2)
    s = hq.Solver(m, N)
    s.set_potential(V)
    X = block(kind, m, N)
    y = host(s.apply_operator(dev(X)))
    h = inputs.grid_h(m)
    c, sigma = 0.5 / (h * h), s.info()["sigma"]
    nb = neighbours(X, m)
    tiny = Fraction(2) ** -1070   # results in the subnormal range are rounded to multiples of 2^-1074
    for p in range(0, m ** 3, 3):
        D = 6 * Fraction(c) + Fraction(V[p]) + Fraction(sigma)
        for q in range(N):
            a = [Fraction(float(v[p, q])) for v in nb]
            cS, Dx = Fraction(c) * sum(a), D * Fraction(X[p, q])
            ref = Dx - cS
            tol = Fraction(2) ** -53 * (2 * abs(cS) + 2 * abs(ref) + 4 * abs(Dx)) + \
                Fraction(2) ** -56 * Fraction(c) * max(abs(v) for v in a) + tiny
            assert abs(Fraction(float(y[p, q])) - ref) <= tol


def test_nonfinite_values_spread_to_their_neighbours_only():
    m, N = 6, 2
    V = inputs.harmonic(m)
    s = hq.Solver(m, N)
    s.set_potential(V)
    X = np.random.default_rng(3).standard_normal((m ** 3, N))
    X[40, 0], X[100, 1], X[101, 1] = np.nan, np.inf, -np.inf
    y = host(s.apply_operator(dev(X)))
    with np.errstate(invalid="ignore"):
        h = inputs.grid_h(m)
        ref = (3.0 / h ** 2 + V)[:, None] * X - 0.5 / h ** 2 * sum(neighbours(X, m))
    assert np.array_equal(np.isnan(y), np.isnan(ref)) and np.array_equal(np.isinf(y), np.isinf(ref))
    fine = np.isfinite(ref)
    assert np.array_equal(y[~fine & ~np.isnan(ref)], ref[~fine & ~np.isnan(ref)])
    np.testing.assert_allclose(y[fine], ref[fine], rtol=1e-12, atol=1e-11)
