"""The digit-sliced products' error bound at the digits that come closest to it.

A value of digits 65, -128, .., -128 (seven of base 256) is a double, and its square's
dropped digit pairs (i + j >= 9) all have one sign: 2^-51.4 of the square.  Bound per
term: 2^-51 |row max| |column max| for the dropped pairs, one rounding of the result and
of its scaling and accumulation over chunks, 2^-51 |result|; the digits of these
values are exact.  Random values round their last digit, 2^-55 of either maximum.  The
Gram reads its sums out every 128 points in 32 fraction bits, so its bar is that of the
other Gram tests (2^-44 |x_i| |x_j| n).
"""
import numpy as np
import pytest

from gpu_common import dev, host, make

pytestmark = pytest.mark.gpu

WORST = float(65 * 2 ** 55 - 128 * sum(2 ** (63 - 8 * i) for i in range(2, 8))) * 2.0 ** -64


def exact(A, M):
    """A @ M in extended precision (64-bit significands or more)."""
    return A.astype(np.longdouble) @ M.astype(np.longdouble)


def test_the_value_is_a_double_with_these_digits():
    f = int(WORST * 2.0 ** 64)
    assert f == 65 * 2 ** 55 - 128 * sum(2 ** (63 - 8 * i) for i in range(2, 8)) and 2 ** 61 <= f < 2 ** 62


@pytest.mark.parametrize("K", [1, 7, 64, 128])
@pytest.mark.parametrize("kind", ["worst", "random"])
def test_block_product(K, kind):
    m, N = 8, 64
    s, _, _ = make(m, N, fp64_tc=2)
    k1, k2 = min(K, N), max(0, K - N)
    rng = np.random.default_rng(K)
    if kind == "worst":
        A, M = np.full((m ** 3, K), WORST), np.full((K, N), WORST)
        M[:, 1::2] *= -2.0 ** 40
    else:
        A, M = rng.standard_normal((m ** 3, K)), rng.standard_normal((K, N))
    A1, A2 = np.ascontiguousarray(A[:, :k1]), np.ascontiguousarray(A[:, k1:])
    out = host(s.block_gemm(dev(A1), dev(M[:k1]), dev(A2) if k2 else None, dev(M[k1:]) if k2 else None))
    ref = exact(A, M)
    scale = K * np.abs(A).max(1)[:, None] * np.abs(M).max(0)[None, :]
    err = np.abs(out.astype(np.longdouble) - ref).astype(float)
    assert np.all(err <= (2.0 ** -51 + 2 * 2.0 ** -55) * scale + 2.0 ** -51 * np.abs(ref).astype(float))


def test_gram():
    """Columns of the value and of alternating signs: <U,U> of a step, h^3 applied after the sum."""
    m, N = 9, 2
    s, _, _ = make(m, N, fp64_tc=2)
    U = np.full((m ** 3, N), WORST)
    U[1::2, 1] *= -1.0
    s.set_state(U, 0)
    g = host(s.step_trace()["gram"])[:N, :N]
    h3 = ((s.cfg.hi - s.cfg.lo) / (m + 1)) ** 3
    ref = np.array([[m ** 3, 1], [1, m ** 3]]) * WORST ** 2 * h3
    assert np.all(np.abs(g - ref) <= 2.0 ** -44 * m ** 3 * WORST ** 2 * h3)
