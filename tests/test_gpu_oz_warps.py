"""Digit-sliced Grams whose warps do not act as one: column counts where lanes of a
converting warp have no values and whole warps no unit, over several flushes, so
that the issuing thread's warp and the idle lanes meet again before each read-out
of the accumulators.  The bar is that of the Gram at tile edges (2^-44 |x_i| |x_j|
n); a repeated Gram is the same bit for bit, since its sums are exact.
"""
import numpy as np
import pytest

from gpu_common import host, make

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,N", [(24, 1), (24, 9), (25, 21), (24, 37), (40, 5), (32, 61)])
def test_gram_of_ragged_warps(m, N):
    s, _, _ = make(m, N, fp64_tc=2, cg_rtol=1e-12)
    g = host(s.step_trace()["gram"])
    r, _, _ = make(m, N, fp64_tc=0, cg_rtol=1e-12)
    ref = host(r.step_trace()["gram"])
    assert np.array_equal(g, g.T)
    scale = np.sqrt(np.abs(np.diag(ref)))
    assert np.all(np.abs(g - ref) <= 2.0 ** -44 * np.outer(scale, scale) * m ** 3 + 1e-14 * np.abs(ref).max())
    for _ in range(3):
        t, _, _ = make(m, N, fp64_tc=2, cg_rtol=1e-12)
        assert np.array_equal(host(t.step_trace()["gram"]), g)
