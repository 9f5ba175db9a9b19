"""FP64 dense kernels at the edges of their tile sizes, against plain FP64 numpy.

A sum of n rounded products in any order is within (n + 2) 2^-53 sum |a||b| of
the exact value, numpy's as well: tolerance 2 (n + 2) 2^-53 sum |a||b| w.
"""
import numpy as np
import pytest

from gpu_common import dev, host
from paper_2605_25149_gb300 import hq, inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Na,Nb", [(1, 1), (15, 15), (16, 17), (32, 32), (33, 31), (48, 48), (49, 64),
                                   (64, 1), (65, 65), (96, 130), (130, 130)])
@pytest.mark.parametrize("m", [3, 11])
def test_gram_tile_edges(m, Na, Nb):
    n, N = m ** 3, 65
    s = hq.Solver(m, min(N, n), fp64_tc=0)
    if max(Na, Nb) > 2 * s.N:
        pytest.skip("wider than twice the context's columns")
    s.set_potential(inputs.harmonic(m))
    rng = np.random.default_rng(Na + 100 * Nb)
    A, B = rng.standard_normal((n, Na)), rng.standard_normal((n, Nb))
    a, b = dev(A), dev(B)
    tol = 2 * (n + 2) * 2.0 ** -53 * 0.7
    assert np.all(np.abs(host(s.gram(a, b, 0.7)) - 0.7 * A.T @ B) <= tol * (np.abs(A).T @ np.abs(B)))
    G = host(s.gram(a, a, 0.7))   # the symmetric form
    assert np.all(np.abs(G - 0.7 * A.T @ A) <= tol * (np.abs(A).T @ np.abs(A)))
    assert np.array_equal(G, G.T)
