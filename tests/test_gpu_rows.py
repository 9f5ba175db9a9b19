"""V-cycles through the whole-row kernels at the edges of their launch shapes.

One x-row per CTA: 16 column vectors up to 32 points per side, 8 up to 64, 4 up
to 128, two points per thread above.  The bars are those of the V-cycle tests
of the separate kernels (1e-5 of the largest value in FP32, 1e-12 in FP64).
"""
import numpy as np
import pytest

from gpu_common import dev, host, make, oracle_mg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,bar", [("mixed", 1e-5), ("fp64", 1e-12)])
@pytest.mark.parametrize("m,N,nu", [(5, 1, 2), (17, 4, 2), (32, 64, 3), (33, 68, 2), (48, 5, 3), (64, 36, 2),
                                    (65, 8, 2), (129, 16, 2)])
def test_vcycle_at_row_shape_edges(m, N, nu, prec, bar):
    s, V, _ = make(m, N, precision=prec, mg_nu1=nu, mg_nu2=nu)
    r = np.random.default_rng(m + N).standard_normal((m ** 3, N)).astype(np.float32 if prec == "mixed" else np.float64)
    z = host(s.mg_vcycle(dev(r)))
    ref = oracle_mg(s, V).vcycle(r.astype(np.float64))
    assert np.abs(z - ref).max() <= bar * np.abs(ref).max()


@pytest.mark.parametrize("m,N", [(5, 2), (64, 12), (130, 4)])
def test_prolongation_in_place_and_zero_correction(m, N):
    """e_out may be e_in; P 0 = 0 leaves the iterate untouched, bit for bit."""
    s, _, _ = make(m, N)
    mc = s.levels()[1]
    e = np.random.default_rng(1).standard_normal((m ** 3, N))
    out = host(s.mg_prolong(0, dev(np.zeros((mc ** 3, N))), dev(e)))
    assert np.array_equal(out, e)
