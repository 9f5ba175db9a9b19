"""Digit-sliced FP64 Grams at the edges of their tiles and slices: rows of 32
points, flushes of 128, 64 output columns, 128 rows.

Bars: the Gram of a step as in the kernel tests (2^-44 |x_i| |x_j| n).  A
refinement round whose projections run on tensor cores (fp64_tc = 2) against one
in SIMT FP64: the corrections t are solved to 1e-2 and differ by the rounding of
the projections, below 1e-10 |t| against the residual that remains, 1e-2 |t|:
residuals to 1e-6, iterations equal.
"""
import numpy as np
import pytest

from gpu_common import host, make

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,N", [(3, 1), (5, 16), (7, 32), (6, 33), (8, 64), (11, 63), (26, 48), (33, 17)])
def test_step_gram_at_tile_edges(m, N):
    grams = []
    for tc in (2, 0):
        s, _, _ = make(m, N, fp64_tc=tc, cg_rtol=1e-12)
        grams.append(host(s.step_trace()["gram"]))
    g, ref = grams
    assert np.array_equal(g, g.T)
    scale = np.sqrt(np.abs(np.diag(ref)))
    assert np.all(np.abs(g - ref) <= 2.0 ** -44 * np.outer(scale, scale) * m ** 3 + 1e-14 * np.abs(ref).max())


@pytest.mark.parametrize("mg32", [0, 1])
@pytest.mark.parametrize("m,N", [(9, 5), (12, 32), (17, 33), (14, 64)])
def test_refinement_round_matches_simt_projections(m, N, mg32):
    out = []
    for tc in (2, 0):
        s, _, _ = make(m, N, fp64_tc=tc, mg_fp32=mg32, tau=0.4, cg_rtol=1e-10)
        s.solve(2e-4, 20000)   # the refinement needs nearly converged pairs
        out.append(s.refine(rounds=1, rtol=1e-2, maxit=500))
    (ra, ia), (rb, ib) = out
    assert ia == ib
    np.testing.assert_allclose(ra, rb, rtol=1e-6, atol=1e-13)
