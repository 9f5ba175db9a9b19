"""The refinement's tensor-core form at its tightest tolerance (1e-8, the default).

There P q follows a recurrence and is not projected anew.  Both forms solve
(A - s_j) t_j = b_j to |r_j| <= 1e-8 |b_j|, and the Ritz pairs' new residuals are r_j plus
terms of second order in t that both share to 1e-8: after one round the residuals
differ by at most 2e-8 |b| and the second-order terms' share, 1e-7 |b| in all with
|b| the norm of all columns (Rayleigh-Ritz mixes them), above a floor of 1e-12 of the
largest |lambda|.  Iteration counts may differ by one: a column may meet the threshold
on either side of it.  The widths with a loose state behind them end at gaps of the
spectrum (35 columns), as the projected operator is definite only there.
"""
import numpy as np
import pytest

from gpu_common import make

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mg32", [0, 1])
@pytest.mark.parametrize("m,N,tc", [(9, 5, 2), (12, 32, 2), (14, 64, 2), (24, 20, 2), (32, 35, 1)])
def test_tight_refinement_matches_simt_projections(m, N, tc, mg32):
    out = []
    for t in (tc, 0):
        s, _, _ = make(m, N, fp64_tc=t, mg_fp32=mg32, tau=0.4, cg_rtol=1e-10)
        s.solve(2e-4, 20000)
        before = s.eigenpairs()
        r, its = s.refine(rounds=1, rtol=1e-8, maxit=500)
        out.append((before, np.asarray(r), its, s.eigenpairs()))
    (b0, ra, ia, ea), (_, rb, ib, eb) = out
    assert abs(ia - ib) <= 1
    top = np.abs(b0["lam_rr"]).max()
    assert np.all(np.abs(ra - rb) <= 1e-7 * np.linalg.norm(b0["residuals"]) + 1e-12 * top)
    # eigenvalues to the square of the residuals that remain, or rounding
    assert np.all(np.abs(ea["lam_rr"] - eb["lam_rr"]) <= 1e-11 * top)


@pytest.mark.parametrize("tc", [2, 1])
def test_default_refinement_reaches_rounding(tc):
    """Two rounds at the default tolerance from residuals of 2e-4: the second round starts
    below 1e-6, so what remains is rounding, far below 1e-9."""
    s, _, _ = make(20, 35, fp64_tc=tc, mg_fp32=1, tau=0.4, cg_rtol=1e-10)
    s.solve(2e-4, 20000)
    r, _ = s.refine()
    assert np.max(r) < 1e-9
