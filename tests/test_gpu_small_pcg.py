"""The one-launch PCG of small FP64 problems with the FP32 preconditioner.

Its recurrence, roundings and summation orders are those of the separate
launches (HQ_FUSED_COARSE=0), so iterates and iteration counts are equal bit for
bit: at level edges (odd sides, the largest that fits, the first that does not),
one column and many, a zero column, a start at the solution and a cap on the
iterations.
"""
import numpy as np
import pytest

from gpu_common import dev, host, make

pytestmark = pytest.mark.gpu


def solve(monkeypatch, fused, m, N, B, X0, rtol, maxit):
    if fused:
        monkeypatch.delenv("HQ_FUSED_COARSE", raising=False)
    else:
        monkeypatch.setenv("HQ_FUSED_COARSE", "0")
    s, _, _ = make(m, N, mg_fp32=1)
    X, its = s.block_pcg(dev(B), X0=dev(X0), rtol=rtol, maxit=maxit)
    return host(X), its


@pytest.mark.parametrize("m,N", [(5, 1), (8, 16), (9, 7), (16, 8), (17, 5), (17, 64), (18, 4)])
@pytest.mark.parametrize("rtol,maxit", [(1e-9, 100), (0.0, 3), (0.0, 0)])
def test_one_launch_pcg_matches_separate_kernels(monkeypatch, m, N, rtol, maxit):
    rng = np.random.default_rng(m * 100 + N)
    B = rng.standard_normal((m ** 3, N))
    B[:, N // 2] *= 1e-3
    X0 = rng.standard_normal((m ** 3, N))
    if N > 1:
        B[:, 0] = X0[:, 0] = 0.0   # |r| = |b| = 0: never active
    a, ia = solve(monkeypatch, True, m, N, B, X0, rtol, maxit)
    b, ib = solve(monkeypatch, False, m, N, B, X0, rtol, maxit)
    np.testing.assert_array_equal(a, b)
    np.testing.assert_array_equal(ia, ib)
