"""3xTF32 block products at the edges of their slice walk: one slice in all (fewer
than are read out late or loaded ahead), one slice per work item, several work
items per CTA, ragged K with and without vector loads, every tile width.  The bar
is that of the kernel tests (2e-6 of the largest value)."""
import numpy as np
import pytest

from gpu_common import dev, host, make

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m", [3, 8, 30])
@pytest.mark.parametrize("N,k1,k2", [(4, 4, 0), (16, 16, 16), (27, 27, 6), (48, 48, 48), (20, 5, 3), (64, 64, 4),
                                     (130, 130, 1)])
def test_mixed_block_gemm_slice_walk(m, N, k1, k2):
    n = m ** 3
    if N > n:
        pytest.skip("more columns than points")
    s, _, _ = make(m, N, precision="mixed", cg_rtol=1e-6)
    rng = np.random.default_rng(m * 1000 + N + k2)
    A1, M1 = rng.standard_normal((n, k1)).astype(np.float32), rng.standard_normal((k1, N))
    A2 = rng.standard_normal((n, k2)).astype(np.float32) if k2 else None
    M2 = rng.standard_normal((k2, N)) if k2 else None
    out = host(s.block_gemm(dev(A1), dev(M1), None if A2 is None else dev(A2), None if M2 is None else dev(M2)))
    ref = A1.astype(np.float64) @ M1
    if k2:
        ref += A2.astype(np.float64) @ M2
    assert np.abs(out - ref).max() <= 2e-6 * np.abs(ref).max()
