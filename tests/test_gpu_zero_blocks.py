"""The FP64 operator on zeros: the first residual of every solve from zero.

Six zero neighbours once took the scaling of the rare exponents, at three and a half
times the operator's usual time.  The bar of 1.5 on the ratio of the two medians
(same kernel, same traffic; zeros do less) leaves room for the timer's 2 us steps.
"""
import numpy as np
import pytest

from gpu_common import host, make, torch_mod

pytestmark = pytest.mark.gpu


def median_us(f, torch):
    for _ in range(3):
        f()
    t = []
    for _ in range(9):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        for _ in range(4):
            f()
        b.record()
        torch.cuda.synchronize()
        t.append(a.elapsed_time(b) * 250.0)
    return float(np.median(t))


@pytest.mark.parametrize("m,N", [(48, 64), (47, 33)])
def test_zero_block_costs_no_more_than_any_other(m, N):
    torch = torch_mod()
    s, _, _ = make(m, N)
    x = torch.randn((m ** 3, N), device="cuda", dtype=torch.float64)
    z = torch.zeros_like(x)
    assert not host(s.apply_operator(z)).any()
    usual, zeros = (median_us(lambda b=b: s.apply_operator(b), torch) for b in (x, z))
    assert zeros <= 1.5 * usual, (zeros, usual)


def test_zeros_beside_values():
    """Half a block of zeros: exact zeros inside, the operator's values at the seam."""
    m, N = 9, 2
    s, V, _ = make(m, N)
    x = np.random.default_rng(5).standard_normal((m ** 3, N))
    x[: m * m * 4] = 0.0
    x[m * m * 2 + 7] = -0.0
    torch = torch_mod()
    y = host(s.apply_operator(torch.from_numpy(x).cuda()))
    assert not y[: m * m * 3].any()
    h = (s.cfg.hi - s.cfg.lo) / (m + 1)
    c = 0.5 / h ** 2
    P = np.zeros((m + 2, m + 2, m + 2, N))
    P[1:-1, 1:-1, 1:-1] = x.reshape(m, m, m, N)
    i = slice(1, -1)
    nb = (P[:-2, i, i] + P[2:, i, i] + P[i, :-2, i] + P[i, 2:, i] + P[i, i, :-2] + P[i, i, 2:]).reshape(-1, N)
    ref = (6 * c + V + s.info()["sigma"])[:, None] * x - c * nb
    np.testing.assert_allclose(y, ref, rtol=1e-13, atol=1e-12)
