"""Prolongation against its definition, out of place and onto its own iterate.

P interpolates linearly between the coarse nodes (zero on the boundary): with fine node
i at position (i + 1) (mc + 1) / (mf + 1) - 1 in coarse index units, weights 1 - t and t of
the nodes around it.  Three nested sums of two rounded products and one addition to the
iterate: 10 roundings of values below the largest of either operand.
"""
import numpy as np
import pytest

from gpu_common import dev, host, make, torch_mod

pytestmark = pytest.mark.gpu


def interpolation(mf, mc):
    P = np.zeros((mf, mc))
    for i in range(mf):
        num = (i + 1) * (mc + 1)
        c, t = num // (mf + 1) - 1, (num % (mf + 1)) / (mf + 1)
        if c >= 0:
            P[i, c] += 1 - t
        if t > 0 and c + 1 < mc:
            P[i, c + 1] += t
    return P


@pytest.mark.parametrize("prec,eps", [("fp64", 2.0 ** -53), ("mixed", 2.0 ** -24)])
@pytest.mark.parametrize("m,N", [(5, 2), (8, 1), (16, 64), (32, 3), (33, 68), (64, 12), (65, 5), (129, 4), (130, 2)])
def test_prolongation(m, N, prec, eps):
    torch = torch_mod()
    s, _, _ = make(m, N, precision=prec, cg_rtol=1e-6 if prec == "mixed" else 1e-10)
    mc = s.levels()[1]
    rng = np.random.default_rng(m + N)
    dt = np.float32 if prec == "mixed" else np.float64
    ec, ef = rng.standard_normal((mc ** 3, N)).astype(dt), rng.standard_normal((m ** 3, N)).astype(dt)
    P = interpolation(m, mc)
    ref = ec.astype(np.float64).reshape(mc, mc, mc, N)
    for axis in range(3):
        ref = np.moveaxis(np.tensordot(P, ref, (1, axis)), 0, axis)
    ref = ref.reshape(m ** 3, N) + ef
    tol = 10 * eps * (np.abs(ec).max() + np.abs(ef).max())
    assert np.abs(host(s.mg_prolong(0, dev(ec), dev(ef))) - ref).max() <= tol
    c, x = dev(ec), dev(ef)
    assert s.lib.hq_mg_prolong(s._ctx, 0, c.data_ptr(), x.data_ptr(), x.data_ptr()) == 0
    torch.cuda.synchronize()
    assert np.abs(host(x) - ref).max() <= tol
