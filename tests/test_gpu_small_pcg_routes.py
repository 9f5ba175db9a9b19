"""The one-launch PCG wherever solves are run: replayed graphs, host-driven steps,
batches, and its error returns, against the separate kernels (HQ_FUSED_COARSE=0).
States and iteration counts are equal bit for bit, statuses equal.
"""
import numpy as np
import pytest

from gpu_common import dev, host, make
from paper_2605_25149_gb300 import hq

pytestmark = pytest.mark.gpu

NOT_CONVERGED, NONFINITE = 7, 9


def context(monkeypatch, m, N, fused=True, graphs=True, **kw):
    for name, off in (("HQ_FUSED_COARSE", not fused), ("HQ_NO_GRAPHS", not graphs)):
        if off:
            monkeypatch.setenv(name, "0" if name == "HQ_FUSED_COARSE" else "1")
        else:
            monkeypatch.delenv(name, raising=False)
    return make(m, N, mg_fp32=1, tau=0.4, **kw)[0]


@pytest.mark.parametrize("m,N", [(12, 5), (17, 8)])
def test_steps(monkeypatch, m, N):
    out = []
    for fused, graphs in ((True, True), (True, False), (False, True)):
        s = context(monkeypatch, m, N, fused, graphs, cg_rtol=1e-10)
        s.profile()
        g = [s.step(k) for k in (1, 3)]
        la = s.profile_read()
        out.append((g, s.pcg_stats(), *s.get_state(with_warm_start=True)))
        assert (la["smooth"][0] == 0) == fused   # no sweep of the finest level by itself
    for o in out[1:]:
        assert o[:2] == out[0][:2] and o[4] == out[0][4]
        assert np.array_equal(o[2], out[0][2]) and np.array_equal(o[3], out[0][3])


@pytest.mark.parametrize("graphs", [True, False])
@pytest.mark.parametrize("fused", [True, False])
def test_iteration_cap_in_a_step(monkeypatch, graphs, fused):
    m, N = 16, 8
    a = context(monkeypatch, m, N, cg_rtol=1e-10)
    a.step(2)
    U, Z, step = a.get_state(with_warm_start=True)
    b = context(monkeypatch, m, N, fused, graphs, cg_rtol=1e-14, cg_maxit=2)
    b.set_state(U, step, Z)
    with pytest.raises(hq.HQError) as e:
        b.step(2)
    assert e.value.status == NOT_CONVERGED


@pytest.mark.parametrize("fused", [True, False])
def test_nonfinite_right_hand_side(monkeypatch, fused):
    m, N = 9, 3
    s = context(monkeypatch, m, N, fused)
    B = np.random.default_rng(1).standard_normal((m ** 3, N))
    B[17, 1] = np.nan
    with pytest.raises(hq.HQError) as e:
        s.block_pcg(dev(B))
    assert e.value.status == NONFINITE
    B[17, 1] = 0.5   # the context goes on
    X, _ = s.block_pcg(dev(B), rtol=1e-10)
    r = host(s.apply_operator(X)) - B
    assert np.all(np.linalg.norm(r, axis=0) <= 1.1e-10 * np.linalg.norm(B, axis=0))


def test_batch_members(monkeypatch):
    shapes = [(16, 8), (12, 5), (20, 6)]   # two in one launch, one as separate kernels
    single = [context(monkeypatch, m, N, cg_rtol=1e-10) for m, N in shapes]
    member = [context(monkeypatch, m, N, cg_rtol=1e-10) for m, N in shapes]
    batch = hq.Batch(member)
    for n in (1, 3):
        g, stat = batch.step(n)
        assert (stat == 0).all()
        for k, (a, b) in enumerate(zip(member, single)):
            assert g[k] == b.step(n)
            assert np.array_equal(a.get_state()[0], b.get_state()[0])
    assert [a.pcg_stats() for a in member] == [b.pcg_stats() for b in single]


def test_batch_member_at_its_iteration_cap(monkeypatch):
    a = context(monkeypatch, 16, 8, cg_rtol=1e-14, cg_maxit=2)
    b = context(monkeypatch, 12, 5, cg_rtol=1e-10)
    with pytest.raises(hq.HQError) as e:
        hq.Batch([a, b]).step(2)
    assert e.value.status == NOT_CONVERGED and "problem 0" in str(e.value)


@pytest.mark.parametrize("scale,rtol,maxit", [(1.0, 1e-9, 1), (1.0, 0.0, 60), (1e-42, 1e-9, 60), (np.nan, 1e-9, 20),
                                              (np.inf, 0.0, 3), (1e200, 1e-9, 20), (1.0, 1e-9, 0)])
def test_failed_solves_are_counted(monkeypatch, scale, rtol, maxit):
    """At the cap, broken down at rounding level (rtol 0; right-hand sides that vanish in FP32),
    with a non-finite value: status and hq_pcg_stats as of the separate kernels."""
    m, N = 9, 3
    B = np.random.default_rng(0).standard_normal((m ** 3, N))
    if np.isfinite(scale):
        B *= scale
    else:
        B[5, 1] = scale
    out = []
    for fused in (True, False):
        s = context(monkeypatch, m, N, fused)
        s.profile()
        try:
            s.block_pcg(dev(B), rtol=rtol, maxit=maxit)
            status = 0
        except hq.HQError as e:
            status = e.status
        out.append((status, s.pcg_stats()))
    assert out[0] == out[1] and out[0][1][0] == 1
