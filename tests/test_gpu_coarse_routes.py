"""Which levels of an FP32 V-cycle share a launch: from the first of at most 19
points per side down.  A side of 20 runs as separate kernels, as the finest level
of a problem and as a coarse one (launch counts per kernel class)."""
import numpy as np
import pytest

from gpu_common import dev, make

pytestmark = pytest.mark.gpu


def launches(m, N, **kw):
    s, _, _ = make(m, N, **kw)
    B = np.random.default_rng(m).standard_normal((m ** 3, N))
    s.block_pcg(dev(B.astype(np.float32) if kw.get("precision") == "mixed" else B), rtol=0.0, maxit=3)
    s.profile()
    s.block_pcg(dev(B.astype(np.float32) if kw.get("precision") == "mixed" else B), rtol=0.0, maxit=3)
    return {k: v[0] for k, v in s.profile_read().items()}


@pytest.mark.parametrize("m,separate", [(18, False), (19, False), (20, True), (21, True)])
def test_finest_level_of_an_fp32_preconditioner(m, separate):
    la = launches(m, 6, mg_fp32=1)
    assert (la["smooth"] > 0) == separate, la


@pytest.mark.parametrize("m,N,one", [(8, 152, True), (16, 304, True), (16, 305, False), (17, 152, True),
                                     (17, 153, False), (18, 4, False)])
def test_one_launch_pcg_by_waves_of_columns(m, N, one):
    """One CTA per column: two waves of the 152 SMs up to 16^3 points, one at 17^3."""
    la = launches(m, N, mg_fp32=1)
    assert (la["stencil"] == 0) == one, la


@pytest.mark.parametrize("m,separate", [(38, False), (39, False), (40, True), (41, True)])
@pytest.mark.parametrize("kw", [dict(mg_fp32=1), dict(precision="mixed", cg_rtol=1e-6)])
def test_second_level(m, separate, kw):
    # fused: one launch per V-cycle below the finest level; separate: a side of 20
    # alone has its sweeps, residual and transfers
    la = launches(m, 4, **kw)
    cycles = 3
    assert (la["coarse_grids"] > 2 * cycles) == separate, la
