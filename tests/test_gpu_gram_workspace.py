"""The SIMT Gram's partial sums stay in their scratch.

The scratch is sized for the 2N x 2N shapes of a step; at some N the N x N plans
have more tiles x chunks (161 .. 192: 6 tiles x 50 chunks against 21 x 14) and used
to run past it into the matrices a step keeps for the next one.  Reading the
iterate between two steps (eigenpairs, monitor) must not change the second, and
the Gram itself has to match its definition to the rounding of n terms.
"""
import numpy as np
import pytest

from gpu_common import dev, host, make

pytestmark = pytest.mark.gpu

# (m, N): symmetric plan too large; both plans; plan of the general Gram only
SHAPES = [(20, 161), (12, 330), (8, 321)]


@pytest.mark.parametrize("m,N", SHAPES)
def test_reading_the_iterate_leaves_the_next_step_alone(m, N):
    out = []
    for read in (False, True):
        s, _, _ = make(m, N, tau=0.2, cg_rtol=1e-10)
        s.step(1)
        if read:
            s.eigenpairs()
            s.monitor()
        s.step(1)
        out.append(s.get_state()[0])
    assert np.array_equal(out[0], out[1])


@pytest.mark.parametrize("m,N", SHAPES)
@pytest.mark.parametrize("sym", [True, False])
def test_gram_of_n_columns(m, N, sym):
    s, _, _ = make(m, N)
    rng = np.random.default_rng(m + N)
    A = rng.standard_normal((m ** 3, N))
    B = A if sym else rng.standard_normal((m ** 3, N))
    a = dev(A)
    g = host(s.gram(a, a if sym else dev(B), 1.0))
    bound = 2.0 ** -53 * m ** 3 * (np.abs(A).T @ np.abs(B))
    assert np.all(np.abs(g - A.T @ B) <= 2 * bound)
