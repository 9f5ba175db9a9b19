"""Relative accuracy of the smallest eigenvalue of a graded Gram.

U = Q D with columns of norms 1 .. 10^-k: <U,U> = D G D with a well-conditioned G.
Componentwise errors E_ij of D G D, |E_ij| <= e d_i d_j, move every eigenvalue by at
most N e / lambda_min(G) of itself.  Forming the Gram gives e = (n + 2) 2^-53 max|q|^2
(n rounded products), the eigensolver 20 N 2^-53 for all its rotations.  The reference
is the smallest singular value of U by one-sided Jacobi in extended precision.
"""
import numpy as np
import pytest

from paper_2605_25149_gb300 import hq, inputs

pytestmark = pytest.mark.gpu


def smallest_sv2(Y):
    """The smallest eigenvalue of Y^T Y: QR by Gram-Schmidt twice, one-sided Jacobi of R^T."""
    Q, N = Y.astype(np.longdouble), Y.shape[1]
    R = np.zeros((N, N), np.longdouble)
    for k in range(N):
        for _ in range(2):
            c = Q[:, :k].T @ Q[:, k]
            Q[:, k] -= Q[:, :k] @ c
            R[:k, k] += c
        R[k, k] = np.sqrt(Q[:, k] @ Q[:, k])
        Q[:, k] /= R[k, k]
    B = R.T.copy()
    for _ in range(30):
        worst = 0.0
        for p in range(N):
            for q in range(p + 1, N):
                a, b, g = B[:, p] @ B[:, p], B[:, q] @ B[:, q], B[:, p] @ B[:, q]
                worst = max(worst, float(abs(g) / np.sqrt(a * b)))
                if abs(g) > 1e-17 * np.sqrt(a * b):
                    z = (b - a) / (2 * g)
                    t = (1 if z >= 0 else -1) / (abs(z) + np.sqrt(1 + z * z))
                    c = 1 / np.sqrt(1 + t * t)
                    B[:, p], B[:, q] = c * B[:, p] - c * t * B[:, q], c * t * B[:, p] + c * B[:, q]
        if worst < 1e-16:
            break
    return float(np.min((B * B).sum(0)))


@pytest.mark.parametrize("N", [2, 5, 8, 16, 31, 48])
@pytest.mark.parametrize("k", [0, 3, 6, 7, 9])
def test_smallest_eigenvalue_of_a_graded_gram(N, k):
    m = 8
    n, h3 = m ** 3, inputs.grid_h(m) ** 3
    Q = np.random.default_rng(N + 100 * k).standard_normal((n, N)) / np.sqrt(n)
    d = np.logspace(0, -k, N)
    U = Q * d / np.sqrt(h3)
    s = hq.Solver(m, N)
    s.set_potential(inputs.harmonic(m))
    s.set_state(U, 0)
    got, ref = s.monitor()["smin"], smallest_sv2(U * np.sqrt(h3))
    e = 2.0 ** -53 * ((n + 2) * np.abs(Q.T @ Q).max() + 20 * N)
    assert abs(got - ref) <= ref * N * e / np.linalg.eigvalsh(Q.T @ Q)[0]


@pytest.mark.parametrize("N", [1, 2, 4, 5, 64, 112, 113])
@pytest.mark.parametrize("k", [-330, 330])
def test_scale_of_the_block_is_immaterial(N, k):
    """Powers of two pass through Gram, eigenvalues and the initial scaling exactly, also where
    the squares of the Gram's entries leave the exponent range (2^660 and 2^-660)."""
    m = 6
    U = np.random.default_rng(N).standard_normal((m ** 3, N))
    out = []
    for f in (1.0, 2.0 ** k):
        s = hq.Solver(m, N)
        s.set_potential(inputs.harmonic(m))
        s.set_state(U * f, 0)
        mon = s.monitor()
        s.set_initial(U * f)
        out.append((mon["smin"] / f / f, mon["smax"] / f / f, s.get_state()[0]))
    assert out[0][:2] == out[1][:2]
    assert np.array_equal(out[0][2], out[1][2])
