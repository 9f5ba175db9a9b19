"""Eigenvalues of the small matrices, read through hq_monitor and hq_eigenpairs.

smin / smax are the extreme eigenvalues of <U,U>.  A backward-stable eigensolver
gives every eigenvalue within p(N) 2^-53 |S|; forming S by n rounded products
adds (n + 2) 2^-53 |u_i||u_j| h^3 per entry, below N (n + 2) 2^-53 max |u|^2 h^3 in
norm.  p(N) = 20 N covers the Jacobi rotations of all sweeps.
"""
import numpy as np
import pytest

from gpu_common import make
from paper_2605_25149_gb300 import hq, inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [1, 2, 3, 31, 64, 65, 111, 112, 113])
@pytest.mark.parametrize("kind", ["random", "graded", "equal"])
def test_extreme_eigenvalues_of_the_gram(N, kind):
    m = 6
    n, h3 = m ** 3, inputs.grid_h(m) ** 3
    rng = np.random.default_rng(N)
    U = rng.standard_normal((n, N)) / np.sqrt(n * h3)
    if kind == "graded":   # column norms over twelve orders of magnitude
        U *= np.logspace(0, -6, N)
    elif kind == "equal":  # orthonormal columns: all eigenvalues equal
        U = np.linalg.qr(U)[0] / np.sqrt(h3)
    s = hq.Solver(m, N)
    s.set_potential(inputs.harmonic(m))
    s.set_state(U, 0)
    mon = s.monitor()
    S = h3 * U.T @ U
    ev = np.linalg.eigvalsh(S)
    tol = 2.0 ** -53 * (20 * N * ev[-1] + 2 * N * (n + 2) * h3 * (np.abs(U) ** 2).max())
    assert abs(mon["smax"] - ev[-1]) <= tol and abs(mon["smin"] - ev[0]) <= tol


@pytest.mark.parametrize("N", [1, 2, 5, 64, 112, 113])
def test_ritz_pairs_are_orthonormal_and_meet_their_residuals(N):
    m = 7
    s, V, _ = make(m, N, cg_rtol=1e-10, cg_maxit=400)
    ev = s.eigenpairs(vectors=True)
    u, lam, h3 = ev["vectors"], ev["lam_rr"], inputs.grid_h(m) ** 3
    G = h3 * u.T @ u
    assert np.abs(G - np.eye(N)).max() <= 1e-11 * N
    X = np.zeros((m + 2, m + 2, m + 2, N))
    X[1:-1, 1:-1, 1:-1] = u.reshape(m, m, m, N)
    c = slice(1, -1)
    nb = (X[c, c, :-2] + X[c, c, 2:] + X[c, :-2, c] + X[c, 2:, c] + X[:-2, c, c] + X[2:, c, c]).reshape(m ** 3, N)
    h = inputs.grid_h(m)
    Hu = (3.0 / h ** 2 + V)[:, None] * u - 0.5 / h ** 2 * nb
    H = h3 * u.T @ Hu
    assert np.abs(H - np.diag(lam)).max() <= 1e-11 * N * np.abs(lam).max()
    assert np.all(np.diff(lam) >= 0)
