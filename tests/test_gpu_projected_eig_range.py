"""Projected eigenproblem of matrices whose entries lie near the ends of what the sums of squares of its Householder
columns hold."""
import numpy as np
import pytest

from gpu_helpers import ensure_built

from paper_2503_22652_gb300 import RChFSIError, Solver

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _build():
    ensure_built()


def _full(m, seed):
    r = np.random.default_rng(seed).uniform(0.5, 1.0, (m, m))
    return np.triu(r) + np.triu(r, 1).T


@pytest.mark.parametrize("N", [12, 60, 340])
def test_overflowing_sum_of_squares_is_not_a_result(N):
    """Squares that are finite and whose sum is not: the call fails or returns non-finite values, it does not
    return eigenvalues as if the columns were already reduced."""
    A = 2.0 ** 511 * _full(N, 1)
    s = Solver(N, nev=1, block=N)
    s.set_dense(A)
    try:
        _, ev = s.rayleigh_ritz(np.eye(N))
    except RChFSIError:
        return
    assert not np.isfinite(ev).all()


# tolerances of the other projected-eigenproblem tests: 50 N eps ||M|| for values, 200 N eps for orthonormality
@pytest.mark.parametrize("N", [12, 60, 130, 340])
@pytest.mark.parametrize("power", [-480, -400, -300, -250, 250, 300, 400, 480])
def test_scaled_matrices(N, power):
    """Scaling A by a power of two scales the eigenvalues."""
    A = _full(N, 2)
    ref = np.linalg.eigvalsh(A)
    s = Solver(N, nev=1, block=N)
    s.set_dense(2.0 ** power * A)
    X, ev = s.rayleigh_ritz(np.eye(N))
    eps = np.finfo(float).eps
    assert np.abs(ev * 2.0 ** -power - ref).max() <= 50 * N * eps * np.abs(ref).max()
    assert np.abs(X.T @ X - np.eye(N)).max() <= 200 * N * eps


@pytest.mark.parametrize("N", [12, 60, 340])
@pytest.mark.parametrize("power", [-200, -260, -400, -505])
def test_columns_of_tiny_entries(N, power):
    """Off-diagonal entries far below the diagonal: in one half of the matrix, then in all of it."""
    eps = np.finfo(float).eps
    for h in (N // 2, 0):
        A = _full(N, 3)
        A[h:, :] *= 2.0 ** power
        A[:h, h:] *= 2.0 ** power
        A[np.arange(h, N), np.arange(h, N)] = np.linspace(1.0, 2.0, N - h)
        ref = np.linalg.eigvalsh(A)
        s = Solver(N, nev=1, block=N, rr_mode="fp64")
        s.set_dense(A)
        X, ev = s.rayleigh_ritz(np.eye(N))
        assert np.abs(ev - ref).max() <= 50 * N * eps * np.abs(ref).max()
        assert np.abs(X.T @ X - np.eye(N)).max() <= 200 * N * eps


@pytest.mark.parametrize("mode", ["emulated", "fp64"])
@pytest.mark.parametrize("power", [-1040, -1030, -1022, 1021, 1022])
def test_gram_matrices_at_the_ends_of_the_range(power, mode):
    """A and B scaled alike: the eigenvalues stay.  Tolerance: 50 N units of the scaled matrices' last place."""
    N = 40
    r = np.random.default_rng(1)
    A, B = r.uniform(-1.0, 1.0, (N, N)), r.uniform(-0.0125, 0.0125, (N, N))
    A, B = A + A.T, np.eye(N) + B + B.T
    L = np.linalg.inv(np.linalg.cholesky(B))
    ref = np.linalg.eigvalsh(L @ A @ L.T)
    s = Solver(N, nev=1, block=N, rr_mode=mode)
    s.set_dense(np.ldexp(A, power), B=np.ldexp(B, power))
    _, ev = s.rayleigh_ritz(np.eye(N))
    assert np.abs(ev - ref).max() <= 50 * N * max(np.finfo(float).eps, 2.0 ** (-1074 - power)) * np.abs(ref).max()


@pytest.mark.parametrize("powers", [(-1000, 0), (0, -1000), (-1000, 90), (900, -60), (-60, 900)])
def test_graded_gram_matrices(powers):
    """A diagonal B of two scales far apart, either first: the pivots are its entries, exact."""
    N = 40
    d = np.where(np.arange(N) < N // 2, 2.0 ** powers[0], 2.0 ** powers[1])
    lam = np.linspace(1.0, 2.0, N)
    s = Solver(N, nev=1, block=N, rr_mode="fp64")
    s.set_dense(np.diag(d * lam), B=np.diag(d))
    _, ev = s.rayleigh_ritz(np.eye(N))
    assert np.abs(ev - lam).max() <= 50 * N * np.finfo(float).eps * 2.0
