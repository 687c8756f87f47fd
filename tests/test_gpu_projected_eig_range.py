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
