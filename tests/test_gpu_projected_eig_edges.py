"""Projected eigenproblem and Cholesky kernels at the orders where their layout changes: 32-row
tiles and chunks, the cluster / grid line of the tridiagonalisation (320), the rows per thread (256),
the FP64 / tensor-core line of the N x N products (128), and spectra that exercise their branches
(diagonal M, a T that splits, widely spread values).  Compared with LAPACK on the same inputs; the
tolerances are 50 N eps ||M|| for values and 200 N eps for orthonormality (backward-stable steps whose
errors grow at most linearly in N)."""
import numpy as np
import pytest

import workloads as wl
from gpu_helpers import ensure_built

from paper_2503_22652_gb300 import Solver

pytestmark = pytest.mark.gpu
EPS = np.finfo(float).eps


@pytest.fixture(scope="module", autouse=True)
def _build():
    ensure_built()


def _run(A, Y):
    s = Solver(A.shape[0], nev=1, block=Y.shape[1])
    s.set_dense(A)
    return s.rayleigh_ritz(Y)


def _check(A, Y, X, ev):
    N = Y.shape[1]
    q, _ = np.linalg.qr(Y)
    ref = np.linalg.eigvalsh(q.T @ A @ q)
    nrm = max(np.abs(ref).max(), 1e-300)
    assert np.abs(ev - ref).max() <= 50 * N * EPS * nrm
    assert np.abs(X.T @ X - np.eye(N)).max() <= 200 * N * EPS
    assert np.abs(X.T @ A @ X - np.diag(ev)).max() <= 200 * N * EPS * nrm


@pytest.mark.parametrize("N", [2, 3, 4, 9, 31, 32, 33, 63, 64, 65, 96, 97, 127, 128, 129, 255, 256, 257, 319, 320,
                               321, 511, 513])
def test_orders(N):
    m = N + 40
    lam = np.linspace(-1.0, 10.0, m)
    A = wl.dense_from_spectrum(wl.orthogonal(m, 5), lam)
    Y = np.random.default_rng(N).standard_normal((m, N))
    X, ev = _run(A, Y)
    _check(A, Y, X, ev)


@pytest.mark.parametrize("N", [5, 40, 130, 330])
@pytest.mark.parametrize("kind", ["diagonal", "blocks", "spread"])
def test_spectra(N, kind):
    m = N + 8
    rng = np.random.default_rng(N + 1)
    Y = np.eye(m)[:, :N].copy()
    if kind == "diagonal":      # no Householder step does anything; T has zero off-diagonals
        A = np.diag(rng.permutation(np.linspace(-3.0, 4.0, m)))
    elif kind == "blocks":      # T splits in the middle
        A = np.zeros((m, m))
        h = N // 2
        for s in (slice(0, h), slice(h, m)):
            B = rng.standard_normal((m, m))[s, s]
            A[s, s] = 0.5 * (B + B.T)
    else:                       # eigenvalues over ten decades
        A = wl.dense_from_spectrum(wl.orthogonal(m, 9), np.logspace(-10, 0, m))
        Y = rng.standard_normal((m, N))
    X, ev = _run(A, Y)
    _check(A, Y, X, ev)


@pytest.mark.parametrize("N,bad", [(40, 0), (40, 33), (100, 31), (100, 96)])
def test_cholesky_reports_an_indefinite_gram(N, bad):
    """B indefinite in one direction of the block: the first non-positive pivot lies in any tile."""
    m = 120
    Y = np.eye(m)[:, :N].copy()
    B = np.eye(m)
    B[bad, bad] = -1.0
    from paper_2503_22652_gb300 import RChFSIError
    s = Solver(m, nev=1, block=N)
    s.set_dense(np.diag(np.arange(1.0, m + 1)), B=B)
    with pytest.raises(RChFSIError) as e:
        s.rayleigh_ritz(Y)
    assert e.value.code == -5  # RCHFSI_ERR_ILL_CONDITIONED
