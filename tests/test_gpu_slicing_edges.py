"""Slicing of the emulated FP64 products in one pass (rows in shared memory) and in separate passes,
at the row lengths where the route changes and at rows that need care: zero rows, values over many
decades, one row.  Compared with NumPy through the Rayleigh-Ritz products; tolerance 1e-13 relative
to the row / column norms (the emulated products carry ~1e-15)."""
import numpy as np
import pytest

from gpu_helpers import ensure_built

from paper_2503_22652_gb300 import Solver

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _build():
    ensure_built()


# m is the length of the K-contiguous rows (one pass up to 8447, then separate), N that of the
# row-contiguous ones (one pass up to 1030)
@pytest.mark.parametrize("m,N", [(33, 1), (64, 20), (257, 31), (1000, 60), (1025, 130), (2113, 129), (2600, 20),
                                 (8500, 24)])
def test_rayleigh_ritz_products(m, N):
    rng = np.random.default_rng(m)
    d = np.logspace(-3, 1, m)
    u = rng.standard_normal((m, 2)) / np.sqrt(m)
    A = np.diag(d) + u @ u.T if m < 4000 else np.diag(d)
    Y = rng.standard_normal((m, N)) * np.logspace(-4, 4, N)[None, :]
    Y[:: 7, : N // 2] = 0.0
    Y[5, :] = 0.0  # a zero row: its slices have no exponent
    s = Solver(m, nev=1, block=N)
    s.set_dense(A)
    X, ev = s.rayleigh_ritz(Y)
    Yn = Y / np.linalg.norm(Y, axis=0)
    q, _ = np.linalg.qr(Yn)
    ref = np.linalg.eigvalsh(q.T @ A @ q)
    assert np.abs(ev - ref).max() <= 1e-12 * np.abs(ref).max()
    assert np.abs(X.T @ X - np.eye(N)).max() <= 1e-11
    assert np.abs(X[5]).max() <= 1e-13
