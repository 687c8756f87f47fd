"""Rayleigh-Ritz where more projected eigenvalues agree than inverse iteration takes (256): the step is finished
from the library's eigenvectors, into host and device arrays, real and complex."""
import numpy as np
import pytest

import workloads as wl
from gpu_helpers import ensure_built

from paper_2503_22652_gb300 import Solver

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _build():
    ensure_built()


def _check(A, X, ev, lam):
    """Tolerances of the degenerate cases of the eigensolver's tests."""
    nrm = np.abs(lam).max()
    np.testing.assert_allclose(ev, lam, rtol=0, atol=1e-11 * nrm)
    np.testing.assert_allclose(X.conj().T @ X, np.eye(len(lam)), atol=1e-10)
    assert np.linalg.norm(A @ X - X * ev[None, :], axis=0).max() <= 1e-9 * nrm


@pytest.mark.parametrize("mode", ["emulated", "fp64"])
@pytest.mark.parametrize("cluster", [256, 257, 280])
def test_real(cluster, mode):
    torch = pytest.importorskip("torch")
    m, N = 340, 300
    lam = np.sort(np.concatenate([np.linspace(0.0, 1.0, 12), np.full(cluster, 2.0),
                                  np.linspace(3.0, 4.0, m - 12 - cluster)]))
    Q = wl.orthogonal(m, 3)
    A = wl.dense_from_spectrum(Q, lam)
    Y = Q[:, :N] @ np.random.default_rng(1).standard_normal((N, N))
    s = Solver(m, nev=1, block=N, rr_mode=mode)
    s.set_dense(A)
    for _ in range(2):
        X, ev = s.rayleigh_ritz(Y)
        _check(A, X, ev, lam[:N])
        X, ev = s.rayleigh_ritz(torch.from_numpy(Y).cuda())
        _check(A, X.cpu().numpy(), np.asarray(ev.cpu() if hasattr(ev, "cpu") else ev), lam[:N])


# the real form has every value twice: 280 of 300 agree in the first
@pytest.mark.parametrize("mode", ["emulated", "fp64"])
@pytest.mark.parametrize("m,N,cluster", [(170, 150, 140), (170, 150, 60), (80, 60, 40), (40, 30, 28)])
def test_complex(m, N, cluster, mode):
    rng = np.random.default_rng(5)
    Q, _ = np.linalg.qr(rng.standard_normal((m, m)) + 1j * rng.standard_normal((m, m)))
    lam = np.sort(np.concatenate([np.linspace(0.0, 1.0, 10), np.full(cluster, 2.0),
                                  np.linspace(3.0, 4.0, m - 10 - cluster)]))
    A = (Q * lam) @ Q.conj().T
    A = 0.5 * (A + A.conj().T)
    Y = Q[:, :N] @ (rng.standard_normal((N, N)) + 1j * rng.standard_normal((N, N)))
    s = Solver(m, nev=1, block=N, field="complex", rr_mode=mode)
    s.set_dense(A)
    for _ in range(2):
        X, ev = s.rayleigh_ritz(Y)
        _check(A, X, ev, lam[:N])


def test_solve():
    """The solve behind it: the wanted values among others that agree in more than 256."""
    m, N = 700, 300
    lam = np.sort(np.concatenate([np.linspace(-1.0, 0.0, 20), np.full(290, 1.0), np.linspace(2.0, 10.0, m - 310)]))
    Q = wl.orthogonal(m, 7)
    A = wl.dense_from_spectrum(Q, lam)
    s = Solver(m, nev=20, block=N, degree=20, precision="fp64", max_iter=60)
    s.set_dense(A)
    X, ev, res, st = s.solve(wl.gaussian_block(m, N, seed=2))
    assert st["max_rel_residual"] <= 1e-8
    np.testing.assert_allclose(ev[:20], lam[:20], atol=1e-9 * 10.0)
