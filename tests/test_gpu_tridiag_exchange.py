"""Tridiagonalisation at orders around multiples of its CTA counts (8 up to order 96, 16 up to 320, 96 up to 512,
128 above), where a CTA runs out of columns at every distance from the last step, with two handles at work at
once, so that CTAs are held back at different points.  Compared with LAPACK; the tolerances are those of the
other projected-eigenproblem tests: 50 N eps ||M|| for values, 200 N eps for orthonormality."""
import threading

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


@pytest.mark.parametrize("orders", [(3, 7, 8), (9, 15, 17), (16, 24, 25), (88, 95, 96), (97, 111, 113), (160, 176, 305),
                                    (320, 321, 335), (383, 384, 385), (480, 511, 512), (513, 639, 641)])
def test_orders_around_the_cta_counts(orders):
    failures = []

    def work(seed, reps):
        for N in orders:
            m = N + 24
            rng = np.random.default_rng(100 * N + seed)
            A = wl.dense_from_spectrum(wl.orthogonal(m, seed), np.sort(rng.uniform(-1.0, 10.0, m)))
            Y = rng.standard_normal((m, N))
            ref = np.linalg.eigvalsh((lambda q: q.T @ A @ q)(np.linalg.qr(Y)[0]))
            s = Solver(m, nev=1, block=N)
            s.set_dense(A)
            for _ in range(reps):
                X, ev = s.rayleigh_ritz(Y)
                err = np.abs(ev - ref).max() / np.abs(ref).max(), np.abs(X.T @ X - np.eye(N)).max()
                if not (err[0] <= 50 * N * EPS and err[1] <= 200 * N * EPS):
                    failures.append((N, seed) + err)

    def guarded(*args):
        try:
            work(*args)
        except Exception as e:  # noqa: BLE001
            failures.append(repr(e))

    threads = [threading.Thread(target=guarded, args=(seed, 6)) for seed in (1, 2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failures
