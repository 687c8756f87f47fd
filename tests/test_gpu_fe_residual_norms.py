"""Column norms of the FE residual, each measured against its own column's scale."""
import numpy as np
import pytest

import workloads as wl
from gpu_helpers import ensure_built

from paper_2503_22652_gb300 import Solver

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _build():
    ensure_built()


@pytest.mark.parametrize("N", [1, 33, 130])
def test_norms_per_column(N):
    q = wl.fe_problem(3)
    rng = np.random.default_rng(N)
    X = rng.standard_normal((q["m"], N)) * np.logspace(-5, 5, N)[None, :]
    X[:, N // 2] = 0.0 if N > 1 else X[:, 0]
    s = Solver(q["m"], nev=1, block=N, rr_mode="emulated")
    s.set_fe(q["cell_dofs"], q["A_cells"], q["B_cell"], q["Dinv"])
    W, r = s.residual(X, np.sort(rng.uniform(-20.0, 30.0, N)))
    # a sum of m squares in FP64, however it is split: m eps / 2, and the root and its rounding
    ref = np.linalg.norm(W, axis=0)
    assert (np.abs(r - ref) <= q["m"] * np.finfo(float).eps * ref).all()
