"""Fixed-point sums of the FP64-accurate cell products where one cell's rows are far below the largest row at the
same dof: what lies below half of the accumulator's last place adds nothing, so a dof at which every product is
zero comes out as zero."""
import numpy as np
import pytest

import workloads as wl
from gpu_helpers import ensure_built

from paper_2503_22652_gb300 import Solver

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _build():
    ensure_built()


# 2^-50 of the largest row at a dof is where the shift of the low part reaches 63, 2^-82 that of the high part
@pytest.mark.parametrize("field", ["real", "complex"])
@pytest.mark.parametrize("power", [-49, -50, -51, -60, -82, -100])
def test_small_cell_rows_add_nothing_to_zero(field, power):
    cplx = field == "complex"
    q = wl.fe_kpoint_problem(3, (0.1, 0.2, -0.3)) if cplx else wl.fe_problem(3)
    dofs, A = q["cell_dofs"], q["A_cells"].copy()
    A[0] *= 2.0 ** power  # (its neighbours keep their size)
    if cplx:
        A = A.real + 1j * 2.0 ** power * A.imag
    m, N = q["m"], 5
    far = dofs[13].reshape(5, 5, 5)[1:4, 1:4, 1:4].ravel()  # the inner dofs of another cell
    zero = np.setdiff1d(np.arange(m), dofs[13])             # dofs that cell does not reach
    assert np.intersect1d(zero, dofs[0]).size > 0
    rng = np.random.default_rng(3)
    X = np.zeros((m, N), dtype=complex if cplx else float)
    X[far] = rng.standard_normal((far.size, N)) + (1j * rng.standard_normal((far.size, N)) if cplx else 0.0)
    s = Solver(m, nev=1, block=N, rr_mode="emulated", field=field)
    s.set_fe(dofs, A, q["B_cell"], q["Dinv"])
    W, _ = s.residual(X, np.linspace(-1.0, 1.0, N))
    assert np.abs(W[dofs[13]]).max() > 0.0
    assert np.array_equal(W[zero], np.zeros_like(W[zero]))
