"""Slices of the FP64-accurate products where rows do not fit in shared memory: rows along K at odd and even
lengths (8- and 16-byte loads, remainders of the four values of a thread), a second block of rows with one row,
and rows contiguous across threads (more than 1056 columns)."""
import numpy as np
import pytest

from oracle import rr
from gpu_helpers import ensure_built, dense_case, make_solver

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _build():
    ensure_built()


# tolerance: products exact to ~1e-15 of their row and column scales, times the condition number of the Gram
# matrix (below 30 for a Gaussian block of these shapes) and ~10^2 for the reduction: 1e-11 of the largest
@pytest.mark.parametrize("m,N", [(1153, 20), (1154, 33), (1155, 37), (2400, 1100)])
def test_rayleigh_ritz_long_rows(m, N):
    case = dense_case(m=m, N=N, generalized=False)
    Y = case["X"].copy()
    Y[:, 1] *= 1e-9  # rows of other scales
    s = make_solver(case, N, rr_mode="emulated")
    X, ev = s.rayleigh_ritz(Y)
    _, evr, _, _ = rr.rayleigh_ritz(Y, lambda v: case["A"] @ v, lambda v: v)
    np.testing.assert_allclose(ev, evr, rtol=0, atol=1e-11 * np.abs(evr).max())
    np.testing.assert_allclose(X.T @ X, np.eye(N), atol=1e-11)
