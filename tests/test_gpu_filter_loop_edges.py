"""The one-launch degree loop of the dense filter at the sizes where its tiles and shares have edges, against the
oracle on equally rounded operands.  Tolerances are those of the reduced-precision parity tests (FP32 accumulation
and storage amplified over the degree)."""
import numpy as np
import pytest

from gpu_helpers import dense_case, ensure_built, lowp_reference, make_solver
from oracle.filters import lambda_p

pytestmark = pytest.mark.gpu

LOWP = {"tf32": (10, 10, "truncate", 2e-3), "bf16": (7, 7, "nearest", 2e-2)}


@pytest.fixture(scope="module", autouse=True)
def _build():
    ensure_built()


# one row tile and one column; tile edges; shares that do not divide N and empty shares; each size of a thread's
# part of a share; the largest N of the loop and the first beyond it
@pytest.mark.parametrize("m,N,prec,p", [(40, 1, "tf32", 3), (128, 16, "bf16", 2), (129, 17, "tf32", 5),
                                        (513, 33, "bf16", 8), (1000, 60, "tf32", 8), (641, 130, "tf32", 6),
                                        (700, 200, "bf16", 6), (600, 256, "tf32", 5), (600, 257, "tf32", 5)])
def test_loop_matches_reference(m, N, prec, p):
    case = dense_case(m=m, N=N, generalized=m == 513)
    bits_op, bits_r, mode, tol = LOWP[prec]
    lmin, lT, lmax = case["bounds"]
    ref = lowp_reference(case, p, bits_op, bits_r, mode, lmin, lT, lmax)
    s = make_solver(case, N, precision=prec)
    base = case["X"] * lambda_p(case["L"], lmin, lT, lmax, p)[None, :]
    for _ in range(2):  # the second call finds used workspaces
        got = s.filter(case["X"], case["L"], case["W"], lmin, lT, lmax, p)
        assert np.linalg.norm(got - ref) <= tol * np.linalg.norm(ref - base)
