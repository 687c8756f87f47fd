"""Dense filters under hbm_budget_bytes: the one-launch degree loop, which needs a larger workspace, is taken only
where everything the call needs fits; below that the per-step products give the result.  A budget that suffices is
never one that a larger budget makes insufficient."""
import numpy as np
import pytest

from gpu_helpers import dense_case, ensure_built, lowp_reference, make_solver
from oracle.filters import lambda_p

from paper_2503_22652_gb300 import RChFSIError

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _build():
    ensure_built()


# (tolerances of the reduced-precision parity tests)
@pytest.mark.parametrize("prec,bits,mode,tol", [("tf32", 10, "truncate", 2e-3), ("bf16", 7, "nearest", 2e-2)])
@pytest.mark.parametrize("chfsi_first", [False, True])
def test_a_larger_budget_is_no_worse(prec, bits, mode, tol, chfsi_first):
    m, N, p = 1000, 60, 6
    case = dense_case(m=m, N=N)
    lmin, lT, lmax = case["bounds"]
    ref = lowp_reference(case, p, bits, bits, mode, lmin, lT, lmax)
    base = case["X"] * lambda_p(case["L"], lmin, lT, lmax, p)[None, :]
    ok = []
    for budget in np.arange(8 << 20, 48 << 20, 512 << 10):
        try:
            s = make_solver(case, N, precision=prec, hbm_budget_bytes=int(budget))
            if chfsi_first:
                s.chfsi_filter(case["X"], lmin, lT, lmax, p)
            got = s.filter(case["X"], case["L"], case["W"], lmin, lT, lmax, p)
        except RChFSIError as e:
            assert "hbm_budget_bytes" in str(e)
            ok.append(False)
            continue
        ok.append(True)
        assert np.linalg.norm(got - ref) <= tol * np.linalg.norm(ref - base)
    assert ok == sorted(ok) and not ok[0] and ok[-1]
