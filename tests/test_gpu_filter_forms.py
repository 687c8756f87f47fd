"""Reduced-precision filters in every form of the degree loop: FE filters of narrow and wide blocks on few and many
cells (at most 32 columns: one launch per step from four cells per SM on), degrees whose steps do not fit one launch
(above 97), and two handles at work at once.  Tolerances: 5e-3 as in the other FE filter tests for short filters; for long
ones the operands' rounding of 2^-11 in every step, added up: degree 2^-11."""
import threading

import numpy as np
import pytest

import workloads as wl
from gpu_helpers import dense_case, ensure_built, lowp_reference, make_solver
from oracle import fe as ofe, filters
from oracle.filters import lambda_p

from paper_2503_22652_gb300 import Solver

pytestmark = pytest.mark.gpu
BOUNDS = (-25.0, 40.0, 2500.0)


@pytest.fixture(scope="module", autouse=True)
def _build():
    ensure_built()


def _fe(n, N, p, kpoint=None):
    q = wl.fe_problem(n) if kpoint is None else wl.fe_kpoint_problem(n, kpoint)
    A = ofe.assemble(q["cell_dofs"], q["A_cells"], q["m"])
    B = ofe.assemble(q["cell_dofs"], q["B_cell"], q["m"])
    d = q["Dinv"]
    rng = np.random.default_rng(N)
    X = rng.standard_normal((q["m"], N)) + (0 if kpoint is None else 1j * rng.standard_normal((q["m"], N)))
    L = np.sort(rng.uniform(-20.0, 30.0, N))
    W = A @ X - (B @ X) * L[None, :]
    exact = filters.rchfsi_filter(lambda R: A @ (d[:, None] * R), lambda R: d[:, None] * R, X, L, W, *BOUNDS, p)
    s = Solver(q["m"], nev=max(1, N // 2), block=N, precision="tf32", field="real" if kpoint is None else "complex")
    s.set_fe(q["cell_dofs"], q["A_cells"], q["B_cell"], q["Dinv"])
    return s, (X, L, W, *BOUNDS, p), exact, X * lambda_p(L, *BOUNDS, p)[None, :]


def _close(got, exact, base, tol):
    return np.linalg.norm(got - exact) <= tol * np.linalg.norm(exact - base)


# 8^3 and 9^3 cells lie on the two sides of four per SM (152), 5^3 and 6^3 of a quarter of that (complex)
@pytest.mark.parametrize("n,N", [(8, 32), (9, 4), (9, 28), (9, 32), (9, 36)])
def test_fe_widths_and_cells(n, N):
    s, args, exact, base = _fe(n, N, 5)
    for _ in range(2):
        assert _close(s.filter(*args), exact, base, 5e-3)


@pytest.mark.parametrize("n", [5, 6])
def test_fe_complex_narrow(n):
    s, args, exact, base = _fe(n, 12, 4, kpoint=(0.1, 0.2, -0.3))
    assert _close(s.filter(*args), exact, base, 5e-3)


# 97: the most that fit one launch
@pytest.mark.parametrize("N", [8, 32, 36, 130])
@pytest.mark.parametrize("p", [97, 98, 120])
def test_fe_long_filters(N, p):
    s, args, exact, base = _fe(2, N, p)
    assert _close(s.filter(*args), exact, base, p * 2.0 ** -11)


@pytest.mark.parametrize("on_device", [False, True])
@pytest.mark.parametrize("p", [97, 98, 120])
def test_dense_long_filters(p, on_device):
    case = dense_case(m=200, N=20)
    lmin, lT, lmax = case["bounds"]
    ref = lowp_reference(case, p, 10, 10, "truncate", lmin, lT, lmax)
    base = case["X"] * lambda_p(case["L"], lmin, lT, lmax, p)[None, :]
    s = make_solver(case, 20, precision="tf32")
    args = [case["X"], case["L"], case["W"]]
    if on_device:
        torch = pytest.importorskip("torch")
        args = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in args]
    got = s.filter(*args, lmin, lT, lmax, p)
    assert _close(got.cpu().numpy() if on_device else got, ref, base, p * 2.0 ** -11)


def test_two_handles_at_once():
    """The one-launch loops ask for all SMs: two dense and two FE handles, each from its own thread."""
    failures = []

    def dense(m, N):
        case = dense_case(m=m, N=N)
        s = make_solver(case, N, precision="tf32")
        args = (case["X"], case["L"], case["W"], *case["bounds"], 8)
        first = s.filter(*args)
        for _ in range(40):
            if not np.array_equal(s.filter(*args), first):
                failures.append(("dense", m))

    def fe(n, N):
        s, args, exact, base = _fe(n, N, 4)
        for _ in range(40):
            if not _close(s.filter(*args), exact, base, 5e-3):
                failures.append(("fe", n))

    def guarded(f, *a):
        try:
            f(*a)
        except Exception as e:  # noqa: BLE001
            failures.append(repr(e))

    threads = [threading.Thread(target=guarded, args=a) for a in ((dense, 500, 60), (dense, 900, 130), (fe, 3, 64),
                                                                  (fe, 4, 132))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failures
