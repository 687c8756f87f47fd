"""The one-launch degree loop of the dense filter and the row-major entry of the filters, at the sizes where
their tiles and shares have edges, against the oracle on equally rounded operands.  Tolerances are
those of the reduced-precision parity tests (FP32 accumulation and storage amplified over the degree)."""
import numpy as np
import pytest

import workloads as wl
from gpu_helpers import dense_case, ensure_built, lowp_reference, make_solver
from oracle.filters import lambda_p

from paper_2503_22652_gb300 import Solver

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


def _overlaps(s, X, L, W, args):
    """The result written over X, over W and over an array that overlaps X shifted by a row."""
    torch = pytest.importorskip("torch")
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    ref = s.filter(dev(X), dev(L), dev(W), *args).cpu().numpy()
    for which in ("X", "W", "shifted"):
        x, w = dev(X), dev(W)
        out = {"X": x, "W": w}.get(which)
        if out is None:
            both = torch.empty((X.shape[0] + 1, X.shape[1]), dtype=torch.float64, device="cuda")
            x = both[:-1].copy_(x)
            out = both[1:]
        s.filter(x, dev(L), w, *args, out=out)
        yield ref, out.cpu().numpy()


def test_output_may_overlap_inputs_dense():
    case = dense_case(m=200, N=23)
    s = make_solver(case, 23, precision="tf32")
    for ref, got in _overlaps(s, case["X"], case["L"], case["W"], (*case["bounds"], 6)):
        assert np.array_equal(ref, got)


# (tolerances of the reduced-precision FE filter parity tests; two runs differ in the order of the cell sums, and
# a TF32 or BF16 rounding that flips is no smaller than that of a single product)
@pytest.mark.parametrize("N,prec,tol", [(24, "tf32", 5e-3), (41, "tf32", 5e-3), (130, "tf32", 5e-3), (41, "bf16", 5e-2)])
def test_output_may_overlap_inputs_fe(N, prec, tol):
    from oracle import fe as ofe, filters
    q = wl.fe_problem(2)
    A = ofe.assemble(q["cell_dofs"], q["A_cells"], q["m"])
    B = ofe.assemble(q["cell_dofs"], q["B_cell"], q["m"])
    d = q["Dinv"]
    rng = np.random.default_rng(5)
    X = rng.standard_normal((q["m"], N))
    L = np.sort(rng.uniform(-20.0, 30.0, N))
    W = A @ X - (B @ X) * L[None, :]
    args = (-25.0, 40.0, 2500.0, 8)
    exact = filters.rchfsi_filter(lambda R: A @ (d[:, None] * R), lambda R: d[:, None] * R, X, L, W, *args)
    base = X * lambda_p(L, *args)[None, :]
    s = Solver(q["m"], nev=N // 2, block=N, precision=prec)
    s.set_fe(q["cell_dofs"], q["A_cells"], q["B_cell"], q["Dinv"])
    for ref, got in _overlaps(s, X, L, W, args):
        for y in (ref, got):
            assert np.linalg.norm(y - exact) <= tol * np.linalg.norm(exact - base)


# one step, an even and an odd number of them; widths around the half tiles and tiles of the step; fewer cells than
# SMs and more; tolerance of the reduced-precision FE filter parity test
@pytest.mark.parametrize("n,N,p", [(2, 4, 2), (2, 64, 3), (3, 68, 4), (3, 128, 5), (2, 132, 3), (6, 48, 4)])
def test_fe_degree_loop(n, N, p):
    from oracle import fe as ofe, filters
    q = wl.fe_problem(n)
    A = ofe.assemble(q["cell_dofs"], q["A_cells"], q["m"])
    B = ofe.assemble(q["cell_dofs"], q["B_cell"], q["m"])
    d = q["Dinv"]
    rng = np.random.default_rng(N)
    X = rng.standard_normal((q["m"], N))
    L = np.sort(rng.uniform(-20.0, 30.0, N))
    W = A @ X - (B @ X) * L[None, :]
    args = (-25.0, 40.0, 2500.0, p)
    exact = filters.rchfsi_filter(lambda R: A @ (d[:, None] * R), lambda R: d[:, None] * R, X, L, W, *args)
    base = X * lambda_p(L, *args)[None, :]
    s = Solver(q["m"], nev=max(1, N // 2), block=N, precision="tf32")
    s.set_fe(q["cell_dofs"], q["A_cells"], q["B_cell"], q["Dinv"])
    for _ in range(2):
        got = s.filter(X, L, W, *args)
        assert np.linalg.norm(got - exact) <= 5e-3 * np.linalg.norm(exact - base)


@pytest.mark.parametrize("N", [1, 31, 65, 130])
def test_fe_residual_rows(N):
    from oracle import fe as ofe
    q = wl.fe_problem(3)
    A = ofe.assemble(q["cell_dofs"], q["A_cells"], q["m"])
    B = ofe.assemble(q["cell_dofs"], q["B_cell"], q["m"])
    rng = np.random.default_rng(N)
    X = rng.standard_normal((q["m"], N)) * np.logspace(-5, 5, N)[None, :]
    X[:, N // 2] = 0.0
    L = np.sort(rng.uniform(-20.0, 30.0, N))
    s = Solver(q["m"], nev=1, block=N, rr_mode="emulated")
    s.set_fe(q["cell_dofs"], q["A_cells"], q["B_cell"], q["Dinv"])
    W, r = s.residual(X, L)
    ref = A @ X - (B @ X) * L[None, :]
    scale = np.abs(A).sum(1).max() * np.linalg.norm(X, axis=0) + 1e-300
    assert (np.linalg.norm(W - ref, axis=0) / scale).max() <= 1e-14
    assert np.allclose(r, np.linalg.norm(ref, axis=0), rtol=1e-12, atol=1e-12 * scale.max() * 1e-3)
    X[3, 0] = np.inf
    W, r = s.residual(X, L)
    assert np.isnan(r[0]) and (N == 1 or np.isfinite(r[1:]).all())
