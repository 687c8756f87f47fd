"""Batched FE filters at block widths on both sides of the step's column tiles (narrow blocks, half tiles, more than
one tile of 128 columns): the batch chooses the form of the step by time, the results are those of the solves one
by one."""
import numpy as np
import pytest

import workloads as wl
from gpu_helpers import ensure_built

from paper_2503_22652_gb300 import Solver, solve_batch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _build():
    ensure_built()


@pytest.mark.parametrize("nev,N", [(16, 24), (44, 68), (100, 132)])
def test_batch_equals_alone(nev, N):
    problems = [wl.fe_problem(4, seed_wells=s) for s in (6, 9)]
    X0 = [wl.gaussian_block(p["m"], N, seed=2 + i) for i, p in enumerate(problems)]

    def solvers():
        out = []
        for p in problems:
            s = Solver(p["m"], nev=nev, block=N, degree=20, precision="tf32", max_iter=150)
            s.set_fe(p["cell_dofs"], p["A_cells"], p["B_cell"], p["Dinv"])
            out.append(s)
        return out

    alone = [s.solve(x) for s, x in zip(solvers(), X0)]
    for (_, ea, _, sa), (_, eb, _, sb) in zip(alone, solve_batch(solvers(), X0)):
        assert sa["max_rel_residual"] <= 1e-8 and sb["max_rel_residual"] <= 1e-8
        # both within the residual tolerance 1e-8 ||A|| of an eigenvalue, quadratically closer in value
        np.testing.assert_allclose(ea[:nev], eb[:nev], rtol=0, atol=1e-9 * np.abs(ea).max())
