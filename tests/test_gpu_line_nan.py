"""A cell that is not a number makes the CFL step of a 1D grid not a number,
wherever in a block of threads it lies."""
import math

import numpy as np
import pytest

import oracle
from paper_1707_00592_gb300 import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

import paper_1707_00592_gb300 as ws  # noqa: E402


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
@pytest.mark.parametrize("n", [14, 127, 300])
def test_cfl_step_of_a_broken_cell(precision, n):
    case = wl.random_state(1, (n,), seed=3, kind="smooth")
    U0 = oracle.prim_to_cons(1, case.Q)
    s = ws.Solver(1, case.n, case.dx, case.bc, precision=precision)
    for x in range(n):
        f = x % 3  # density, momentum or energy
        U = U0.copy()
        U[f, 0, 0, 3 + x] = np.nan
        assert math.isnan(s.step(s.tensor(U), want_dt=True)), (x, f)
    assert s.step(s.tensor(U0), want_dt=True) > 0.0
