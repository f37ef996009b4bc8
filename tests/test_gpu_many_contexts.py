"""More grid contexts than there are slots for steps in mapped memory: all
report the same steps, and a slot that is given back serves the next context."""
import pytest

import oracle
from paper_1707_00592_gb300 import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

import paper_1707_00592_gb300 as ws  # noqa: E402


@pytest.mark.parametrize("ndim,n,precision", [(1, (40,), "fp64"), (1, (40,), "mixed"), (2, (20, 16), "mixed")])
def test_steps_with_and_without_a_slot(ndim, n, precision):
    case = wl.random_state(ndim, n, seed=2, kind="shock")
    U = oracle.prim_to_cons(ndim, case.Q)

    def steps(s):
        V = s.tensor(U)
        return [s.step(V, want_dt=True) for _ in range(3)]

    def new():
        return ws.Solver(ndim, case.n, case.dx, case.bc, precision=precision)

    many = [new() for _ in range(70)]
    want = steps(many[0])
    assert all(steps(s) == want for s in many)
    for s in many[3:60:4]:
        s.close()
    assert all(steps(new()) == want for _ in range(20))
