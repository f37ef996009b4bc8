"""A 1D grid whose increments have more than 2^31 elements: one step of uniform
air with a two-phase block at its far end equals, bit for bit, the step of a
short grid that holds the block and the air around it."""
import pytest

from paper_1707_00592_gb300 import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

import paper_1707_00592_gb300 as ws  # noqa: E402

N = 2**29 + 37  # 4 N > 2^31
BLOCK, MARGIN = 40, 100


def run(n, precision):
    """The last 2 MARGIN + BLOCK cells after a step of n cells, and the step."""
    G, P = wl.material(*wl.AIR)
    s = ws.Solver(1, (n,), (1e-3,), precision=precision)
    U = None
    try:
        Q = s.tensor()
        for f, v in enumerate((1.2, 0.0, 1e5, G, P)):
            Q[f] = v
        at = 3 + n - MARGIN - BLOCK
        Q[:, 0, 0, at:at + BLOCK] = torch.tensor(
            wl.random_state(1, (BLOCK,), seed=5, kind="two_phase").Q[:, 0, 0, 3:-3], device="cuda")
        U = s.prim_to_cons(Q)
        del Q
        dt = s.step(U, want_dt=True)
        assert s.nonphysical() == 0
        return dt, U[:, 0, 0, 3 + n - 2 * MARGIN - BLOCK:3 + n].clone()
    finally:
        s.close()
        del U
        torch.cuda.empty_cache()


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_far_end(precision):
    torch.cuda.empty_cache()
    if torch.cuda.mem_get_info()[0] < 150 * 2**30:
        pytest.skip("needs 150 GB of free device memory")
    dt, end = run(N, precision)
    dt0, end0 = run(2 * MARGIN + BLOCK, precision)
    assert dt == dt0 and torch.equal(end, end0)
