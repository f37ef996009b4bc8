"""The 3D default configuration on both sides of its line: a step with it
equals, bit for bit, one with 32 x 15 tiles loaded cell by cell."""
import pytest

from paper_1707_00592_gb300 import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

import paper_1707_00592_gb300 as ws  # noqa: E402


# one CTA of either tile per SM; 32 x 15 once and 32 x 7 more than 1.5 times per SM; more of both
@pytest.mark.parametrize("n,height", [((24, 30, 40), 7), ((40, 22, 36), 15), ((45, 24, 30), 15), ((66, 34, 34), 7)])
def test_default_3d(n, height):
    case = wl.random_state(3, n, seed=7, kind="two_phase")
    out = []
    for index in (None, 1):
        s = ws.Solver(3, case.n, case.dx, case.bc, precision="mixed")
        if index is None:
            assert ws.ws_get_stage_config(s.ctx)["tile_y"] == height
        else:
            ws.ws_set_stage_config(s.ctx, index)
        U = s.prim_to_cons(s.tensor(case.Q))
        for _ in range(2):
            s.step(U)
        out.append(U[:, 3:-3, 3:-3, 3:-3].clone())
    assert torch.equal(out[0], out[1])
