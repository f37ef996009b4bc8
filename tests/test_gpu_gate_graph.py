"""The gated step's graph with CFL steps: a redone step takes the wave rate and
the inadmissible-cell count of its own state, on every replay, and leaves the
context as it was for the plain steps that follow."""
import numpy as np
import pytest

import oracle
from paper_1707_00592_gb300 import learned
from paper_1707_00592_gb300 import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

import paper_1707_00592_gb300 as ws  # noqa: E402


def spot():
    """Air with a cell of hot light gas, which mixes away: the wave rate falls with every step.  Jumps in density
    from cell to cell at one side, where the linear weights fail."""
    n = (70, 47)
    y, x = np.mgrid[0:n[1], 0:n[0]]
    at = np.hypot(x - 35, y - 23.5) < 1.0
    G, P = wl.material(*wl.AIR)
    rho = np.where(x > 50, np.random.default_rng(3).uniform(1.2, 6.0, at.shape), 1.2)
    Q = wl._fill(2, n, [np.where(at, 0.024, rho), 300.0 * np.sin(x * 2 * np.pi / n[0]), 50.0 + 0.0 * x, 1e5 + 0.0 * x,
                        G + 0.0 * x, P + 0.0 * x])
    return n, (1e-3, 1e-3), (("transmissive", "transmissive"),) * 2, oracle.prim_to_cons(2, Q)


@pytest.mark.parametrize("mood", [True, False])
@pytest.mark.parametrize("first", [0, 1])
def test_redone_cfl_steps(mood, first):
    n, dx, bc, Uo = spot()
    runs = []
    for gated in (False, True):
        stream = torch.cuda.Stream()
        s = ws.Solver(2, n, dx, bc, precision="mixed", mood=mood, stream=stream)
        P = torch.tensor(learned.init_params(1), dtype=torch.float32, device="cuda")
        torch.cuda.synchronize()
        run = []
        with torch.cuda.stream(stream):
            U = s.tensor(Uo)

            def steps(k):
                for _ in range(k):
                    run.append((s.step(U, want_dt=True), s.nonphysical(), U.cpu().numpy()))

            steps(first)  # an odd and an even number of plain steps before
            if gated:  # linear weights everywhere: every step fails the drift check and is redone without the gate
                ws.ws_set_mlp(s.ctx, P, 1e30, ws.GATE_REDO_DRIFT | ws.GATE_REDO_NONPHYS)
            steps(6)
            if gated:
                st = ws.ws_gate_stats(s.ctx)
                assert st["steps"] == 6 and st["redone"] == 6, st
                ws.ws_set_mlp(s.ctx, None, 0.0)
            steps(3)
        s.close()
        runs.append(run)
    dts = [r[0] for r in runs[0]]
    assert all(b > a for a, b in zip(dts, dts[1:]))
    for (dp, bp, up), (dg, bg, ug) in zip(*runs):
        assert dp == dg and bp == bg and np.array_equal(up, ug)
