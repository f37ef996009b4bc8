"""A cell that is not a number makes the CFL step of a mixed-precision grid or
tube not a number, also where its thread goes on to further cells."""
import numpy as np
import pytest

import oracle
from paper_1707_00592_gb300 import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

import paper_1707_00592_gb300 as ws  # noqa: E402


@pytest.mark.parametrize("n,stride", [((70, 47), 11), ((40, 21, 9), 23)])
@pytest.mark.parametrize("config", [None, 0, 4])
def test_grids(n, stride, config):
    ndim = len(n)
    case = wl.random_state(ndim, n, seed=3, kind="smooth")
    s = ws.Solver(ndim, case.n, case.dx, case.bc, precision="mixed")
    if config is not None:
        ws.ws_set_stage_config(s.ctx, config)
    U0 = s.tensor(oracle.prim_to_cons(ndim, case.Q))
    for k in range(0, int(np.prod(n)), stride):
        at = tuple(3 + int(i) if d < ndim else 0 for d, i in
                   zip((2, 1, 0), reversed(np.unravel_index(k, n[::-1])[::-1] + (0,) * (3 - ndim))))
        U = U0.clone()
        U[(ndim + 1,) + at] = np.nan
        assert np.isnan(s.step(U, want_dt=True)), at


@pytest.mark.parametrize("extra", [0, 1000])  # chunks on 256 threads, on 128
def test_tubes(extra):
    lens = np.array([300] * 150 + [2000] * extra)
    off = np.concatenate([[0], np.cumsum(lens + 6)]).astype(np.int64)
    G, P = wl.material(*wl.AIR)
    s = ws.Solver(1, (1,), (1.0,), tube_offsets=off, precision="mixed")
    for first in (0, 1):
        U = s.tensor()
        for f, v in zip((0, 2, 3, 4), (1.2, 1e5 * G + P, G, P)):
            U[f] = v
        for t in range(150):  # another cell in each
            U[t % 3, int(off[t]) + 3 + 2 * t + first] = np.nan
        dt = s.step(U, want_dt=True)
        assert np.isnan(dt[:150]).all() and np.isfinite(dt[150:]).all()
