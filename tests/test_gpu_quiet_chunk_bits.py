"""Quiet chunks of tubes, bit for bit: the same jumps in tubes whose chunks are
quiet but for them, and in tubes where a bump far from every jump keeps every
chunk moving.  As long as the bumps are out of reach the cells and MOOD bytes
around the jumps are the same."""
import numpy as np
import pytest

from paper_1707_00592_gb300 import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

import paper_1707_00592_gb300 as ws  # noqa: E402

CHUNK, STEPS = 255, 7
NEAR = 54  # jumps lie 122 cells and more from the bumps, whose reach is 9 cells per step


@pytest.mark.parametrize("extra", [0, 1100])  # chunks on 256 threads, on 128
@pytest.mark.parametrize("weights", ["modified", "js"])
def test_jump_crosses_into_quiet_chunks(extra, weights):
    Ga, Pa = wl.material(*wl.AIR)
    Gw, Pw = wl.material(*wl.WATER)
    n = 4 * CHUNK
    at = [c * CHUNK + s for c in (1, 2, 3) for s in (-6, -4, -3, -2, -1, 0, 1, 2, 3, 5)]
    tubes = len(at) + extra
    off = np.arange(tubes + 1, dtype=np.int64) * (n + 6)
    x = np.arange(-3, n + 3)
    Q = np.empty((5, tubes, n + 6))
    for t in range(tubes):
        left, water = x < at[t % len(at)], t % 2 == 0
        Q[:, t] = [np.where(left, 1000.0 if water else 2.0, 1.0), 30.0 + 0.0 * x, np.where(left, 3.0e6, 1.0e5),
                   np.where(left, Gw if water else Ga, Ga), np.where(left, Pw if water else Pa, Pa)]
    B = Q.copy()
    for c in range(4):
        B[0, :, 3 + c * CHUNK + CHUNK // 2] *= 1.001
    s, r = (ws.Solver(1, (1,), (1.0,), tube_offsets=off, precision="mixed", weights=weights) for _ in range(2))
    U, V = (k.prim_to_cons(k.tensor(q.reshape(5, -1))) for k, q in ((s, Q), (r, B)))
    first = U.clone()
    dt = float(s.step(U.clone(), want_dt=True).min())
    assert NEAR + 9 * STEPS + 4 < CHUNK // 2 - 5
    near = torch.tensor(np.array([np.abs(x - at[t % len(at)]) <= NEAR for t in range(tubes)]).ravel(), device="cuda")
    for _ in range(STEPS):
        s.step(U, dt)
        r.step(V, dt)
        assert torch.equal(U[:, near], V[:, near])
        (_, m), (_, k) = s.mood(with_mask=True), r.mood(with_mask=True)
        assert torch.equal(m.reshape(3, -1)[:, near], k.reshape(3, -1)[:, near])
    moved = (U != first).any(0).reshape(tubes, -1)
    assert bool((moved.sum(1) > 10).all())
