"""Chunks of a tube that hold one state are left out of the tube stages: the
waves must cross into them as if every chunk were evaluated.  Contacts and
pressure steps sit on and around the ends of chunks; after enough steps for
waves to reach the next chunks the states stay with the FP64 oracle, and cells
no wave has reached stay as they were."""
import numpy as np
import pytest

import oracle
from paper_1707_00592_gb300 import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

import paper_1707_00592_gb300 as ws  # noqa: E402


def batch(extra):
    """Tubes of 255 k + d cells with a step in pressure and density at cell 255 + s."""
    Ga, Pa = wl.material(*wl.AIR)
    Gw, Pw = wl.material(*wl.WATER)
    cols, off, steps = [], [0], []
    for k in (1, 2, 4):
        for d in (-2, 0, 1, 3, 100):
            for s in (-4, -3, -1, 0, 1, 3, 120):
                n = 255 * k + d
                at = min(max(255 + s, 10), n - 5)
                steps.append(at)
                x = np.arange(-3, n + 3)
                left = x < at
                water = (k + s) % 2 == 0
                cols.append(np.stack([np.where(left, 1000.0 if water else 2.0, 1.0), 30.0 + 0.0 * x,
                                      np.where(left, 3.0e6, 1.0e5), np.where(left, Gw if water else Ga, Ga),
                                      np.where(left, Pw if water else Pa, Pa)]))
                off.append(off[-1] + n + 6)
    for _ in range(extra):  # more tubes, for a batch that fills the GPU
        cols.append(cols[0])
        off.append(off[-1] + cols[0].shape[1])
    return np.array(off, dtype=np.int64), np.concatenate(cols, axis=1), steps


@pytest.mark.parametrize("extra", [0, 1100])
@pytest.mark.parametrize("graph", [False, True])
def test_waves_cross_into_quiet_chunks(extra, graph):
    off, Q, steps = batch(extra)
    stream = torch.cuda.Stream()
    s = ws.Solver(1, (1,), (1.0,), tube_offsets=off, precision="mixed", stream=stream)
    with torch.cuda.stream(stream):
        ws.ws_set_graph(s.ctx, graph)
        U = s.prim_to_cons(s.tensor(Q))
        U0 = U.cpu().numpy()
        for _ in range(40):
            s.step(U)
        bad = s.nonphysical()
        _, mask = s.mood(with_mask=True)
    Ug = U.cpu().numpy()
    stop = int(off[105])
    Uo = U0[:, :stop].copy()
    for _ in range(40):
        Uo, _ = oracle.tubes_step(off[:106], Uo)
    for t in range(105):
        a, b = off[t] + 3, off[t + 1] - 3
        for f in range(5):
            scale = np.abs(Uo[f, a:b]).max()
            assert np.abs(Ug[f, a:b] - Uo[f, a:b]).max() <= 2e-4 * max(scale, 1.0), (t, f)
        # 40 steps of at most half a cell: nothing has changed 230 cells away
        far = np.abs(np.arange(b - a) - steps[t]) > 230
        assert (Ug[:, a:b] == U0[:, a:b])[:, far].all()
    m = mask.cpu().numpy().reshape(3, -1)
    faces = np.zeros(m.shape[1], bool)
    for t in range(len(off) - 1):
        faces[off[t] + 2:off[t + 1] - 3] = True
    assert (m[:, faces] <= 10).all() and (m[:, ~faces] == 255).all()
    assert bad == 0
