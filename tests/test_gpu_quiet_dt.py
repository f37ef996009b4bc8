"""A time step that is not finite reaches every cell, those of quiet tiles and
chunks too."""
import math

import numpy as np
import pytest

from paper_1707_00592_gb300 import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

import paper_1707_00592_gb300 as ws  # noqa: E402

G, P = wl.material(*wl.AIR)
REST = (1.2, 1e5 * G + P, G, P)  # rho, E, Gamma, Pi


def same(a, b):
    return bool(((a == b) | (torch.isnan(a) & torch.isnan(b))).all())


# a broken cell, and a given step beyond the FP32 range
@pytest.mark.parametrize("cell,dt", [(True, 0.0), (False, 1e300)])
@pytest.mark.parametrize("config", [None, 1, 8])
@pytest.mark.parametrize("resident", [False, True])
def test_tiles(cell, dt, config, resident):
    n = (1027, 601)  # enough tiles for the short way of quiet ones
    bc = (("transmissive", "transmissive"),) * 2
    out = []
    for census in (False, True):  # the census step evaluates every face
        s = ws.Solver(2, n, (1e-3, 1e-3), bc, precision="mixed")
        if config is not None:
            ws.ws_set_stage_config(s.ctx, config)
        if resident and not census:
            ws.ws_set_resident(s.ctx, True)
        U = s.tensor()
        for f, v in zip((0, 3, 4, 5), REST):
            U[f] = v
        if cell:
            U[3, 0, 50, 40] = math.nan
        used = s.census_step(U, dt)["dt"] if census else s.step(U, dt, want_dt=True)
        out.append((used, U[:, 0, 3:-3, 3:-3].clone(), s.nonphysical(), s.mood(with_mask=True)))
        s.close()
    (da, ua, ba, (ca, ma)), (db, ub, bb, (cb, mb)) = out
    assert math.isnan(da) if cell else da == db == dt
    assert same(ua, ub) and bool(torch.isnan(ua).all())
    assert ba == bb == n[0] * n[1]
    assert np.array_equal(ca, cb) and bool((ma == mb).all())


@pytest.mark.parametrize("cell,dt", [(True, 0.0), (False, 1e300)])
@pytest.mark.parametrize("mood", [True, False])
@pytest.mark.parametrize("graph", [False, True])
@pytest.mark.parametrize("extra", [0, 1100])  # both chunk layouts
def test_chunks(cell, dt, mood, graph, extra):
    lens = [900, 255, 1021, 256, 2000] + [1300] * extra
    off = np.concatenate([[0], np.cumsum(np.array(lens) + 6)]).astype(np.int64)
    stream = torch.cuda.Stream()
    out = []
    for broken in (False, True):
        s = ws.Solver(1, (1,), (1.0,), tube_offsets=off, precision="mixed", mood=mood, stream=stream)
        with torch.cuda.stream(stream):
            ws.ws_set_graph(s.ctx, graph)
            U = s.tensor()
            for f, v in zip((0, 2, 3, 4), REST):
                U[f] = v
            for t in (0, 2):  # a step in pressure, so that some chunks move
                U[2, int(off[t]) + 403:int(off[t + 1])] *= 1.5
            if broken and cell:  # a cell of the third tube
                U[2, int(off[2]) + 3 + 657] = math.nan
            used = s.step(U, dt if broken else 0.0, want_dt=True)
            out.append((used, U.clone(), s.nonphysical(), s.mood(with_mask=True)[1].reshape(3, -1).clone()))
        s.close()
    stream.synchronize()
    (d0, u0, b0, m0), (d1, u1, b1, m1) = out
    assert b0 == 0 and bool(torch.isfinite(u0).all())
    hit = [2] if cell else range(len(lens))
    if cell:
        assert [t for t in range(len(lens)) if math.isnan(d1[t])] == [2]
    cells = torch.zeros(int(off[-1]), dtype=torch.bool, device="cuda")
    faces = cells.clone()
    for t in hit:
        cells[int(off[t]) + 3:int(off[t + 1]) - 3] = True
        faces[int(off[t]) + 2:int(off[t + 1]) - 3] = True
    assert bool(torch.isnan(u1[:, cells]).all()) and torch.equal(u0[:, ~cells], u1[:, ~cells])
    assert b1 == sum(lens[t] for t in hit)
    # the states of the later stages are not numbers: both sides take the last resort
    assert bool((m1[1:, faces] == (10 if mood else 0)).all()) and torch.equal(m0[:, ~faces], m1[:, ~faces])
