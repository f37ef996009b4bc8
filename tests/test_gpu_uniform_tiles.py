"""Tiles of one state take a short way through the fused stages: same states,
time steps and MOOD records, bit for bit, as the census step, which always
evaluates every face."""
import numpy as np
import pytest

from paper_1707_00592_gb300 import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

import paper_1707_00592_gb300 as ws  # noqa: E402

WALLS = ("reflective", "reflective")
OPEN = ("transmissive", "transmissive")
RING = ("periodic", "periodic")


def state(ndim, n, velocity):
    """Air moving with `velocity`, a water block in one corner of it and a
    single cell of higher pressure: tiles of one state, of two, and nearly of one."""
    case = wl.random_state(ndim, n, seed=1, kind="smooth")
    Q = case.Q
    Ga, Pa = wl.material(*wl.AIR)
    Gw, Pw = wl.material(*wl.WATER)
    sl = wl.interior(ndim, case.n)
    Q[sl] = 0.0
    vals = [1.2, *velocity[:ndim], 1e5, Ga, Pa]
    for f, v in enumerate(vals):
        Q[(f,) + sl[1:]] = v
    # periodic axes that end in a tile of 1 to 4 cells among the sizes below
    block = (slice(None),) + tuple(slice(3, 3 + max(1, int(n[d]) // 3)) if d < ndim else slice(None) for d in (2, 1, 0))
    for f, v in zip((0, ndim + 2, ndim + 3), (1000.0, Gw, Pw)):
        Q[(f,) + block[1:]] = v
    cell = tuple(3 + int(n[d]) - 5 if d < ndim else 0 for d in (2, 1, 0))
    Q[(ndim + 1,) + cell] *= 1.0 + 1e-6
    return case


@pytest.mark.parametrize("ndim,n,bc", [(2, (1027, 601), (OPEN, OPEN)), (2, (964, 631), (RING, WALLS)),
                                       (2, (1300, 512), (WALLS, RING)), (2, (70, 47), (WALLS, OPEN)),
                                       (3, (70, 41, 37), (RING, WALLS, OPEN))])
@pytest.mark.parametrize("velocity", [(0.0, 0.0, 0.0), (30.0, -20.0, 10.0)])
@pytest.mark.parametrize("mood", [True, False])
def test_equals_every_face_evaluated(ndim, n, bc, velocity, mood):
    case = state(ndim, n, velocity)
    sl = wl.interior(ndim, case.n)
    for cfg in range(0, 16 if ndim == 2 else 8, 2 if mood else 5):
        kw = dict(precision="mixed", mood=mood)
        a, b = ws.Solver(ndim, case.n, case.dx, bc, **kw), ws.Solver(ndim, case.n, case.dx, bc, **kw)
        for s in (a, b):
            ws.ws_set_stage_config(s.ctx, cfg)
        ws.ws_set_resident(a.ctx, cfg % 3 == 0)
        Ua = a.prim_to_cons(a.tensor(case.Q))
        Ub = b.prim_to_cons(b.tensor(case.Q))
        for _ in range(4):
            dt = a.step(Ua, want_dt=True)
            assert dt == b.census_step(Ub)["dt"]
            assert np.array_equal(Ua.cpu().numpy()[sl], Ub.cpu().numpy()[sl])
            assert a.nonphysical() == b.nonphysical()
            (ca, ma), (cb, mb) = a.mood(with_mask=True), b.mood(with_mask=True)
            assert np.array_equal(ca, cb) and bool((ma == mb).all())
        a.close()
        b.close()
