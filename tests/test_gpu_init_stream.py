"""A context on a stream that does not wait for the legacy default stream, which
is busy: what ws_init sets is set before the first step, and not after it."""
import numpy as np
import pytest

import oracle
from paper_1707_00592_gb300 import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

import paper_1707_00592_gb300 as ws  # noqa: E402


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_busy_default_stream(precision):
    ndim, n = 2, (40, 35)
    case = wl.random_state(ndim, n, seed=12, kind="two_phase")
    Uo = oracle.prim_to_cons(ndim, case.Q)
    warm = ws.Solver(ndim, case.n, case.dx, case.bc, precision=precision)  # loads the library and its kernels
    U, V = warm.tensor(Uo), warm.tensor(Uo)
    dto = warm.step(V, want_dt=True)
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    torch.cuda._sleep(int(4e8))  # 0.2 s of the default stream
    s = ws.Solver(ndim, case.n, case.dx, case.bc, precision=precision, stream=side)
    dt = s.step(U, want_dt=True)
    torch.cuda.synchronize()
    sl = wl.interior(ndim, case.n)
    assert dt == dto and torch.equal(U[sl], V[sl])
    with torch.cuda.stream(side):
        counts, mask = s.mood(with_mask=True)
    side.synchronize()
    want_counts, want = warm.mood(with_mask=True)
    assert int(want.sum()) > 0 and torch.equal(mask, want) and np.array_equal(counts, want_counts)


def test_busy_default_stream_tubes():
    off = np.array([0, 300, 1300, 1700], dtype=np.int64)
    G, P = wl.material(*wl.AIR)
    out = []
    side = torch.cuda.Stream()
    for busy in (False, True):
        U = torch.zeros((5, 1700), dtype=torch.float64, device="cuda")
        for f, v in zip((0, 2, 3, 4), (1.2, 1e5 * G + P, G, P)):
            U[f] = v
        U[2, 700:] *= 1.5
        torch.cuda.synchronize()
        if busy:
            torch.cuda._sleep(int(4e8))
        s = ws.Solver(1, (1,), (1.0,), tube_offsets=off, precision="mixed", stream=side)
        dt = s.step(U, want_dt=True)
        torch.cuda.synchronize()
        with torch.cuda.stream(side):
            _, mask = s.mood(with_mask=True)
        side.synchronize()
        out.append((dt, U, mask))
    assert np.array_equal(out[0][0], out[1][0])
    assert torch.equal(out[0][1], out[1][1]) and torch.equal(out[0][2], out[1][2])
