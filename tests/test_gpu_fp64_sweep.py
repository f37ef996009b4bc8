"""The FP64 sweep at its edges, bit for bit against the oracle: chunks of 16
faces, the switch to many chunks per CTA with products on the integer pipe,
epsilons that take the literal evaluation, and magnitudes outside the integer
operations' range."""
import numpy as np
import pytest

import oracle
from paper_1707_00592_gb300 import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

import paper_1707_00592_gb300 as ws  # noqa: E402


def same(a, b):
    return bool(np.all((a == b) | (np.isnan(a) & np.isnan(b))))


def check(case, Uo, steps=1, eps=None, mood=True, weights="modified", fixed_dt=0.0):
    kw = {} if eps is None else {"eps": eps}
    s = ws.Solver(case.ndim, case.n, case.dx, case.bc, mood=mood, weights=weights, **kw)
    g = oracle.Grid(case.ndim, case.n, case.dx, case.bc, mood=mood, weights=weights, **kw)
    sl = wl.interior(case.ndim, case.n)
    U = s.tensor(Uo)
    L = s.flux_divergence(U).cpu().numpy()
    Lo, mo = oracle.rhs(g, Uo)
    assert same(L[sl], Lo[sl])
    _, mask = s.mood(with_mask=True)
    assert same(mask.cpu().numpy()[:s.nmask], np.concatenate([m.ravel() for m in mo]))
    U = s.tensor(Uo)
    for _ in range(steps):
        dt = s.step(U, fixed_dt, want_dt=True)
        Uo, dto = oracle.step(g, Uo, fixed_dt)[:2]
        assert dt == dto
    assert same(U.cpu().numpy()[sl], Uo[sl])


@pytest.mark.parametrize("n", [14, 15, 16, 31, 95, 96])
@pytest.mark.parametrize("weights", ["modified", "js"])
def test_chunk_edges(n, weights):
    case = wl.random_state(1, (n,), seed=n, kind="two_phase")
    check(case, oracle.prim_to_cons(1, case.Q), steps=3, weights=weights)


# about 300 CTAs of all chunks is where the launch changes
@pytest.mark.parametrize("ndim,n", [(1, (24239,)), (1, (24400,)), (2, (113, 127)), (2, (150, 110)), (3, (22, 21, 20)),
                                    (3, (24, 23, 22))])
@pytest.mark.parametrize("weights", ["modified", "basic", "js"])
@pytest.mark.parametrize("mood", [True, False])
def test_launch_sizes(ndim, n, weights, mood):
    case = wl.random_state(ndim, n, seed=11, kind="two_phase")
    check(case, oracle.prim_to_cons(ndim, case.Q), steps=2, mood=mood, weights=weights)


@pytest.mark.parametrize("eps", [1e-49, 1e-51, 1e-200, 1e-300, 1e49, 1e60])
@pytest.mark.parametrize("n", [(40, 35), (150, 110)])
def test_epsilons(eps, n):
    case = wl.random_state(2, n, seed=13, kind="shock")
    check(case, oracle.prim_to_cons(2, case.Q), eps=eps)


# velocities that die out towards zero, as ahead of a wave; states scaled to
# both ends of the range; one cell that is not a number
@pytest.mark.parametrize("what", ["fade", "tiny", "huge", "nan", "inf", "rest"])
@pytest.mark.parametrize("n", [(40, 35), (150, 110)])
@pytest.mark.parametrize("weights", ["modified", "js"])
def test_magnitudes(what, n, weights):
    case = wl.random_state(2, n, seed=17, kind="smooth")
    Q = case.Q.copy()
    x = np.arange(Q.shape[3])[None, None, :] / Q.shape[3]
    if what == "fade":
        Q[1] *= 10.0 ** (-320.0 * x)
        Q[2] *= 10.0 ** (-100.0 * x)
    elif what == "rest":
        Q[1] = Q[2] = 0.0
        Q[3] = 1.0
    elif what == "tiny":
        Q[3] *= 1e-120
        Q[1] *= 1e-60
        Q[2] *= 1e-60
    elif what == "huge":
        Q[3] *= 1e120
        Q[1] *= 1e60
        Q[2] *= 1e60
    U = oracle.prim_to_cons(2, Q)
    fixed_dt = 0.0
    if what in ("nan", "inf"):
        U[4, 0, 20, 20] = float(what)
        fixed_dt = 1e-4  # the solver's CFL step is then NaN, the oracle's maximum passes over the cell
    check(case, U, weights=weights, fixed_dt=fixed_dt)
