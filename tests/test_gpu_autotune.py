"""ws_autotune times its candidates on faces that are evaluated, also when the
state it is given is still at rest nearly everywhere, as an initial state is:
tuning takes as long as on a state that moves everywhere."""
import time

import pytest

from paper_1707_00592_gb300 import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

import paper_1707_00592_gb300 as ws  # noqa: E402


def seconds(s, U):
    best = 1e9
    for _ in range(3):
        torch.cuda.synchronize()
        t = time.perf_counter()
        ws.ws_autotune(s.ctx, U, 10)
        torch.cuda.synchronize()
        best = min(best, time.perf_counter() - t)
    return best


def test_candidates_work():
    G, P = wl.material(*wl.AIR)
    s = ws.Solver(2, (3000, 1000), (1e-3, 1e-3), precision="mixed")
    rest = s.tensor()
    for f, v in zip((0, 3, 4, 5), (1.2, 1e5 * G + P, G, P)):
        rest[f] = v
    g = torch.Generator(device="cuda")
    g.manual_seed(1)
    moving = rest * (1.0 + 1e-4 * torch.rand(rest.shape, generator=g, device="cuda", dtype=torch.float64))
    # (at rest a face takes the linear weights, which cost less than WENO-IS)
    assert seconds(s, rest) > 0.6 * seconds(s, moving)
