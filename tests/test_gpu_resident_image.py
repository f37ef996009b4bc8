"""ws_set_resident keeps every cell's own image, also where cells of different
internal energy share one FP32 pressure: fluid at rest whose energies differ in
the last FP32 bit, then a wave through it, bit for bit as without the image."""
import numpy as np
import pytest

from paper_1707_00592_gb300 import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

import paper_1707_00592_gb300 as ws  # noqa: E402


def energies():
    """Two neighbouring FP32 energies of air at about 1e5 Pa with one pressure, whichever way 1 / Gamma is rounded."""
    r = np.float32(0.4)
    e = np.float32(250000.0)
    while True:
        f = np.nextafter(e, np.float32(np.inf))
        if all(e * q == f * q for q in (np.nextafter(r, np.float32(0)), r, np.nextafter(r, np.float32(1)))):
            return float(e), float(f)
        e = f


# config 8 and 10: rows of 32 x 7 tiles
@pytest.mark.parametrize("config", [None, 8, 10])
def test_image_of_quiet_tiles(config):
    # enough tiles for the short way of quiet ones; the last row of tiles is three cells high
    n, bc = (1027, 605), (("transmissive", "transmissive"), ("periodic", "periodic"))
    G, P = wl.material(*wl.AIR)
    lo, hi = energies()
    rng = np.random.default_rng(4)
    ny, nx = n[1] + 6, n[0] + 6
    U = np.zeros((6, 1, ny, nx))
    U[0], U[4], U[5] = 1.2, G, P
    U[3] = np.where(rng.random((1, ny, nx)) < 0.5, lo, hi)
    # heavy gas of high pressure up to four cells from the last tile but one, and weights and an epsilon
    # with which its disturbance is through that tile and the last one after two steps
    U[0, :, 3 + 500:3 + 592] = 120.0
    U[3, :, 3 + 500:3 + 592] = 100.0 * lo
    kw = dict(precision="mixed", weights="basic", eps=0.1)
    a, b = (ws.Solver(2, n, (1.0, 1e-3), bc, **kw) for _ in range(2))
    for s in (a, b):
        if config is not None:
            ws.ws_set_stage_config(s.ctx, config)
    ws.ws_set_resident(a.ctx, True)
    Ua, Ub = a.tensor(U), b.tensor(U)
    for _ in range(80):
        a.step(Ua)
        b.step(Ub)
        assert torch.equal(Ua[:, 0, 3:-3, 3:-3], Ub[:, 0, 3:-3, 3:-3])
    assert bool((Ua[3, 0, 3, 3:-3] > 1.1 * hi).all())  # the wave has crossed
