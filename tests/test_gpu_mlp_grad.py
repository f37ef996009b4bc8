"""Edges of the gate's gradient kernel against the FP64 back-propagation: tiles
of 128 samples and their remainders, and contributions too large for the
two-part 32-bit sums."""
import numpy as np
import pytest

from oracle import mlp_oracle as mo

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

import paper_1707_00592_gb300 as ws  # noqa: E402


@pytest.mark.parametrize("n", [1, 127, 128, 129, 300, 40000])
@pytest.mark.parametrize("scale", [1.0, 40.0])  # 40: contributions above 2^-3 also at n = 300
def test_gradient(n, scale):
    rng = np.random.default_rng(n)
    p = mo.init(3).astype(np.float32)
    X = (scale * rng.normal(size=(n, mo.NIN))).astype(np.float32)
    y = (rng.random(n) < 0.3).astype(np.uint8)
    P, Xd, yd = (torch.tensor(a, device="cuda") for a in (p, X, y))
    g = torch.empty(mo.NPARAM, dtype=torch.float32, device="cuda")
    loss = torch.empty(1, dtype=torch.float32, device="cuda")
    got = []
    for _ in range(2):  # the sums start from zero every time
        ws.ws_mlp_grad(P, Xd, yd, 3.0, g, loss)
        torch.cuda.synchronize()
        got.append((g.cpu().numpy().copy(), loss.item()))
    assert np.array_equal(got[0][0], got[1][0]) and got[0][1] == got[1][1]
    g64 = mo.grad(p.astype(np.float64), X.astype(np.float64), y, 3.0)
    assert np.abs(got[0][0] - g64).max() <= 2e-4 * np.abs(g64).max()
