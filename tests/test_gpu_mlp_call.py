"""A gradient call starts from zero sums, whatever an earlier call left: one
whose last launch never ran here."""
import ctypes

import numpy as np
import pytest

from oracle import mlp_oracle as mo

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

import paper_1707_00592_gb300 as ws  # noqa: E402


def test_after_an_unfinished_call():
    rt = ctypes.CDLL("libcudart.so.13")
    rng = np.random.default_rng(2)
    n = 1000
    P, X = (torch.tensor(a, dtype=torch.float32, device="cuda") for a in (mo.init(3), rng.normal(size=(n, mo.NIN))))
    y = torch.tensor((rng.random(n) < 0.3).astype(np.uint8), device="cuda")
    g, loss = torch.empty(mo.NPARAM, device="cuda"), torch.empty(1, device="cuda")

    def call(stream=None):
        ws.ws_mlp_grad(P, X, y, 3.0, g, loss, stream)

    call()
    want = g.cpu().numpy().copy(), loss.item()
    # the same call as a graph without its last launch
    stream = torch.cuda.Stream()
    graph, ex, count = ctypes.c_void_p(), ctypes.c_void_p(), ctypes.c_size_t()
    torch.cuda.synchronize()
    assert rt.cudaStreamBeginCapture(ctypes.c_void_p(stream.cuda_stream), 2) == 0
    call(stream)
    assert rt.cudaStreamEndCapture(ctypes.c_void_p(stream.cuda_stream), ctypes.byref(graph)) == 0
    assert rt.cudaGraphGetNodes(graph, None, ctypes.byref(count)) == 0
    nodes = (ctypes.c_void_p * count.value)()
    assert rt.cudaGraphGetNodes(graph, nodes, ctypes.byref(count)) == 0
    last = []
    for node in nodes:
        k = ctypes.c_size_t()
        assert rt.cudaGraphNodeGetDependentNodes(ctypes.c_void_p(node), None, None, ctypes.byref(k)) == 0
        if k.value == 0:
            last.append(node)
    assert len(last) == 1 and count.value > 1
    assert rt.cudaGraphDestroyNode(ctypes.c_void_p(last[0])) == 0
    assert rt.cudaGraphInstantiate(ctypes.byref(ex), graph, ctypes.c_ulonglong(0)) == 0
    assert rt.cudaGraphLaunch(ex, ctypes.c_void_p(stream.cuda_stream)) == 0
    torch.cuda.synchronize()
    call()
    torch.cuda.synchronize()
    got = g.cpu().numpy(), loss.item()
    assert rt.cudaGraphExecDestroy(ex) == 0 and rt.cudaGraphDestroy(graph) == 0
    assert np.array_equal(got[0], want[0]) and got[1] == want[1]
