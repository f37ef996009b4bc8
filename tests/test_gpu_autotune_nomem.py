"""Tuning batched tubes while device memory runs out: the call fails, and the
context steps on as before, its graph included.  The allocations fail on the
host, in a stand-in for cudaMalloc that the child process preloads."""
import os
import subprocess
import sys

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

FAKE = r"""
#define _GNU_SOURCE
#include <dlfcn.h>
#include <stddef.h>
static int left = 0;
void fail_call(int k) { left = k; }  /* the k-th call from now on fails; 0: none */
int calls_left(void) { return left; }
int cudaMalloc(void **p, size_t n) {
  static int (*real)(void **, size_t);
  if (!real) real = (int (*)(void **, size_t))dlsym(RTLD_NEXT, "cudaMalloc");
  if (left > 0 && --left == 0) return 2; /* cudaErrorMemoryAllocation */
  return real(p, n);
}
"""

CHILD = r"""
import ctypes, sys
sys.path.insert(0, sys.argv[1])
import numpy as np, torch
import paper_1707_00592_gb300 as ws
from paper_1707_00592_gb300 import workloads as wl
fake = ctypes.CDLL(sys.argv[2])
off, Q = wl.riemann_tubes(40, 100, 900, 0)
stream = torch.cuda.Stream()
with torch.cuda.stream(stream):
    a, b = (ws.Solver(1, (1,), (1.0,), tube_offsets=off, precision="mixed", stream=stream) for _ in range(2))
    Ua, Ub = a.prim_to_cons(a.tensor(Q)), b.prim_to_cons(b.tensor(Q))
    ws.ws_set_graph(a.ctx, True)
    failed = 0
    for k in range(1, 20):
        a.step(Ua)
        b.step(Ub)
        fake.fail_call(k)
        try:
            ws.ws_autotune(a.ctx, Ua, 1)
        except ws.WsError as e:
            failed += 1
            assert "cudaMalloc" in str(e), e
        used = fake.calls_left() == 0
        fake.fail_call(0)
        for _ in range(2):
            a.step(Ua)
            b.step(Ub)
            assert torch.equal(Ua, Ub) and a.nonphysical() == b.nonphysical(), k
        if not used:
            break
    assert failed == k - 1 and failed > 5, (failed, k)
torch.cuda.synchronize()
print("ok")
"""


def test_context_survives(tmp_path):
    src, lib, child = (str(tmp_path / n) for n in ("fake.c", "fake.so", "child.py"))
    open(src, "w").write(FAKE)
    open(child, "w").write(CHILD)
    subprocess.check_call(["gcc", "-shared", "-fPIC", "-o", lib, src, "-ldl"])
    r = subprocess.run([sys.executable, child, ROOT, lib], env={**os.environ, "LD_PRELOAD": lib}, capture_output=True,
                       text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout + r.stderr
