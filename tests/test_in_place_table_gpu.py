"""Which direct calls read their work table in host memory.

A call is recorded into a CUDA graph and the graph's copy nodes are counted:
none where the kernel reads the table in place (few requests per stream), one
where it is copied first (long request lists, whose rows walk the list with
dependent reads).  The numbers of both are compared with the oracle.  A child
process does it: the recorded handles' events stay unusable.
"""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r"""
import ctypes
import numpy as np
import torch
import oracle
from paper_1501_07701_gb300 import mtgp, workloads
torch.cuda.init()
torch.zeros(1, device="cuda")
rt = ctypes.CDLL("libcudart.so.13")
p, op = mtgp.mtgp_params_generate(11213, workloads.PARAM_SEED), oracle.params_generate(11213, workloads.PARAM_SEED)
seeds = np.arange(128, dtype=np.uint32)
kept = []   # not freed: their events were recorded into a graph

def call(st, ids, counts, out, s):
    mtgp.mtgp_generate_u32(st, ids, counts, out, s)

def copies(ids, counts):
    st = mtgp.mtgp_init_statuses(p, seeds)
    kept.append(st)
    out = torch.empty(int(counts.sum()), dtype=torch.int32, device="cuda")
    s = torch.cuda.Stream()
    for _ in range(4):                      # the handle's table buffers exist
        call(st, ids, counts, out, s)
    s.synchronize()
    states = np.stack([oracle.init_state(op, int(x)) for x in seeds])
    for _ in range(4):
        ref = []
        for i, k in zip(ids, counts):
            o, states[i] = oracle.generate(op, states[i], int(k), oracle.U32)
            ref.append(o)
    assert np.array_equal(out.cpu().numpy().view(np.uint32), np.concatenate(ref))
    h, g, n = ctypes.c_void_p(s.cuda_stream), ctypes.c_void_p(), ctypes.c_size_t()
    assert rt.cudaStreamBeginCapture(h, 2) == 0          # relaxed
    call(st, ids, counts, out, s)
    assert rt.cudaStreamEndCapture(h, ctypes.byref(g)) == 0
    assert rt.cudaGraphGetNodes(g, None, ctypes.byref(n)) == 0
    nodes = (ctypes.c_void_p * n.value)()
    assert rt.cudaGraphGetNodes(g, nodes, ctypes.byref(n)) == 0
    types = []
    for x in nodes:
        t = ctypes.c_int()
        assert rt.cudaGraphNodeGetType(ctypes.c_void_p(x), ctypes.byref(t)) == 0
        types.append(t.value)
    assert types.count(0) == 1                           # one kernel
    return types.count(1)                                # copies

for n, per in ((1, 1), (100, 1), (200, 4), (5, 5), (16, 16), (300, 300)):
    print(n, per, copies((np.arange(n) // per).astype(np.uint32), np.full(n, 40, np.uint64)))
"""


def test_long_request_lists_are_copied():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1501_07701_gb300 import build
    build.build()
    r = subprocess.run([sys.executable, "-c", CHILD], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-3000:]
    got = {tuple(map(int, line.split()[:2])): int(line.split()[2]) for line in r.stdout.splitlines() if line}
    assert got == {(1, 1): 0, (100, 1): 0, (200, 4): 0, (5, 5): 1, (16, 16): 1, (300, 300): 1}
