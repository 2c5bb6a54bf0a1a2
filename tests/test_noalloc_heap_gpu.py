"""The allocation-free call enters no heap allocator on a warm handle.

A child process preloads a counter of `operator new` calls made from
libmtgp.so.  After one call on a handle, calls of other sizes, which run with
other launch shapes, must count none, and an ordinary call after them shows
that the counter counts.
"""
import os
import shutil
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

COUNTER = r"""
#include <cstdlib>
#include <cstring>
#include <dlfcn.h>
#include <new>
static bool g_on;
static unsigned long long g_n;
extern "C" void counter_start() { g_n = 0; g_on = true; }
extern "C" unsigned long long counter_stop() { g_on = false; return g_n; }
static void* take(size_t n, void* from)
{
    Dl_info i;
    if (g_on && dladdr(from, &i) && i.dli_fname && strstr(i.dli_fname, "libmtgp.so"))
        ++g_n;
    void* p = malloc(n ? n : 1);
    if (!p)
        throw std::bad_alloc();
    return p;
}
void* operator new(size_t n) { return take(n, __builtin_return_address(0)); }
void* operator new[](size_t n) { return take(n, __builtin_return_address(0)); }
void operator delete(void* p) noexcept { free(p); }
void operator delete[](void* p) noexcept { free(p); }
void operator delete(void* p, size_t) noexcept { free(p); }
void operator delete[](void* p, size_t) noexcept { free(p); }
"""

CHILD = r"""
import ctypes, sys
import numpy as np
import torch
from paper_1501_07701_gb300 import mtgp, workloads
c = ctypes.CDLL(sys.argv[1])
c.counter_stop.restype = ctypes.c_ulonglong
sms = torch.cuda.get_device_properties(0).multi_processor_count
for mexp in (3217, 11213, 44497):
    p = mtgp.mtgp_params_generate(mexp, workloads.PARAM_SEED)
    n = 1024
    ids = np.arange(n, dtype=np.uint32)
    out = torch.empty(n * 64 + 10000, dtype=torch.int32, device="cuda")
    few = (ids[:16], np.full(16, 64, np.uint64))
    many = (ids, np.full(n, 64, np.uint64))
    uneven = (ids[:700], np.where(ids[:700] == 5, 9999, 8).astype(np.uint64))
    shared = (ids % 7, np.full(n, 40, np.uint64))
    other = mtgp.mtgp_init_statuses(p, ids)
    for i, k in (few, many, uneven, shared):     # the process has launched every kernel once
        mtgp.mtgp_generate_noalloc(other, i, k, mtgp.MTGP_U32, out)
    torch.cuda.synchronize()
    st = mtgp.mtgp_init_statuses(p, ids)
    mtgp.mtgp_generate_noalloc(st, *few, mtgp.MTGP_U32, out)
    c.counter_start()
    for i, k in (many, uneven, shared, few):
        mtgp.mtgp_generate_noalloc(st, i, k, mtgp.MTGP_U32, out)
    print("noalloc", mexp, c.counter_stop())
    c.counter_start()
    mtgp.mtgp_generate_u32(st, *many, out)
    print("ordinary", mexp, c.counter_stop())
    torch.cuda.synchronize()
    mtgp.mtgp_check(st)
"""


def test_no_heap_allocation_when_the_launch_shape_changes(tmp_path):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no C++ compiler")
    from paper_1501_07701_gb300 import build
    build.build()
    (tmp_path / "c.cpp").write_text(COUNTER)
    so = str(tmp_path / "counter.so")
    subprocess.run([cxx, "-O1", "-shared", "-fPIC", "-o", so, str(tmp_path / "c.cpp"), "-ldl"], check=True)
    r = subprocess.run([sys.executable, "-c", CHILD, so], cwd=ROOT, capture_output=True, text=True, timeout=300,
                       env=dict(os.environ, LD_PRELOAD=so))
    assert r.returncode == 0, r.stderr[-3000:]
    counts = {tuple(line.split()[:2]): int(line.split()[2]) for line in r.stdout.splitlines() if line}
    assert len(counts) == 6
    for (what, mexp), n in counts.items():
        assert n > 0 if what == "ordinary" else n == 0, counts
