"""xtrg_tc_gemm from many host threads: no page-locked memory per thread, and
more calls at a time than there are page-locked words for their error flags."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# counts the page-locked allocations and frees of the process
COUNTER = r"""
#include <dlfcn.h>
#include <stddef.h>
static int allocs, frees;
static void* real(const char* name) { return dlsym(dlopen("libcudart.so.13", RTLD_LAZY | RTLD_NOLOAD), name); }
extern "C" int cudaHostAlloc(void** p, size_t n, unsigned f) {
  __atomic_add_fetch(&allocs, 1, __ATOMIC_RELAXED);
  return ((int (*)(void**, size_t, unsigned))real("cudaHostAlloc"))(p, n, f);
}
extern "C" int cudaFreeHost(void* p) {
  __atomic_add_fetch(&frees, 1, __ATOMIC_RELAXED);
  return ((int (*)(void*))real("cudaFreeHost"))(p);
}
extern "C" int pinned_allocs() { return allocs; }
extern "C" int pinned_frees() { return frees; }
"""

SETUP = r"""
import ctypes, sys, threading
sys.path.insert(0, ROOT)
import torch
from paper_1801_00142_gb300 import _lib

class Call:
    def __init__(self, seed, M, N, K):
        g = torch.Generator(device="cuda").manual_seed(seed)
        kw = dict(generator=g, device="cuda", dtype=torch.float64)
        self.size = (M, N, K)
        self.A, self.B = torch.randn(M, K, **kw), torch.randn(N, K, **kw)
        self.C = torch.zeros(M, N, device="cuda", dtype=torch.float64)
        self.n = _lib.xtrg_tc_gemm_workspace_bytes(M, N, K, 1, 3, 1)
        self.ws = torch.empty(self.n + 256, dtype=torch.uint8, device="cuda")
        self.stream = torch.cuda.Stream()
        self.want = self.A @ self.B.T
        self.bound = 2.0 ** -22 * (self.A.abs() @ self.B.abs().T)

    def run(self):
        M, N, K = self.size
        p = (self.ws.data_ptr() + 255) // 256 * 256
        _lib.xtrg_tc_gemm(self.A.data_ptr(), self.B.data_ptr(), self.C.data_ptr(), M, N, K, 1, 3, 6, 1,
                          p, self.n, self.stream.cuda_stream)

    def right(self):
        return bool(((self.C - self.want).abs() <= self.bound).all())

failed = []
def body(c, times, start=None):
    try:
        if start:
            start.wait()
        for _ in range(times):
            c.run()
    except Exception as e:
        failed.append(repr(e))
"""

THREADS = SETUP + r"""
calls = [Call(s, 60, 44, 52) for s in range(12)]
torch.cuda.synchronize()
lib = ctypes.CDLL(None)
before = lib.pinned_allocs(), lib.pinned_frees()
for c in calls:     # one short-lived thread after the other
    t = threading.Thread(target=body, args=(c, 1))
    t.start()
    t.join()
after = lib.pinned_allocs(), lib.pinned_frees()   # before torch takes any for its own reads
assert not failed and all(c.right() for c in calls), failed[:3]
print("allocs", after[0] - before[0], "frees", after[1] - before[1])
"""

MANY = SETUP + r"""
calls = [Call(s, 33 + s % 5, 20 + s % 7, 40) for s in range(80)]
torch.cuda.synchronize()
start = threading.Barrier(80)
ts = [threading.Thread(target=body, args=(c, 20, start)) for c in calls]
for t in ts:
    t.start()
for t in ts:
    t.join()
torch.cuda.synchronize()
assert not failed and all(c.right() for c in calls), failed[:3]
print("ok")
"""


def _run(script, **env):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1801_00142_gb300.build import build
    build()
    r = subprocess.run([sys.executable, "-c", f"ROOT = {ROOT!r}\n" + script], capture_output=True,
                       text=True, timeout=300, env={**os.environ, **env})
    assert r.returncode == 0, r.stderr[-2000:]
    return r.stdout.strip().splitlines()[-1]


def test_threads_take_no_pinned_memory_of_their_own(tmp_path):
    src, so = tmp_path / "count.cpp", tmp_path / "count.so"
    src.write_text(COUNTER)
    subprocess.run(["g++", "-shared", "-fPIC", "-O1", str(src), "-o", str(so), "-ldl"], check=True)
    assert _run(THREADS, LD_PRELOAD=str(so)) == "allocs 1 frees 0"


def test_more_calls_at_a_time_than_flag_words():
    assert _run(MANY) == "ok"
