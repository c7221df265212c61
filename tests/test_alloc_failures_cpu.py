"""A one-call proof gives everything back when a host allocation fails in it.

A child process preloads an `operator new` that counts live blocks and fails its
n-th call on request.  For every n that the call reaches, `vl_prove_batch` and
`vl_prove_matmul_noalloc` return (VL_ENOMEM, or whatever the call ends with where
the library does without the block), and no block is left behind: the plan that
the call made for itself goes with it.  No GPU is needed: the descriptor tables
are packed before the first copy, which is where the call then ends.
"""
import os
import shutil
import subprocess
import sys

import pytest

from paper_2508_21393_gb300 import binding as B

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PRELOAD = r"""
#include <stdlib.h>
#include <atomic>
#include <new>
static std::atomic<long> live{0}, count{0}, fail_at{0};
extern "C" long alloc_live() { return live; }
extern "C" long alloc_count() { return count; }
extern "C" void alloc_arm(long n) { count = 0; fail_at = n; }
static void* take(size_t n, size_t align) {
  if (++count == fail_at) return nullptr;
  void* p = align > 16 ? aligned_alloc(align, (n + align - 1) / align * align) : malloc(n ? n : 1);
  if (p) live++;
  return p;
}
static void give(void* p) { if (p) { live--; free(p); } }
static void* must(void* p) { if (!p) throw std::bad_alloc(); return p; }
void* operator new(size_t n) { return must(take(n, 0)); }
void* operator new[](size_t n) { return must(take(n, 0)); }
void* operator new(size_t n, std::align_val_t a) { return must(take(n, (size_t)a)); }
void* operator new(size_t n, const std::nothrow_t&) noexcept { return take(n, 0); }
void operator delete(void* p) noexcept { give(p); }
void operator delete[](void* p) noexcept { give(p); }
void operator delete(void* p, size_t) noexcept { give(p); }
void operator delete(void* p, std::align_val_t) noexcept { give(p); }
void operator delete(void* p, size_t, std::align_val_t) noexcept { give(p); }
void operator delete(void* p, const std::nothrow_t&) noexcept { give(p); }
"""

CHILD = r"""
import ctypes, sys
sys.path.insert(0, sys.argv[1])
import numpy as np
from paper_2508_21393_gb300 import binding as B
L, A = B.lib(), ctypes.CDLL(None)
A.alloc_live.restype = A.alloc_count.restype = ctypes.c_long
A.alloc_arm.argtypes = [ctypes.c_long]
P, Q = np.zeros((5, 7), np.int16), np.zeros((7, 3), np.int16)
space = B.VL_HOST if sys.argv[2] == "batch" else B.VL_DEVICE
fake = lambda M: B.vl_mat(M.ctypes.data, M.shape[0], M.shape[1], M.shape[1], B.VL_I16, 0, space, 0)
job = B.vl_job()
job.P, job.Q = fake(P), fake(Q)
jobs = (B.vl_job * 3)(job, job, job)
out = (B.vl_proof * 3)()
ws = ctypes.create_string_buffer(32 << 20)
at = (ctypes.addressof(ws) + 255) // 256 * 256
def call():
    if sys.argv[2] == "batch":
        return L.vl_prove_batch(jobs, 3, ctypes.c_void_p(at), ctypes.c_size_t(16 << 20), out, B.VL_HOST, None, None)
    return L.vl_prove_matmul_noalloc(ctypes.byref(job.P), ctypes.byref(job.Q), ctypes.byref(job.fs), out, None)
last = call()  # first-use state of the library and the runtime
A.alloc_arm(0)
before = A.alloc_live()
assert call() == last and A.alloc_live() == before
total = A.alloc_count()
codes = set()
for n in range(1, total + 1):
    A.alloc_arm(n)
    code = call()
    A.alloc_arm(0)
    codes.add(code)
    assert A.alloc_live() == before, (n, total, code, A.alloc_live() - before)
print(total, last, sorted(codes))
"""


@pytest.mark.skipif(not sys.platform.startswith("linux") or shutil.which("g++") is None, reason="needs g++, LD_PRELOAD")
@pytest.mark.parametrize("entry", ["batch", "noalloc"])
def test_failed_allocation_leaves_nothing_behind(tmp_path, entry):
    if not os.path.exists(B.LIB_PATH):
        from paper_2508_21393_gb300 import build
        build.build(quiet=True)
    src, lib = tmp_path / "count.cpp", tmp_path / "libcount.so"
    src.write_text(PRELOAD)
    subprocess.run(["g++", "-std=c++17", "-O1", "-w", "-shared", "-fPIC", str(src), "-o", str(lib)], check=True)
    env = dict(os.environ, LD_PRELOAD=str(lib), CUDA_VISIBLE_DEVICES="")
    res = subprocess.run([sys.executable, "-c", CHILD, ROOT, entry], env=env, capture_output=True, text=True, timeout=300)
    assert res.returncode == 0, res.stderr[-2000:]
    total, last, codes = res.stdout.strip().split(" ", 2)
    assert int(total) > 10 and str(B.VL_ENOMEM) in codes, res.stdout
