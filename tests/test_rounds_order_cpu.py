"""The rounds of a proof do not depend on when each warp runs.

rounds_dev.cuh runs on the CPU, one fibre per CUDA thread (tests/emulator), under
orders that keep some warps back as long as its barriers allow: the look-ahead
warps, the hash and its schedules, each single warp, seeded shuffles.  Whatever
the order, the proof equals the oracle's byte for byte.  (On a GPU the warps take
turns every few cycles, so a missing barrier between steps that are microseconds
apart does not show there.)
"""
import ctypes
import os
import random
import shutil
import subprocess

import numpy as np
import pytest

import oracle
from paper_2508_21393_gb300 import binding as B

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2508_21393_gb300", "csrc")
CUDA = os.environ.get("CUDA_HOME", "/usr/local/cuda")

# Barrier and cluster instructions -> the emulator's calls.
REPLACED = {
    "transcript_dev.cuh": [
        ('asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");', "emu::bar_sync(id, threads);"),
        ('asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(threads) : "memory");', "emu::bar_arrive(id, threads);"),
    ],
    "rounds_dev.cuh": [
        ('asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(x));', "x = emu::cluster_rank();"),
        ('asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(x));', "x = emu::cluster_size();"),
        ('asm volatile("barrier.cluster.arrive.release.aligned;\\n\\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");',
         "emu::cluster_sync();"),
        ('asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : '
         '"r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank));', "a = 0;"),
        ('asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory");',
         "(void)a; emu::st_cluster(p, rank, v);"),
    ],
}


@pytest.fixture(scope="module")
def emulated(tmp_path_factory):
    if shutil.which("g++") is None or not os.path.exists(os.path.join(CUDA, "include", "cuda_runtime.h")):
        pytest.skip("needs g++ and the CUDA headers")
    src = tmp_path_factory.mktemp("rounds")
    for name in os.listdir(CSRC):
        if not name.endswith((".cuh", ".h")):
            continue
        with open(os.path.join(CSRC, name)) as f:
            text = f.read()
        for old, new in REPLACED.get(name, []):
            assert text.count(old) == 1, (name, old)
            text = text.replace(old, new)
        if name == "rounds_dev.cuh":
            text = text.replace("namespace vl {", "namespace emu {\nvoid st_cluster(const void*, uint32_t, uint32_t);\n}\n"
                                                  "namespace vl {", 1)
        with open(src / name, "w") as f:
            f.write(text)
    lib = str(src / "librounds.so")
    here = os.path.join(ROOT, "tests", "emulator")
    subprocess.run(["g++", "-std=c++17", "-O1", "-w", "-shared", "-fPIC", "-I", str(src), "-I", here,
                    "-I", os.path.join(ROOT, "include"), "-I", os.path.join(CUDA, "include"),
                    os.path.join(here, "rounds.cpp"), "-o", lib], check=True)
    return ctypes.CDLL(lib)


def _orders(warps, ctas):
    """Orders of one block's warps, the last to run last; blocks forward and backward."""
    look = [w for w in range(warps) if w & 2 and w != 2]
    rest = [w for w in range(warps) if w not in look]
    one = [list(range(warps)), list(range(warps))[::-1], rest + look, look + rest, rest[::-1] + look[::-1]]
    one += [[v for v in range(warps) if v != w] + [w] for w in (0, 1, 2, warps - 1)]
    rng = random.Random(warps)
    one += [rng.sample(range(warps), warps) for _ in range(2)]
    for o in one:
        yield [c * warps + w for c in range(ctas) for w in o]
        if ctas > 1:
            yield [c * warps + w for c in reversed(range(ctas)) for w in o]


@pytest.mark.parametrize("k,ctas,threads", [(1, 1, 128), (2, 1, 256), (3, 1, 256), (13, 1, 128), (13, 1, 512),
                                            (70, 1, 256), (300, 1, 128), (300, 1, 256), (600, 2, 256)])
def test_any_order_of_the_warps_gives_the_same_proof(emulated, k, ctas, threads):
    rng = np.random.default_rng(k)
    P = rng.integers(-(1 << 15), 1 << 15, size=(1, k)).astype(np.int16)
    Q = rng.integers(-(1 << 15), 1 << 15, size=(k, 1)).astype(np.int16)
    want = oracle.prove_matmul(P, Q, seed=5)
    T = oracle.Transcript(5, 1, k, 1, 0, 0)
    T.squeeze(b"u", 0)
    T.squeeze(b"v", 0)
    a, b = (np.ascontiguousarray(x.reshape(-1)).ctypes.data_as(ctypes.c_void_p) for x in (P, Q))
    for order in _orders(threads // 32, ctas):
        out = B.vl_proof()
        o = (ctypes.c_int * len(order))(*order)
        assert emulated.emu_rounds(k, a, b, T.state, ctas, threads, int(threads >= 256), o, ctypes.byref(out)) == 1
        assert B.proof_bytes(out) == want.to_bytes(), order
