"""The device's field arithmetic against Python integers, operand by operand.

Proofs reach these functions with pseudo-random elements; here they get the
operands at which a carry, a conditional subtraction or a quotient estimate goes
the rare way: 0, 1, r - 1, limbs of all ones, multiples of r and their neighbours,
sums at the stated limits.  Every result is exact.
"""
import ctypes
import itertools
import os
import random
import subprocess

import numpy as np
import pytest

from paper_2508_21393_gb300 import build

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no GPU", allow_module_level=True)

R = 0x73eda753299d7d483339d80809a1d80553bda402fffe5bfeffffffff00000001
INV = pow(1 << 256, -1, R)
IN, OUT = 40, 20
RNG = random.Random(11)


def _limbs(*hot):
    return sum(0xffffffff << (32 * i) for i in hot)


# reduced elements
EL = sorted({x for x in [0, 1, 2, R - 1, R - 2, (R - 1) // 2, (R + 1) // 2, (1 << 256) % R, pow(1 << 256, 2, R), R - (1 << 32),
                         1 << 32, 1 << 254, (1 << 255) - (1 << 192)] + [_limbs(i) for i in range(7)]
             + [_limbs(*range(i)) for i in range(1, 8)] + [_limbs(0, 2, 4, 6), _limbs(1, 3, 5)] + [1 << (32 * i) for i in range(8)]
             + [RNG.randrange(R) for _ in range(12)] if x < R})
# any 256-bit value
ANY = EL + [R, R + 1, 2 * R - 1, 2 * R, 2 * R + 1, (1 << 256) - 1, (1 << 256) - (1 << 32), _limbs(7), _limbs(1, 3, 5, 7)]
PAIRS = list(itertools.product(EL, EL))


@pytest.fixture(scope="module")
def ops(tmp_path_factory):
    lib = str(tmp_path_factory.mktemp("field") / "libfield.so")
    here = os.path.dirname(os.path.abspath(__file__))
    subprocess.run([build.nvcc(), *build.ARCH, "-O3", "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "-I", build.CSRC, "-o", lib,
                    os.path.join(here, "field_ops.cu")], check=True)
    return ctypes.CDLL(lib)


def _run(ops, op, rows, words):
    """rows: per row a list of (value, words); the results as integers of `words` words."""
    data = bytearray()
    for row in rows:
        b = b"".join(v.to_bytes(4 * n, "little") for v, n in row)
        assert len(b) <= 4 * IN
        data += b.ljust(4 * IN, b"\0")
    a = np.frombuffer(bytes(data), dtype=np.uint32)
    out = np.zeros(len(rows) * OUT, dtype=np.uint32)
    assert ops.field_ops(op, a.ctypes.data_as(ctypes.c_void_p), out.ctypes.data_as(ctypes.c_void_p), len(rows)) == 0
    raw = out.tobytes()
    return [int.from_bytes(raw[4 * OUT * i:4 * OUT * i + 4 * words], "little") for i in range(len(rows))]


def test_add_sub_products(ops):
    assert _run(ops, 0, [[(a, 8), (b, 8)] for a, b in PAIRS], 8) == [(a + b) % R for a, b in PAIRS]
    assert _run(ops, 1, [[(a, 8), (b, 8)] for a, b in PAIRS], 8) == [(a - b) % R for a, b in PAIRS]
    wide = list(itertools.product(ANY, EL))  # the first factor need not be reduced
    assert _run(ops, 2, [[(a, 8), (b, 8)] for a, b in wide], 8) == [a * b * INV % R for a, b in wide]
    assert _run(ops, 3, [[(a, 8)] for a in ANY], 8) == [a * INV % R for a in ANY]


def test_inverse(ops):
    xs = EL + [1 << i for i in range(255) if 1 << i < R] + [R - (1 << i) for i in range(250)] + [RNG.randrange(R) for _ in range(500)]
    assert _run(ops, 14, [[(x, 8)] for x in xs], 8) == [pow(x, -1, R) if x else 0 for x in xs]


def test_column_sums(ops):
    top = (1 << 64) - 1
    rows = [[0] * 8, [top] * 7 + [(1 << 64) - (1 << 34)], [1] * 8, [0xffffffff] * 8, [1 << 32] * 8, [top, 0] * 4, [0, top] * 4]
    for i in range(8):
        rows += [[top if j == i else 0 for j in range(8)], [top if j <= i else 0 for j in range(8)]]
    for m in (1, 2, 3, (1 << 33) - 1):  # multiples of r and their neighbours
        rows += [[((m * R + d) >> (32 * j)) & 0xffffffff if j < 7 else (m * R + d) >> 224 for j in range(8)] for d in (-1, 0, 1)]
    rows += [[RNG.randrange(1 << RNG.randrange(1, 65)) for _ in range(8)] for _ in range(500)]
    rows = [r for r in rows if sum(c << (32 * j) for j, c in enumerate(r)) < 1 << 289 and max(r) <= top]
    value = [sum(c << (32 * j) for j, c in enumerate(r)) for r in rows]
    words = [[(c, 2) for c in r] for r in rows]
    assert _run(ops, 11, words, 10) == value
    assert _run(ops, 4, words, 8) == [v * INV % R for v in value]


def test_wide_sums(ops):
    full = 1 << 544
    acc = [0, 1, (1 << 512) - 1, (1 << 512), (1 << 256) - 1, full - 1 - R * R, R * R, (1 << 34) * R * R - R * R] + [
        RNG.randrange(1 << RNG.randrange(1, 543)) for _ in range(4)]
    rows = [(w, a, b) for w in acc for a, b in PAIRS[::7] if w + a * b < full]
    assert _run(ops, 5, [[(w, 17), (a, 8), (b, 8)] for w, a, b in rows], 17) == [w + a * b for w, a, b in rows]
    # nine limbs hold the reduced sum
    ws = [w for w in acc + [w + a * b for w, a, b in rows[::5]] if (w >> 256) + R < 1 << 288]
    got = _run(ops, 6, [[(w, 17)] for w in ws], 16)
    for w, g in zip(ws, got):
        v = sum(((g >> (64 * j)) & ((1 << 64) - 1)) << (32 * j) for j in range(8))
        assert v % R == w * INV % R and v <= (w >> 256) + R
    z9 = [0, 1, (1 << 278) - 1, (1 << 288) - 1, _limbs(8), _limbs(*range(8)), RNG.randrange(1 << 278)]
    rows = [(w, a, z) for w in acc for a in EL for z in z9 if w + a * z < full]
    assert _run(ops, 9, [[(w, 17), (a, 8), (z, 9)] for w, a, z in rows], 17) == [w + a * z for w, a, z in rows]
    ms = [0, 1, 2, 65535, 65534, 1 << 15, RNG.randrange(65536)]
    rows = [(w, a, b, m) for w in acc[:5] for a, b in PAIRS[::11] for m in ms if w + a * b * m < full]
    assert _run(ops, 10, [[(w, 17), (a, 8), (b, 8), (m, 1)] for w, a, b, m in rows], 17) == [w + a * b * m for w, a, b, m in rows]


def test_nine_limb_sums(ops):
    s = [0, 1, _limbs(*range(8)), (1 << 288) - 1 - R, RNG.randrange(1 << 280)]
    rows = [(x, a) for x in s for a in EL]
    assert _run(ops, 12, [[(x, 9), (a, 8)] for x, a in rows], 9) == [x + a for x, a in rows]
    rows = [(x, y) for x in s for y in s + EL if x + y < 1 << 288]
    assert _run(ops, 13, [[(x, 9), (y, 9)] for x, y in rows], 9) == [x + y for x, y in rows]


def test_reduction_by_a_quotient_estimate(ops):
    limit = 1 << 273
    qs = list(range(6)) + [limit // R - d for d in range(4)] + [1 << i for i in range(17)] + [RNG.randrange(limit // R) for _ in range(2000)]
    ts = [q * R + d for q in qs for d in (-2, -1, 0, 1, R - 1)]
    # the estimate reads the bits from 2^241 up: values just below the next step lose most
    ts += [(x << 241) - 1 for x in [1, 2, 3, (1 << 32) - 1, 1 << 32] + [RNG.randrange(1, 1 << 32) for _ in range(2000)]]
    ts += [limit - 1] + [RNG.randrange(limit) for _ in range(2000)]
    ts = [t for t in ts if 0 <= t < limit]
    assert _run(ops, 7, [[(t, 9)] for t in ts], 8) == [t % R for t in ts]
    rows = [(a, m) for a in EL for m in [0, 1, 2, 3, 65535, 65536, (1 << 18) - 1, RNG.randrange(1 << 18)]]
    assert _run(ops, 8, [[(a, 8), (m, 1)] for a, m in rows], 8) == [a * m % R for a, m in rows]
