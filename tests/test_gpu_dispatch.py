"""GPU parity at the edges of the kernels' dispatch rules: every proof equals
the oracle's byte for byte (integer work, no tolerance), or, for batches too
long for the oracle, the same statement proved alone.

The rules: matmul rounds on clusters of 8, 4 or 2 CTAs, or on 512, 256 or 128
threads, by the number of proofs, short rounds on four lanes per pair and vectors
of at most 256 entries in shared memory; batched claims' last rounds in one
cluster; CUDA-core fold tiles cut by the number of products; linear reductions
of at most 128 entries on register fragments (16-entry steps, 32-line tiles,
blocks of 256 to 1024 lines); lookup tails on clusters, 512 or 128 threads, each
from another round on, the table kernel's entries per thread.
"""
import numpy as np
import pytest

import oracle
from oracle import batch as OB
from oracle import lookup as OL
from paper_2508_21393_gb300 import binding as B

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no GPU", allow_module_level=True)


def _rand(rng, shape, lo=-(1 << 15), hi=1 << 15):
    return rng.integers(lo, hi, size=shape).astype(np.int16)


def _ws(n):
    return torch.empty(max(n, 256), dtype=torch.uint8, device="cuda")


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _prove(jobs, opts=None):
    n = B.vl_workspace_bytes(jobs, opts)
    ws = _ws(n)
    return [B.proof_bytes(p) for p in B.vl_prove_batch(jobs, ws.data_ptr(), n, opts=opts)]


@pytest.mark.parametrize("k", [1, 2, 3, 4, 5, 8, 9, 31, 32, 33, 64, 65, 128, 129, 256, 257, 512, 513, 1024, 1025, 2049, 4100,
                               8193])
def test_rounds_at_every_vector_length(k):
    rng = np.random.default_rng(k)
    P, Q = _rand(rng, (3, k)), _rand(rng, (k, 2))
    want = oracle.prove_matmul(P, Q, 0, 0, seed=k).to_bytes()
    job = B.job(_dev(P), _dev(Q), 0, 0, k)
    for variant, threads in ((0, 0), (4, 0), (7, 0), (0, 192), (0, 256), (8, 0)):
        o = B.vl_batch_opts()
        o.rounds_variant, o.rounds_threads = variant, threads
        assert _prove([job], o) == [want], (variant, threads)


@pytest.mark.parametrize("count", [19, 20, 38, 39, 76, 77, 152, 153, 304, 305, 608, 609])
def test_rounds_threads_by_number_of_proofs(count):
    rng = np.random.default_rng(count)
    ks = [1, 2, 7, 16, 40, 129, 300, 600, 5000]
    mats = {k: (_dev(_rand(rng, (5, k))), _dev(_rand(rng, (k, 3)))) for k in ks}
    jobs = [B.job(*mats[ks[i % len(ks)]], 0, 0, i) for i in range(count)]
    got = _prove(jobs)
    o = B.vl_batch_opts()
    o.rounds_variant = 4
    for i in list(range(16)) + [count - 1]:
        assert _prove([jobs[i]], o) == [got[i]]


@pytest.mark.parametrize("m,k,n,mont", [(1, 300, 1, 0), (33, 1025, 31, 0), (65, 257, 1030, 0), (17, 300, 65, 1),
                                        (130, 70, 129, 1)])
def test_cuda_core_fold_tiles_of_lone_and_many_products(m, k, n, mont):
    rng = np.random.default_rng(m + k + n)
    P, Q = _rand(rng, (m, k)), _rand(rng, (k, n))
    want = oracle.prove_matmul(P, Q, 0, 0, seed=9).to_bytes()
    if mont:
        ops = []
        for M in (P, Q):
            e = torch.zeros((*M.shape, 8), dtype=torch.int32, device="cuda")
            B.vl_encode(B.mat(_dev(M)), e.data_ptr())
            ops.append(e)
    else:  # leading dimensions that TMA cannot address
        ops = []
        for M in (P, Q):
            buf = torch.zeros((M.shape[0], (M.shape[1] + 7) // 8 * 8 + 3), dtype=torch.int16, device="cuda")
            buf[:, :M.shape[1]] = _dev(M)
            ops.append(buf[:, :M.shape[1]])
    job = B.job(*ops, 0, 0, 9)
    assert _prove([job]) == [want]
    assert _prove([job] * 40) == [want] * 40


@pytest.mark.parametrize("count,k", [(1, 1), (7, 1), (2, 2), (9, 5), (1, 8192), (9, 1500), (64, 128), (65, 256), (130, 70),
                                     (512, 3), (512, 40), (513, 3), (520, 36)])
def test_batched_claims_tails(count, k):
    """Batches whose last rounds run in one cluster, from every kind of first round, and larger ones without."""
    rng = np.random.default_rng(count + k)
    jobs = [{"P": _rand(rng, (2, k)), "Q": _rand(rng, (k, 1 + i % 2)), "tp": 0, "tq": 0} for i in range(count)]
    cj = [B.job(_dev(j["P"]), _dev(j["Q"]), 0, 0, 0) for j in jobs]
    n = B.vl_batch_workspace_bytes(cj)
    ws = _ws(n)
    res = B.vl_prove_matmul_batched(cj, 11, ws.data_ptr(), n)
    assert res.to_bytes() == OB.prove_matmul_batch(jobs, seed=11).to_bytes()


def _linear(mats, trans, seed):
    jobs = [B.lin_job([B.mat(_dev(M.T if t else M), t) for M, t in zip(mats, trans)], list(range(1, len(mats) + 1)),
                      seed)]
    n = B.vl_linear_workspace_bytes(jobs)
    ws = _ws(n)
    return B.lin_proof_bytes(B.vl_prove_linear(jobs, ws.data_ptr(), n)[0])


@pytest.mark.parametrize("red", [1, 2, 7, 8, 9, 15, 16, 17, 33, 63, 64, 65, 80, 127, 128])
@pytest.mark.parametrize("lines", [128, 161, 300])
def test_short_linear_reductions(red, lines):
    rng = np.random.default_rng(1000 * red + lines)
    mats = [_rand(rng, (lines, red)) for _ in range(3)]
    want = oracle.prove_linear(mats, [1, 2, 3], seed=red).to_bytes()
    assert _linear(mats, [0, 1, 0], red) == want
    tmats = [M.T.copy() for M in mats]
    want = oracle.prove_linear(tmats, [1, 2, 3], seed=red).to_bytes()
    assert _linear(tmats, [0, 0, 1], red) == want


@pytest.mark.parametrize("value", [-(1 << 15), (1 << 15) - 1, -1, 0, 255, 256])
@pytest.mark.parametrize("red", [64, 128])
def test_short_linear_reductions_of_extreme_entries(value, red):
    mats = [np.full((200, red), value, np.int16), np.full((200, red), -(1 << 15), np.int16)]
    want = oracle.prove_linear(mats, [1, 2], seed=3).to_bytes()
    assert _linear(mats, [0, 1], 3) == want


def test_short_linear_blocks_of_every_length():
    """Enough lines for 512- and 1024-line blocks: every proof equals the same
    statement proved alone (256-line blocks)."""
    rng = np.random.default_rng(5)
    jobs = []
    for i in range(40):
        rows, cols = (4096 + 37 * i, 5 + i) if i % 2 else (3 + i, 4000 + 64 * i)
        M = _dev(_rand(rng, (rows, cols)))
        jobs.append(B.lin_job([B.mat(M), B.mat(M), B.mat(M)], [1, 5, 9], i))
    for count in (12, 40):
        n = B.vl_linear_workspace_bytes(jobs[:count])
        ws = _ws(n)
        got = [B.lin_proof_bytes(p) for p in B.vl_prove_linear(jobs[:count], ws.data_ptr(), n)]
        for i in (0, 1, count - 2, count - 1):
            n = B.vl_linear_workspace_bytes([jobs[i]])
            ws = _ws(n)
            assert B.lin_proof_bytes(B.vl_prove_linear([jobs[i]], ws.data_ptr(), n)[0]) == got[i]


LOOKUPS = [(1, 0), (2, 1), (3, 0), (4, 2), (7, 3), (8, 1), (16, 4), (100, 2), (700, 8), (1500, 11), (3000, 3), (5000, 8),
           (5000, 12), (9000, 13)]


def _lookup_job(n, log2_n, seed):
    rng = np.random.default_rng(100 * n + log2_n)
    S = (rng.integers(0, 1 << log2_n, size=(1, n)) - 5).astype(np.int16)
    return S, B.lookup_job(B.mat(_dev(S)), -5, log2_n, seed)


@pytest.mark.parametrize("n,log2_n", LOOKUPS)
def test_lookup_alone(n, log2_n):
    S, job = _lookup_job(n, log2_n, 7)
    need = B.vl_lookup_workspace_bytes([job])
    ws = _ws(need)
    got = B.lookup_proof_bytes(B.vl_prove_lookup([job], ws.data_ptr(), need)[0])
    assert got == OL.prove_lookup(S, -5, log2_n, seed=7).to_bytes()


@pytest.mark.parametrize("count", [19, 20, 38, 39, 76, 77, 152, 153])
def test_lookup_batches_on_both_sides_of_the_tail_rule(count):
    shapes = LOOKUPS + [(40000, 8), (70000, 12), (33000, 15)]
    jobs = [_lookup_job(*shapes[i % len(shapes)], i)[1] for i in range(count)]
    need = B.vl_lookup_workspace_bytes(jobs)
    ws = _ws(need)
    got = [B.lookup_proof_bytes(p) for p in B.vl_prove_lookup(jobs, ws.data_ptr(), need)]
    for i in range(min(count, len(shapes))):
        need = B.vl_lookup_workspace_bytes([jobs[i]])
        w1 = _ws(need)
        assert B.lookup_proof_bytes(B.vl_prove_lookup([jobs[i]], w1.data_ptr(), need)[0]) == got[i]
