"""Performance cases of the proving library: what a user has it prove, through its public calls.

Every case proves statements over int16 fixed-point matrices with LLaMA-like
shapes (hidden sizes 4096 and 5120, ranks 8 to 64, sequences of 256 to 2048
tokens) and the value distributions of ``workload.py``: activations and
upstream gradients ~ round(N(0, 2^8)), weights and LoRA factors
~ round(N(0, 0.02 * 2^8)), single products uniform over int16.  Outputs are
the proofs (bytes and canonical field elements): two correct provers agree on
every byte.
"""

import math

import numpy as np
import torch

from paper_2508_21393_gb300 import binding as B
from paper_2508_21393_gb300 import workload as W

LIMB_MACS = 128       # 32 x 32-bit multiply-adds of one Montgomery product of 8-limb elements
ENTRY_MACS = 8        # 32 x 16-bit multiply-adds of one fold entry (255-bit weight times int16)


def listed():
    return [
        # The smallest call: one product by itself, latency of launches and hashes.
        {"name": "matmul_small", "kind": "matmul", "m": 64, "k": 128, "n": 64, "ld_pad": 0},
        # A product cut out of larger tensors: odd sizes, leading dimensions that are no multiple of
        # 16 bytes (as a view of a tensor has), one call with its own plan.
        {"name": "matmul_ragged", "kind": "matmul", "m": 601, "k": 2057, "n": 1033, "ld_pad": 3},
        # Operands that a program holds as field elements: encoded on the GPU, then proved.
        {"name": "matmul_encoded", "kind": "encoded", "m": 512, "k": 2048, "n": 256},
        # One adapted projection (its eight products) of a 7B model, proved again and again by a plan.
        {"name": "projection_7b", "kind": "step", "layers": 1, "projections": 1, "seq": 1024, "hidden": 4096,
         "ranks": "16", "tune": False},
        # One request of a proving service: W resident on the GPU, the activations and factors in
        # pinned host memory, proofs back to the host, one call.
        {"name": "request_13b", "kind": "request", "seq": 1024, "hidden": 5120, "rank": 8},
        # The headline: every product of one LoRA step of a 7B model, tuned plan.
        {"name": "step_7b", "kind": "step", "layers": 32, "projections": 4, "seq": 512, "hidden": 4096,
         "ranks": "8,16,64", "tune": True},
        # The same of a 13B model with long sequences (hidden 5120, padded to 8192 in the proofs).
        {"name": "step_13b", "kind": "step", "layers": 40, "projections": 4, "seq": 2048, "hidden": 5120,
         "ranks": "16", "tune": True},
        # The parameter updates of the 7B step: linear relations on every LoRA factor.
        {"name": "updates_7b", "kind": "updates", "layers": 32, "projections": 4, "hidden": 4096, "ranks": "8,16,64"},
        # One range lookup by itself: the remainders of one projection's H.
        {"name": "lookup_one", "kind": "lookups", "layers": 1, "projections": 1, "tables": "H", "seq": 512,
         "hidden": 4096, "ranks": "16"},
        # Every range lookup of the 7B step's rescale remainders.
        {"name": "lookups_7b", "kind": "lookups", "layers": 32, "projections": 4, "tables": "H,dH,GA,GB", "seq": 512,
         "hidden": 4096, "ranks": "8,16,64"},
        # The products of several layers that share an inner dimension, as one batched-claim proof.
        {"name": "claims_7b", "kind": "claims", "layers": 8, "projections": 4, "seq": 512, "hidden": 4096,
         "ranks": "8,16,64"},
        # Chained proofs of the projections of one layer (intermediates never opened).
        {"name": "chain_7b", "kind": "chain", "layers": 1, "projections": 4, "seq": 512, "hidden": 4096, "ranks": "16"},
    ]


def _log(rng, lo, hi):
    """An integer spread over the logarithm of [lo, hi]."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["matmul", "encoded", "step", "step", "request", "updates", "lookups", "lookups", "claims",
                       "chain"])
    hidden = 8 * _log(rng, 32, 640)
    seq = _log(rng, 33, 2048)
    rank = rng.choice([3, 4, 8, 13, 16, 24, 32, 64])
    ranks = ",".join(str(r) for r in sorted(set([rank, rng.choice([8, 16, 64])])))
    if kind == "matmul":
        return {"kind": kind, "m": _log(rng, 1, 3000), "k": _log(rng, 1, 9000), "n": _log(rng, 1, 3000),
                "ld_pad": rng.choice([0, 0, 1, 3, 8, 40])}
    if kind == "encoded":
        return {"kind": kind, "m": _log(rng, 5, 900), "k": _log(rng, 5, 3000), "n": _log(rng, 5, 900)}
    if kind == "request":
        return {"kind": kind, "seq": seq, "hidden": hidden, "rank": rank}
    layers, projections = _log(rng, 1, 24), rng.choice([1, 2, 4])
    if kind == "step":
        return {"kind": kind, "layers": layers, "projections": projections, "seq": seq, "hidden": hidden,
                "ranks": ranks, "tune": rng.random() < 0.25}
    if kind == "updates":
        return {"kind": kind, "layers": layers, "projections": projections, "hidden": hidden, "ranks": ranks}
    if kind == "lookups":
        return {"kind": kind, "layers": layers, "projections": projections,
                "tables": rng.choice(["H", "H,dH", "GA,GB", "H,dH,GA,GB"]), "seq": seq, "hidden": hidden,
                "ranks": ranks}
    layers = _log(rng, 1, 6)
    return {"kind": kind, "layers": layers, "projections": projections, "seq": seq, "hidden": hidden, "ranks": ranks}


# ------------------------------------------------------------------ inputs --

def _uniform(g, rows, cols):
    return torch.randint(-(1 << 15), 1 << 15, (rows, cols), generator=g, device="cuda", dtype=torch.int32).to(torch.int16)


def _gauss(g, rows, cols, sigma):
    x = torch.randn((rows, cols), generator=g, device="cuda", dtype=torch.float32)
    return x.mul_(sigma).round_().clamp_(W.I16_MIN, W.I16_MAX).to(torch.int16)


def _product(a, b):
    """Exact integer product (every partial sum is below 2^53)."""
    return (a.double() @ b.double()).to(torch.int64)


def _rescale(z, shift=W.RESCALE_SHIFT):
    return ((z + (1 << (shift - 1))) >> shift).clamp_(W.I16_MIN, W.I16_MAX).to(torch.int16)


def _remainder(z, shift):
    return ((z + (1 << (shift - 1))) & ((1 << shift) - 1)).to(torch.int16)


def _projections(case):
    """(layer, projection name, rank) of every projection of the case."""
    ranks = [int(r) for r in case["ranks"].split(",")]
    return [(l, p, ranks[l % len(ranks)]) for l in range(case["layers"]) for p in W.PROJECTIONS[:case["projections"]]]


def _tensors(g, seq, hidden, rank):
    """One projection: X, W, A, B, dY and the rescaled intermediates H, dH."""
    t = {"X": _gauss(g, seq, hidden, W.ACT_SIGMA), "W": _gauss(g, hidden, hidden, W.WEIGHT_SIGMA),
         "A": _gauss(g, hidden, rank, W.WEIGHT_SIGMA), "B": _gauss(g, rank, hidden, W.WEIGHT_SIGMA),
         "dY": _gauss(g, seq, hidden, W.ACT_SIGMA)}
    t["XA"], t["dYB"] = _product(t["X"], t["A"]), _product(t["dY"], t["B"].t())
    t["H"], t["dH"] = _rescale(t["XA"]), _rescale(t["dYB"])
    return t


PRODUCTS = {"F1": ("X", "W", 0, 0), "F2": ("X", "A", 0, 0), "F3": ("H", "B", 0, 0), "B1": ("dY", "B", 0, 1),
            "B2": ("H", "dY", 1, 0), "B3": ("X", "dH", 1, 0), "B4": ("dY", "W", 0, 1), "B5": ("dH", "A", 0, 1)}


def _jobs(t, layer, proj, seed, names=W.PRODUCTS):
    out = []
    for name in names:
        p, q, tp, tq = PRODUCTS[name]
        out.append(B.job(t[p], t[q], tp, tq, W.proof_seed(seed, layer, proj, name)))
    return out


def _buffer(nbytes):
    return torch.zeros(max(int(nbytes), 256), dtype=torch.uint8, device="cuda")


class _State(dict):
    """Inputs, plan and buffers of a case; the plan is released with them."""

    def __init__(self, **kw):
        super().__init__(**kw)
        self.release = None

    def __del__(self):
        if self.release is not None:
            torch.cuda.synchronize()
            self.release()


def _size(ctype):
    return B.ctypes.sizeof(ctype)


def prepare(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed * 1000003 + 17)
    kind = case["kind"]
    if kind == "matmul":
        m, k, n, pad = case["m"], case["k"], case["n"], case["ld_pad"]
        P, Q = _uniform(g, m, k + pad)[:, :k], _uniform(g, k, n + pad)[:, :n]
        job = B.job(P, Q, 0, 0, W.proof_seed(seed, 0, "x", "M"))
        need = B.vl_workspace_bytes([job])
        return _State(kind=kind, job=job, ws=_buffer(need), need=need)
    if kind == "encoded":
        m, k, n = case["m"], case["k"], case["n"]
        P, Q = _uniform(g, m, k), _uniform(g, k, n)
        Pe = torch.zeros((m, k, 8), dtype=torch.int32, device="cuda")
        Qe = torch.zeros((k, n, 8), dtype=torch.int32, device="cuda")
        job = B.job(Pe, Qe, 0, 0, W.proof_seed(seed, 0, "x", "M"))
        need = B.vl_workspace_bytes([job])
        return _State(kind=kind, P=B.mat(P), Q=B.mat(Q), Pe=Pe, Qe=Qe, job=job, ws=_buffer(need), need=need)
    if kind == "request":
        t = _tensors(g, case["seq"], case["hidden"], case["rank"])
        host = {x: t[x].cpu().pin_memory() for x in ("X", "A", "B", "dY", "H", "dH")}
        host["W"] = t["W"]
        jobs = _jobs(host, 0, "q", seed)
        need = B.vl_workspace_bytes(jobs)
        return _State(kind=kind, jobs=jobs, ws=_buffer(need), need=need)
    if kind == "step":
        jobs = []
        for layer, proj, rank in _projections(case):
            jobs += _jobs(_tensors(g, case["seq"], case["hidden"], rank), layer, proj, seed)
        opts = B.vl_batch_opts()
        if case["tune"]:
            need = B.vl_workspace_bytes(jobs)
            # candidates with shorter tiles keep accumulators: room for the largest
            most = max(need, max(B.vl_workspace_bytes(jobs, _with(engine=e, seg=s)) for e, s in
                                 ((0, 1024), (0, 4096), (1, 0))))
            ws = _buffer(most + (64 << 20))
            opts, _ = B.vl_autotune(jobs, ws.data_ptr(), ws.numel(), base=opts)
        plan = B.vl_plan_create(jobs, opts)
        need = B.vl_plan_workspace_bytes(plan)
        if not case["tune"] or need > ws.numel():
            ws = _buffer(need)
        st = _State(kind=kind, jobs=jobs, plan=plan, ws=ws, need=need, out=_buffer(_size(B.vl_proof) * len(jobs)))
        st.release = lambda: B.vl_plan_destroy(plan)
        return st
    if kind == "updates":
        jobs, hidden = [], case["hidden"]
        for layer, proj, rank in _projections(case):
            for name, (rows, cols) in (("A", (hidden, rank)), ("B", (rank, hidden))):
                F = _gauss(g, rows, cols, W.WEIGHT_SIGMA)
                G = _gauss(g, rows, cols, 4 * W.WEIGHT_SIGMA)
                F2 = F - G
                jobs.append(B.lin_job([B.mat(F2), B.mat(F), B.mat(G)], [1, -1, 1],
                                      W.proof_seed(seed, layer, proj, "U" + name)))
        return _planned(kind, B.LinPlan(jobs), B.vl_lin_proof, jobs)
    if kind == "lookups":
        jobs, seq, hidden = [], case["seq"], case["hidden"]
        for layer, proj, rank in _projections(case):
            X, dY = _gauss(g, seq, hidden, W.ACT_SIGMA), _gauss(g, seq, hidden, W.ACT_SIGMA)
            A, Bm = _gauss(g, hidden, rank, W.WEIGHT_SIGMA), _gauss(g, rank, hidden, W.WEIGHT_SIGMA)
            XA, dYB = _product(X, A), _product(dY, Bm.t())
            tables = {"H": lambda: (XA, W.RESCALE_SHIFT), "dH": lambda: (dYB, W.RESCALE_SHIFT),
                      "GA": lambda: (_product(X.t(), _rescale(dYB)), W.UPDATE_SHIFT),
                      "GB": lambda: (_product(_rescale(XA).t(), dY), W.UPDATE_SHIFT)}
            for name in case["tables"].split(","):
                z, shift = tables[name]()
                jobs.append(B.lookup_job(B.mat(_remainder(z, shift)), 0, shift,
                                         W.proof_seed(seed, layer, proj, "R" + name)))
        return _planned(kind, B.LookupPlan(jobs), B.vl_lookup_proof, jobs)
    if kind == "claims":
        jobs = []
        for layer, proj, rank in _projections(case):
            t = _tensors(g, case["seq"], case["hidden"], rank)
            jobs += _jobs(t, layer, proj, seed, ("F1", "F2", "B1", "B4"))  # inner dimension: hidden
        plan = B.ClaimsPlan(jobs, W.proof_seed(seed, 0, "x", "claims"))
        need = plan.workspace_bytes()
        outs = [_buffer(_size(B.vl_batch_proof))] + [_buffer(32 * len(jobs)) for _ in range(3)]
        st = _State(kind=kind, jobs=jobs, plan=plan, ws=_buffer(need), need=need, outs=outs)
        st.release = plan.destroy
        return st
    assert kind == "chain"
    jobs = []
    for layer, proj, rank in _projections(case):
        t = _tensors(g, case["seq"], case["hidden"], rank)
        t["rhoH"], t["rhodH"] = (_remainder(t[z], W.RESCALE_SHIFT) for z in ("XA", "dYB"))
        jobs.append(B.chain_job(t, W.proof_seed(seed, layer, proj, "chain")))
    plan = B.ChainPlan(jobs)
    need = plan.workspace_bytes()
    st = _State(kind=kind, jobs=jobs, plan=plan, ws=_buffer(need), need=need)
    st.release = plan.destroy
    return st


def _with(engine, seg):
    o = B.vl_batch_opts()
    o.fold_engine, o.tc_seg = engine, seg
    return o


def _planned(kind, plan, proof, jobs):
    need = plan.workspace_bytes()
    # the jobs keep the operands alive: the plan holds their addresses only
    st = _State(kind=kind, jobs=jobs, plan=plan, ws=_buffer(need), need=need, out=_buffer(_size(proof) * len(jobs)))
    st.release = plan.destroy
    return st


def _host_bytes(proofs):
    return np.frombuffer(proofs, dtype=np.uint8)


def run(st):
    kind, ws, need = st["kind"], st["ws"].data_ptr(), st["need"]
    if kind == "matmul":
        j = st["job"]
        return _host_bytes(B.vl_prove_matmul(j.P, j.Q, j.fs, ws, need))
    if kind == "encoded":
        B.vl_encode(st["P"], st["Pe"].data_ptr())
        B.vl_encode(st["Q"], st["Qe"].data_ptr())
        j = st["job"]
        return {"P": st["Pe"], "Q": st["Qe"], "proof": _host_bytes(B.vl_prove_matmul(j.P, j.Q, j.fs, ws, need))}
    if kind == "request":
        return _host_bytes(B.vl_prove_batch(st["jobs"], ws, need))
    if kind == "step":
        B.vl_plan_run(st["plan"], ws, need, st["out"].data_ptr(), B.VL_DEVICE)
        return st["out"]
    if kind in ("updates", "lookups"):
        st["plan"].run(ws, need, out=st["out"].data_ptr(), out_space=B.VL_DEVICE)
        return st["out"]
    if kind == "claims":
        st["plan"].run(ws, need, device_out=[o.data_ptr() for o in st["outs"]])
        return st["outs"]
    return _host_bytes(st["plan"].run(ws, need))


# -------------------------------------------------------------------- work --

def _cube(x):
    return 1 << max(0, int(x) - 1).bit_length()


def _product_macs(m, k, n):
    """Fold entries at ENTRY_MACS; the rounds at three products per pair of
    the first and seven per pair of every later round; one product per entry
    of the two eq tables."""
    K = _cube(k)
    rounds = 3 * (K // 2) + 7 * (K // 2 - 1) if K > 1 else 1
    return (m * k + k * n) * ENTRY_MACS + (max(0, rounds) + m + n) * LIMB_MACS


def _shapes(seq, hidden, rank, names=W.PRODUCTS):
    s = {"F1": (seq, hidden, hidden), "F2": (seq, hidden, rank), "F3": (seq, rank, hidden),
         "B1": (seq, hidden, rank), "B2": (rank, seq, hidden), "B3": (hidden, seq, rank),
         "B4": (seq, hidden, hidden), "B5": (seq, rank, hidden)}
    return [s[x] for x in names]


def work(case):
    """bytes: every distinct input matrix and every proof once; flops: two
    per 32-bit integer multiply-add of the folds and field products."""
    kind = case["kind"]
    if kind in ("matmul", "encoded"):
        m, k, n = case["m"], case["k"], case["n"]
        entries = m * k + k * n
        macs, nbytes = _product_macs(m, k, n), 2 * entries + _size(B.vl_proof)
        if kind == "encoded":
            nbytes += 2 * 32 * entries  # the encoded operands are written and read
            macs += entries * (2 * LIMB_MACS)
        return {"bytes": nbytes, "flops": 2 * macs}
    if kind == "request":
        projections = [(0, "q", case["rank"])]
    else:
        projections = _projections(case)
    hidden, seq = case["hidden"], case.get("seq", 0)
    macs = nbytes = 0
    for _, _, r in projections:
        if kind in ("step", "request", "claims"):
            names = W.PRODUCTS if kind != "claims" else ("F1", "F2", "B1", "B4")
            macs += sum(_product_macs(*s) for s in _shapes(seq, hidden, r, names))
            nbytes += 2 * (2 * seq * hidden + hidden * hidden + 2 * hidden * r + 2 * seq * r)
            nbytes += len(names) * (_size(B.vl_proof) if kind != "claims" else 96)
        elif kind == "updates":
            macs += 6 * hidden * r * ENTRY_MACS + 6 * hidden * 2 * LIMB_MACS
            nbytes += 12 * hidden * r + 2 * _size(B.vl_lin_proof)
        elif kind == "lookups":
            for name in case["tables"].split(","):
                n, shift = (seq * r, W.RESCALE_SHIFT) if name in ("H", "dH") else (hidden * r, W.UPDATE_SHIFT)
                macs += 10 * max(_cube(n), 1 << shift) * LIMB_MACS
                nbytes += 2 * n + _size(B.vl_lookup_proof)
        else:
            members = ("F1", "F3", "B4", "B5", "B3", "B2", "F2", "F2", "B1", "B1")
            macs += sum(_product_macs(*s) for s in _shapes(seq, hidden, r, members))
            nbytes += 2 * (2 * seq * hidden + hidden * hidden + 2 * hidden * r + 4 * seq * r) + _size(B.vl_chain_proof)
    return {"bytes": nbytes, "flops": 2 * macs}


def exact(case, seed):
    """Proofs are bytes and canonical field elements that follow from hashes:
    there is no 64-bit value to be near to, only the one right answer."""
    return None
