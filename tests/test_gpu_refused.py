"""A refused call leaves the caller's stream alone: it returns while earlier work
is still running there, and a capture that is under way goes on."""
import numpy as np
import pytest

import oracle
from paper_2508_21393_gb300 import binding as B

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no GPU", allow_module_level=True)


def _setup():
    rng = np.random.default_rng(4)
    P, Q = (rng.integers(-(1 << 15), 1 << 15, size=s).astype(np.int16) for s in ((6, 40), (40, 5)))
    job = B.job(torch.from_numpy(P).cuda(), torch.from_numpy(Q).cuda(), 0, 0, 3)
    need = B.vl_workspace_bytes([job])
    ws = torch.zeros(need + 256, dtype=torch.uint8, device="cuda")
    want = oracle.prove_matmul(P, Q, seed=3).to_bytes()
    assert B.proof_bytes(B.vl_prove_batch([job], ws.data_ptr(), need)[0]) == want
    return job, need, ws, want


def _refused(job, need, ws, stream, out=None):
    out = out or {}
    for at, size, code in ((0, need - 1, B.VL_ENOMEM), (16, need, B.VL_EINVAL)):
        with pytest.raises(B.VLError) as e:
            B.vl_prove_batch([job], ws.data_ptr() + at, size, stream=stream.cuda_stream, **out)
        assert e.value.code == code


def test_refused_calls_do_not_wait_for_the_stream():
    job, need, ws, want = _setup()
    dev = torch.zeros(B.ctypes.sizeof(B.vl_proof), dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        torch.cuda._sleep(1 << 29)  # a quarter of a second of the GPU's clock
    _refused(job, need, ws, s)
    _refused(job, need, ws, s, {"out": dev.data_ptr(), "out_space": B.VL_DEVICE})
    assert not s.query()
    s.synchronize()
    assert B.proof_bytes(B.vl_prove_batch([job], ws.data_ptr(), need)[0]) == want


def test_refused_calls_leave_a_capture_alone():
    job, need, ws, want = _setup()
    x = torch.zeros(1000, device="cuda")
    s = torch.cuda.Stream()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=s, capture_error_mode="relaxed"):
        x.add_(1)
        _refused(job, need, ws, s)
        x.add_(1)
    graph.replay()
    torch.cuda.synchronize()
    assert float(x.sum()) == 2000
    assert B.proof_bytes(B.vl_prove_batch([job], ws.data_ptr(), need)[0]) == want
