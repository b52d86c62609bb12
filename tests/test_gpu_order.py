"""What a launch may overlap: which verification calls start early, and that every kernel of the library that is
launched while its predecessor is still running waits for it before it reads or writes."""
import pytest
import torch

from paper_2602_15318_b200 import binding as B
from paper_2602_15318_b200 import workloads as W

from gpu_util import check, oracle_verify

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _new(case):
    return (torch.full_like(case.q, float("nan")), torch.full((case.B, case.q.shape[2], case.T), float("nan"), dtype=torch.float32, device=DEV))


def _call(ctx, case, stream=None):
    out, lse = _new(case)
    B.sparrow_verify_attn(ctx, case.q, case.k, case.v, case.kv_len, case.parents, case.T, out, lse, stream)
    return out, lse


@pytest.mark.parametrize("between", ["refused", "captured"])
def test_a_call_that_is_not_in_the_stream_is_not_the_previous_call(between, monkeypatch, capfd):
    """Behind a call of another context (or another kernel of the library) a call takes stream order, also when a
    call of its own context that was refused, or went into a graph, lies between the two on the host."""
    monkeypatch.setenv("SPARROW_LOG", "1")
    a = W.make_verify_case(8400, [100], 8, "chain", DEV, capacity=2200)
    b = W.make_verify_case(8401, [2000], 8, "random", DEV, capacity=2200)
    ctx_a = B.Context.for_cache(a.k, W.SCALE, max_T=8)
    ctx_b = B.Context.for_cache(b.k, W.SCALE)
    # room for the partials of ten work items: enough for a's four, too little for a call of 2,000 keys
    part = lambda items: 2 * ((items * 129 * 272 + 255) // 256 * 256)
    most = torch.cuda.get_device_properties(0).multi_processor_count + W.HKV
    ctx_a.set_workspace(ctx_a.workspace.data_ptr(), ctx_a.workspace_bytes(8) - part(most) + part(10))
    for c in (ctx_a, ctx_b):
        c.set_call_overlap(True)
    _call(ctx_a, a)
    _call(ctx_a, a)
    torch.cuda.synchronize()
    lines = [l for l in capfd.readouterr().err.splitlines() if l.startswith("[sparrow] verify call")]
    assert ["starts early" in l for l in lines] == [False, True]
    _call(ctx_b, b)
    if between == "refused":
        with pytest.raises(B.SparrowError) as e:
            _call(ctx_a, b)
        assert e.value.status == 5
    else:
        s = torch.cuda.Stream()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=s):
            _call(ctx_a, a)
    out, lse = _call(ctx_a, a)
    torch.cuda.synchronize()
    lines = [l for l in capfd.readouterr().err.splitlines() if l.startswith("[sparrow] verify call")]
    assert "stream order" in lines[-1] and "starts early" not in lines[-1]
    check(out, lse, *oracle_verify(a))
    assert ctx_a.last_device_status() == 0 and ctx_b.last_device_status() == 0
