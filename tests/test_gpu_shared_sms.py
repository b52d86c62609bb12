"""Lone verification calls whose one wave over all SMs cannot be resident at once, because calls of other contexts on
other streams hold SMs: the results are the bits of undisturbed calls and no wait gives up."""
import os
import subprocess
import sys
import time

import pytest
import torch

from paper_2602_15318_b200 import binding as B
from paper_2602_15318_b200 import workloads as W

from gpu_util import check, oracle_verify, sample_rows

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _new(case):
    return (torch.full_like(case.q, float("nan")), torch.full((case.B, case.q.shape[2], case.T), float("nan"), dtype=torch.float32, device=DEV))


def _call(ctx, case, out, lse, stream):
    B.sparrow_verify_attn(ctx, case.q, case.k, case.v, case.kv_len, case.parents, case.T, out, lse, stream)


@pytest.mark.parametrize("kv_a,T_a,kv_b,T_b", [
    ([9000], 16, [7000], 12),               # one row block
    ([9000] * 8, 30, [9000], 16),           # items of two row blocks
    ([20000, 100, 6000], 12, [5000], 30),   # a sequence that is one piece beside others
])
def test_two_contexts_with_one_wave_each_beside_a_long_call(kv_a, T_a, kv_b, T_b):
    """A call of a third context holds about a third of the SMs for some 0.4 ms.  The first lone call starts on the
    others; the second, on a stream of higher priority, is given the SMs that the first one's last CTAs need."""
    a = W.make_verify_case(8100 + T_a, kv_a, T_a, "random", DEV)
    b = W.make_verify_case(8200 + T_b, kv_b, T_b, "chain", DEV)
    long_kv = 500_000
    gen = torch.Generator(device=DEV).manual_seed(83)
    k, v = (torch.empty((1, W.HKV, long_kv + 64, W.D), dtype=torch.bfloat16, device=DEV).normal_(generator=gen) for _ in range(2))
    q = torch.empty((1, 16, W.HQ, W.D), dtype=torch.bfloat16, device=DEV).normal_(generator=gen)
    parents = torch.tensor([W.chain_parents(16)], dtype=torch.int32, device=DEV)
    out, lse = torch.empty_like(q), torch.empty((1, W.HQ, 16), dtype=torch.float32, device=DEV)
    ctx, ctx_a, ctx_b = B.Context.for_cache(k, W.SCALE), B.Context.for_cache(a.k, W.SCALE), B.Context.for_cache(b.k, W.SCALE)
    hold = B.VerifyBatch([(q, k, v, [long_kv], parents, 16, out, lse)])         # (a batch keeps the policy's 55 pieces)
    low, high = torch.cuda.Stream(priority=0), torch.cuda.Stream(priority=-1)
    alone = []
    for c, case in ((ctx_a, a), (ctx_b, b)):
        o, l = _new(case)
        _call(c, case, o, l, None)
        torch.cuda.synchronize()
        rows = sample_rows(84, case.B, case.T, 40)
        check(o, l, *oracle_verify(case, rows), rows=rows)
        alone.append((o, l))
    worst = 0.0
    for _ in range(12):
        (oa, la), (ob, lb) = _new(a), _new(b)
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        B.sparrow_verify_attn_batch(ctx, hold)
        _call(ctx_a, a, oa, la, low)
        _call(ctx_b, b, ob, lb, high)
        torch.cuda.synchronize()
        worst = max(worst, time.perf_counter() - t0)
        assert torch.equal(oa, alone[0][0]) and torch.equal(la, alone[0][1])
        assert torch.equal(ob, alone[1][0]) and torch.equal(lb, alone[1][1])
    for c in (ctx, ctx_a, ctx_b):
        assert c.last_device_status() == 0
    assert worst < 0.2, f"{worst:.3f} s"


def test_contexts_created_at_once_by_several_threads_are_alike():
    """The first contexts of a process, created by sixteen threads at the same time: none may do without what another
    one is still asking the device for.  All of them plan a call alike, with merges in clusters."""
    code = """
import ctypes, sys, threading
import torch
from paper_2602_15318_b200 import binding as B
from paper_2602_15318_b200 import workloads as W
case = W.make_verify_case(8300, [1500], 16, "random", "cuda:0")
torch.cuda.synchronize()
L, n = B.lib(), 16
create, gate, made = L.sparrow_create, threading.Barrier(n), []
layout = B.Layout(1, W.HQ, W.HKV, W.D, case.k.shape[2], W.SCALE, W.HKV * case.k.shape[2] * W.D, case.k.shape[2] * W.D)
handles = [ctypes.c_void_p() for _ in range(n)]
def make(i):
    h, l = ctypes.byref(handles[i]), ctypes.byref(layout)
    gate.wait()
    made.append(create(h, l, 0))
sys.setswitchinterval(1e-6)
threads = [threading.Thread(target=make, args=(i,)) for i in range(n)]
[t.start() for t in threads]
[t.join() for t in threads]
assert made == [0] * n
ctx = []
for h in handles:
    c = B.Context(1, case.k.shape[2], layout.kv_stride_batch, layout.kv_stride_head, W.SCALE, allocate_workspace=False)
    L.sparrow_destroy(c.handle)
    c.handle, c.address = h, h.value
    size = c.workspace_bytes(16)
    c.workspace = torch.empty(size + 256, dtype=torch.uint8, device="cuda:0")
    c.set_workspace((c.workspace.data_ptr() + 255) // 256 * 256, size)
    ctx.append(c)
for c in ctx:
    out = torch.empty_like(case.q)
    lse = torch.empty((1, W.HQ, 16), dtype=torch.float32, device="cuda:0")
    B.sparrow_verify_attn(c, case.q, case.k, case.v, case.kv_len, case.parents, 16, out, lse)
torch.cuda.synchronize()
"""
    r = subprocess.run([sys.executable, "-c", code], cwd=ROOT, env={**os.environ, "SPARROW_LOG": "1", "PYTHONPATH": ROOT},
                       capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stderr[-2000:]
    plans = [line.split(";", 1)[1] for line in r.stderr.splitlines() if line.startswith("[sparrow] verify call")]
    assert len(plans) == 16 and len(set(plans)) == 1 and "merged in clusters of" in plans[0], plans
