"""How the pieces of a call are merged (in clusters of one or of two row blocks, through the workspace, by the combine
kernel), at the sizes where each way can go wrong.  The way that a call takes is read from its log line, so that a change of the
plan's estimates shows here; results against the oracle, tolerances as everywhere (gpu_util)."""
import re
import time

import pytest
import torch

import oracle
from paper_2602_15318_b200 import binding as B
from paper_2602_15318_b200 import workloads as W

from gpu_util import check, oracle_verify, sample_rows

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _context(monkeypatch, case):
    monkeypatch.setenv("SPARROW_LOG", "1")
    ctx = B.Context.for_cache(case.k, W.SCALE, n_q_heads=case.q.shape[2])
    monkeypatch.delenv("SPARROW_LOG")
    return ctx


def _new(case):
    return (torch.full_like(case.q, float("nan")), torch.full((case.B, case.q.shape[2], case.T), float("nan"), dtype=torch.float32, device=DEV))


def _call(ctx, case, out, lse, stream=None):
    B.sparrow_verify_attn(ctx, case.q, case.k, case.v, case.kv_len, case.parents, case.T, out, lse, stream)


def _plans(capfd):
    """(row blocks an item, CTAs of a cluster or 0, pieces of each sequence, finishers inside the kernel) of each call logged so far."""
    found = []
    for line in capfd.readouterr().err.splitlines():
        if line.startswith("[sparrow] verify call"):
            cluster, fin = re.search(r"merged in clusters of (\d+)", line), re.search(r"(\d+) finisher", line)
            found.append((int(re.search(r"(\d+) per item", line).group(1)), int(cluster.group(1)) if cluster else 0,
                          [int(x) for x in re.findall(r"in (\d+) piece", line)], int(fin.group(1)) if fin and "counter protocol" in line else 0))
    return found


def _check(case, out, lse, n=32):
    rows = [r for r in sample_rows(9100 + case.T, case.B, case.T, n) if r[2] < case.q.shape[2]]
    check(out, lse, *oracle_verify(case, rows), rows=rows)


@pytest.mark.parametrize("hq,hkv,kv_len,T,tree,per_item,cluster,pieces", [
    (28, 4, [96 * 128 - 16], 16, "random", 1, 16, [16]),      # the longest pieces of six tiles
    (28, 4, [96 * 128 - 15], 16, "random", 1, 0, [37]),       # one key more: through the workspace
    (28, 4, [112 * 128 - 16], 16, "chain", 1, 16, [16]),      # seven tiles against four
    (28, 4, [112 * 128 - 15], 16, "chain", 1, 0, [37]),
    (28, 4, [26112], 3, "chain", 1, 0, [37]),                 # 84 rows, one for each finisher
    (28, 4, [16384], 64, "random", 1, 0, [9]),                # sixteen units
    (28, 4, [26000] * 2, 56, "random", 2, 0, [9, 9]),         # two row blocks
    (28, 4, [15781] * 3, 59, "random", 2, 0, [6, 6, 6]),
    (28, 4, [20000, 100, 6000], 12, "random", 1, 0, None),    # one piece beside others
])
def test_edge_of_clusters_and_workspace(hq, hkv, kv_len, T, tree, per_item, cluster, pieces, capfd, monkeypatch):
    case = W.make_verify_case(9000 + T + len(kv_len), kv_len, T, tree, DEV, hq=hq, hkv=hkv)
    ctx = _context(monkeypatch, case)
    first = None
    capfd.readouterr()
    for _ in range(3):
        out, lse = _new(case)
        _call(ctx, case, out, lse)
        torch.cuda.synchronize()
        assert ctx.last_device_status() == 0
        first = first or (out, lse)
        assert torch.equal(out, first[0]) and torch.equal(lse, first[1])
    for plan in _plans(capfd):
        assert plan[:2] == (per_item, cluster) and (pieces is None or plan[2] == pieces), plan
        assert (plan[3] > 0) == (cluster == 0)
    _check(case, *first)


@pytest.mark.parametrize("hq,hkv,kv_len,T,per_item,cluster", [
    (28, 4, [33 * 128 - 18], 18, 1, 14),            # fourteen pieces, five of three tiles: only their CTAs use the whole ring
    (32, 4, [81 * 128 - 16], 16, 1, 16),            # sixteen pieces, one of six tiles, the others of five
    (28, 4, [12295] * 4, 56, 2, 4),                 # two row blocks, 97 tiles in four pieces: one odd, three even
    (28, 4, [12295 + 128 * 2, 12295, 9000, 12000], 64, 2, 4),     # ragged, the second row block half full
    (28, 4, [3115] * 6, 19, 2, 5),                  # five tiles each, one token in the second block
    (28, 4, [8455, 8455, 8000, 8455, 8455, 8100, 8455, 8455], 20, 2, 4),
])
def test_pieces_of_clusters_that_fill_the_ring(hq, hkv, kv_len, T, per_item, cluster, capfd, monkeypatch):
    """Peers write to a stage of the ring that the piece has used, behind its last use: the same bits call after call, of
    every cluster, while the next call's clusters start behind."""
    case = W.make_verify_case(9300 + T + len(kv_len), kv_len, T, "random", DEV, hq=hq, hkv=hkv)
    ctx = _context(monkeypatch, case)
    outs = [_new(case) for _ in range(8)]
    capfd.readouterr()
    for _ in range(3):
        for o, l in outs:
            _call(ctx, case, o, l)
    torch.cuda.synchronize()
    assert ctx.last_device_status() == 0
    for plan in _plans(capfd):
        assert plan[:2] == (per_item, cluster) and plan[2] == [cluster] * len(kv_len), plan
    for o, l in outs:
        assert torch.equal(o, outs[0][0]) and torch.equal(l, outs[0][1])
    _check(case, *outs[0])


@pytest.mark.parametrize("kv_a,T_a,kv_b,T_b,blocks", [
    ([26112], 16, [20000], 12, (1, 1)),             # one row block, one wave each
    ([26000] * 2, 56, [26112], 16, (2, 1)),         # items of two row blocks
    ([20000, 100, 6000], 12, [24000], 16, (1, 1)),  # a sequence that is one piece beside others
])
def test_two_workspace_merges_beside_a_long_call(kv_a, T_a, kv_b, T_b, blocks, capfd, monkeypatch):
    """Two lone calls that both fill the GPU and merge through the workspace, beside a call of a third context that holds
    about a third of the SMs for longer than finishers are patient: some leave, and the last to arrive merges for them."""
    a = W.make_verify_case(9400 + T_a, kv_a, T_a, "random", DEV)
    b = W.make_verify_case(9450 + T_b, kv_b, T_b, "chain", DEV)
    long_kv = 900_000
    gen = torch.Generator(device=DEV).manual_seed(94)
    k, v = (torch.empty((1, W.HKV, long_kv + 64, W.D), dtype=torch.bfloat16, device=DEV).normal_(generator=gen) for _ in range(2))
    q = torch.empty((1, 16, W.HQ, W.D), dtype=torch.bfloat16, device=DEV).normal_(generator=gen)
    parents = torch.tensor([W.chain_parents(16)], dtype=torch.int32, device=DEV)
    out, lse = torch.empty_like(q), torch.empty((1, W.HQ, 16), dtype=torch.float32, device=DEV)
    ctx, ctx_a, ctx_b = B.Context.for_cache(k, W.SCALE), _context(monkeypatch, a), _context(monkeypatch, b)
    hold = B.VerifyBatch([(q, k, v, [long_kv], parents, 16, out, lse)])
    low, high = torch.cuda.Stream(priority=0), torch.cuda.Stream(priority=-1)
    alone = []
    capfd.readouterr()
    for c, case in ((ctx_a, a), (ctx_b, b)):
        o, l = _new(case)
        _call(c, case, o, l)
        torch.cuda.synchronize()
        _check(case, o, l, 40)
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
    plans = _plans(capfd)
    assert len(plans) == 26
    for plan in plans:                                # every call merges through the workspace, all its CTAs finishers
        assert plan[1] == 0 and plan[3] > 32, plan
    assert {p[0] for p in plans} == set(blocks)
    assert worst < 0.2, f"{worst:.3f} s"


def test_kinds_of_merge_in_turn_on_one_context(capfd, monkeypatch):
    """Cluster, workspace, one piece, workspace of two row blocks: enqueued without synchronisation, in turn and in front of a
    batch."""
    cap = 26112 + 64
    cases = [W.make_verify_case(9500 + i, [kv, kv], T, tree, DEV, capacity=cap)
             for i, (kv, T, tree) in enumerate([(700, 8, "chain"), (26112, 16, "random"), (60, 12, "random"), (26000, 56, "random")])]
    ctx = _context(monkeypatch, cases[0])
    capfd.readouterr()
    results = []
    for _ in range(4):
        for c in cases:
            results.append(_new(c))
            _call(ctx, c, *results[-1])
        outs = [_new(c) for c in cases]
        B.sparrow_verify_attn_batch(ctx, B.VerifyBatch([(c.q, c.k, c.v, c.kv_len, c.parents, c.T, o, l) for c, (o, l) in zip(cases, outs)]))
        results += outs
    torch.cuda.synchronize()
    assert ctx.last_device_status() == 0
    plans = _plans(capfd)
    assert [(p[0], p[1] > 1, p[2][0] > 1) for p in plans[:4]] == [(1, True, True), (1, False, True), (1, False, False), (2, False, True)], plans[:4]
    for i, (out, lse) in enumerate(results):
        assert torch.equal(out, results[i % 8][0]) and torch.equal(lse, results[i % 8][1])
    for i, (out, lse) in enumerate(results[:8]):
        _check(cases[i % 4], out, lse, 24)


@pytest.mark.parametrize("kv,T,per_item", [(26112, 16, 1), (26000, 56, 2)])
def test_late_inputs_of_a_call_that_merges_through_the_workspace(kv, T, per_item, capfd, monkeypatch):
    """Each device input in turn is written by the kernel directly before the call, which lets its dependents start at
    once and writes 0, 50 or 400 us later."""
    case = W.make_verify_case(9600 + T, [kv, kv] if per_item == 2 else [kv], T, "random", DEV)
    ctx = _context(monkeypatch, case)
    capfd.readouterr()
    want = _new(case)
    _call(ctx, case, *want)
    torch.cuda.synchronize()
    _check(case, *want, 24)
    for name in ("q", "k", "v", "parents"):
        true = getattr(case, name)
        live = torch.zeros(true.numel() + 64, dtype=true.dtype, device=DEV)          # (whole 16-byte words)
        src = torch.zeros_like(live)
        src[:true.numel()] = true.flatten()
        for delay in (0, 50, 400):
            live.zero_() if name != "parents" else live.fill_(-1)
            x = {n: getattr(case, n) for n in ("q", "k", "v", "parents")}
            x[name] = live[:true.numel()].view(true.shape)
            out, lse = _new(case)
            torch.cuda.synchronize()
            B.sparrow_debug_early_trigger_copy(ctx, src, live, live.numel() * live.element_size(), delay)
            B.sparrow_verify_attn(ctx, x["q"], x["k"], x["v"], case.kv_len, x["parents"], T, out, lse)
            torch.cuda.synchronize()
            assert torch.equal(out, want[0]) and torch.equal(lse, want[1]), f"{name} written {delay} us late"
    assert ctx.last_device_status() == 0
    for plan in _plans(capfd):
        assert plan[:2] == (per_item, 0) and plan[3] > 32, plan


@pytest.mark.parametrize("n_text,T_tree,T_new,window,launches", [
    (16 * 64 - 32, 64, 18, 300, 2),         # seventeen tiles, one unit a KV head: partial rows and the combine kernel
    (16 * 64 - 33, 33, 5, 0, 1),            # sixteen: one cluster a KV head
    (2500, 64, 9, 0, 2),                    # nodes in two tiles far behind
])
def test_gathered_trees_merged_by_the_combine_kernel(n_text, T_tree, T_new, window, launches):
    idx = list(range(40, 40 + n_text)) + list(range(4000, 4000 + T_tree))
    case = W.make_anchor_case(9700 + n_text, idx, window + 4000 - 40 - n_text if window else 0, T_tree, 1, DEV)
    parents = torch.tensor([W.random_tree_parents(9750 + n_text, 99, T_tree)], dtype=torch.int32, device=DEV)
    q = case.q[:, T_tree - T_new:].contiguous()
    ctx = B.Context.for_cache(case.k, W.SCALE)
    before = ctx.launch_count()
    out, lse = torch.full_like(q, float("nan")), torch.full((1, W.HQ, T_new), float("nan"), dtype=torch.float32, device=DEV)
    B.sparrow_anchor_attn_tree(ctx, q, case.k, case.v, case.anchor_idx, case.n_anchor, case.window, parents, T_tree, T_new, out, lse)
    torch.cuda.synchronize()
    assert ctx.last_device_status() == 0 and ctx.launch_count() - before == launches
    check(out, lse, *oracle.anchor_attn_tree(W.bf16_bits(q), W.bf16_bits(case.k), W.bf16_bits(case.v), case.anchor_idx.cpu().numpy(),
                                             case.window, parents.cpu().numpy(), W.SCALE))


@pytest.mark.parametrize("hq,hkv,kv_len,T,per_item,pieces", [
    (32, 8, [17017, 17019, 12086], 51, 1, [3, 3, 3]),
    (28, 4, [32768], 64, 1, [9]),
    (28, 4, [500], 16, 1, [5]),                     # never in clusters
])
def test_route_of_a_captured_call(hq, hkv, kv_len, T, per_item, pieces, capfd, monkeypatch):
    """A call captured into a graph plans with the lone call's estimates and merges in the combine kernel."""
    case = W.make_verify_case(9800 + T, kv_len, T, "random", DEV, hq=hq, hkv=hkv)
    ctx = _context(monkeypatch, case)
    out, lse = _new(case)
    capfd.readouterr()
    g, s = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    before = ctx.launch_count()
    with torch.cuda.graph(g, stream=s):
        _call(ctx, case, out, lse, s)
    assert ctx.launch_count() - before == 2
    g.replay()
    torch.cuda.synchronize()
    assert ctx.last_device_status() == 0
    assert _plans(capfd) == [(per_item, 0, pieces, 0)]
    _check(case, out, lse)
