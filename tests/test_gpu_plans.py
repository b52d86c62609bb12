"""The plan that a verification call takes, read from the log line: sizes on both sides of the rules that choose
between items of one and of two row blocks and that cut long pieces, each with its result against the oracle."""
import re

import pytest
import torch

from paper_2602_15318_b200 import binding as B
from paper_2602_15318_b200 import workloads as W

from gpu_util import check, oracle_verify, sample_rows

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _plan(capfd, monkeypatch, hq, hkv, kv_len, T, route, policy):
    monkeypatch.setenv("SPARROW_LOG", "1")
    case = W.make_verify_case(8500 + len(kv_len) + T, kv_len, T, "random", DEV, hq=hq, hkv=hkv)
    ctx = B.Context.for_cache(case.k, W.SCALE, n_q_heads=hq)
    ctx.set_plan_policy(policy)
    out = torch.full_like(case.q, float("nan"))
    lse = torch.full((case.B, hq, T), float("nan"), dtype=torch.float32, device=DEV)
    capfd.readouterr()
    if route == "batch":
        B.sparrow_verify_attn_batch(ctx, B.VerifyBatch([(case.q, case.k, case.v, case.kv_len, case.parents, T, out, lse)]))
    else:
        B.sparrow_verify_attn(ctx, case.q, case.k, case.v, case.kv_len, case.parents, T, out, lse)
    torch.cuda.synchronize()
    assert ctx.last_device_status() == 0
    rows = [r for r in sample_rows(8600, case.B, T, 24) if r[2] < hq]
    check(out, lse, *oracle_verify(case, rows), rows=rows)
    line = [l for l in capfd.readouterr().err.splitlines() if l.startswith("[sparrow] verify call")][0]
    per_item, items = map(int, re.search(r"(\d+) per item, (\d+) items", line).groups())
    return per_item, items, [int(x) for x in re.findall(r"in (\d+) piece", line)]


@pytest.mark.parametrize("hq,hkv,kv_len,T,route,per_item,items", [
    (28, 4, [100] * 24, 20, "batch", 2, 96),        # short sequences in a batch: two row blocks share an item
    (28, 4, [100] * 24, 20, "single", 2, 96),       # alone: 192 items of one would take two waves
    (28, 4, [100] * 16, 20, "single", 1, 128),      # one wave of items of one
    (28, 4, [100] * 16, 20, "batch", 2, 64),
    (28, 4, [1600] * 16, 40, "batch", 1, 192),      # three row blocks of longer sequences: no half-empty items
    (32, 8, [100] * 24, 41, "batch", 2, 192),       # another head geometry
])
def test_row_blocks_per_item(hq, hkv, kv_len, T, route, per_item, items, capfd, monkeypatch):
    got = _plan(capfd, monkeypatch, hq, hkv, kv_len, T, route, B.PLAN_BALANCED)
    assert got[:2] == (per_item, items)


@pytest.mark.parametrize("hq,hkv,kv_len,T,policy,pieces", [
    (28, 4, [9000] * 8, 16, B.PLAN_THROUGHPUT, [1] * 8),                  # 32 whole units stay whole
    (28, 4, [9000, 5000] * 4, 16, B.PLAN_THROUGHPUT, [1] * 8),            # uneven ones too, with one row block
    (32, 8, [9000, 8000, 8500], 20, B.PLAN_THROUGHPUT, [1] * 3),
    (28, 4, [48 * 128 - 32] + [1000] * 5, 32, B.PLAN_THROUGHPUT, [1] * 6),        # uneven, two row blocks, 48 tiles
    (28, 4, [48 * 128 - 31] + [1000] * 5, 32, B.PLAN_THROUGHPUT, [2] + [1] * 5),  # one key more
    (28, 4, [9000], 50, B.PLAN_THROUGHPUT, [2]),                          # 12 units: 24 pieces
    (28, 4, [30000], 16, B.PLAN_THROUGHPUT, [5]),                         # 47 tiles a piece as the policy makes them
    (28, 4, [41000], 16, B.PLAN_THROUGHPUT, [7]),                         # 65 tiles: cut again
])
def test_long_pieces_of_a_batch(hq, hkv, kv_len, T, policy, pieces, capfd, monkeypatch):
    got = _plan(capfd, monkeypatch, hq, hkv, kv_len, T, "batch", policy)
    assert got[2] == pieces
