"""Single calls that share the GPU with no other call: how their pieces are merged depends on sizes (one
piece, a thread-block cluster per unit, the workspace).  Sizes at the edges of those rules, against the
oracle; tolerances as everywhere (gpu_util)."""
import pytest
import torch

import oracle
from paper_2602_15318_b200 import binding as B
from paper_2602_15318_b200 import workloads as W

from gpu_util import check, oracle_anchor, oracle_verify, run_anchor, run_verify

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("hq,hkv,kv_len,T,tree", [
    (28, 4, [120], 8, "chain"),             # exactly one tile: no merge
    (28, 4, [121], 8, "random"),            # one key more
    (28, 4, [1000], 18, "chain"),           # the largest draft block of one row block
    (28, 4, [4096 - 16], 16, "random"),     # 32 tiles: the longest pieces a cluster of 16 takes
    (28, 4, [4096 - 15], 16, "random"),     # 33 tiles: through the workspace
    (28, 4, [500], 36, "random"),           # 252 rows: shares that straddle the two row blocks
    (28, 4, [500], 64, "chain"),            # two row groups, a chain as deep as a tree gets
    (28, 4, [2048 - 40], 40, "random"),     # 16 tiles, two row blocks
    (28, 4, [2049 - 40], 40, "random"),     # 17 tiles
    (4, 4, [700], 1, "chain"),              # one row per unit: most CTAs of a cluster finish nothing
    (16, 1, [1500], 64, "random"),          # 16 query heads per KV head, four row groups
    (8, 8, [1100], 9, "chain"),             # 9 rows in a cluster: one or two for each CTA to merge
    (28, 4, [26000], 3, "chain"),           # 84 rows through the workspace, one for each finisher
    (28, 4, [9000], 30, "random"),          # 840 rows, six or fewer for each
    (28, 4, [130, 2000, 700], 12, "random"),  # ragged lengths in clusters of two
    (28, 4, [100] * 40, 20, "random"),      # more units than SMs
])
def test_verify_alone(hq, hkv, kv_len, T, tree):
    case = W.make_verify_case(7100 + hq + T + kv_len[0], kv_len, T, tree, DEV, hq=hq, hkv=hkv)
    ctx = B.Context.for_cache(case.k, W.SCALE, n_q_heads=hq)
    ref = oracle_verify(case)
    for _ in range(2):                      # (the second call follows the first without a synchronisation of its own)
        out, lse, _ = run_verify(case, ctx)
        check(out, lse, *ref)


@pytest.mark.parametrize("hq,hkv,kv_len,T,tree", [
    (28, 4, [32 * 128 - 7], 8, "chain"),      # sixteen pieces, one of them of three tiles: only its CTA uses the ring's last stage
    (28, 4, [33 * 128], 16, "random"),        # two of three tiles
    (28, 4, [40 * 128 + 1], 18, "random"),    # three tiles, and one with a few keys
    (28, 4, [16 * 6 * 128 - 9], 9, "chain"),  # six tiles each: the ring goes round twice
    (28, 4, [3000], 64, "random"),            # sixteen units
    (28, 4, [1500, 700], 36, "random"),       # two row blocks, more tiles than their ring has stages
    (28, 4, [2500] * 8, 33, "random"),
    (8, 8, [6000, 900, 3000], 20, "random"),  # ragged: some pieces leave the last stage alone
    (16, 1, [5000], 20, "random"),
])
def test_long_pieces_in_clusters_repeat_bit_for_bit(hq, hkv, kv_len, T, tree):
    """Pieces that use the ring stage which their peers' rows come to."""
    case = W.make_verify_case(7500 + hq + T + kv_len[0], kv_len, T, tree, DEV, hq=hq, hkv=hkv)
    ctx = B.Context.for_cache(case.k, W.SCALE, n_q_heads=hq)
    out, lse, _ = run_verify(case, ctx)
    check(out, lse, *oracle_verify(case))
    for _ in range(20):
        again, lse_again, _ = run_verify(case, ctx)
        assert torch.equal(out, again) and torch.equal(lse, lse_again)


def test_verify_alone_back_to_back_and_in_front_of_a_batch():
    """Lone calls of different kinds (cluster, workspace, one piece) and a batch that overlaps its own calls,
    enqueued without synchronisation on one context: every result its own, in the batch bit for bit."""
    cap = 9000 + 64
    cases = [W.make_verify_case(7300 + i, [kv], T, tree, DEV, capacity=cap)
             for i, (kv, T, tree) in enumerate([(700, 8, "chain"), (9000, 16, "random"), (60, 12, "random"), (1500, 33, "chain")])]
    refs = [oracle_verify(c) for c in cases]
    ctx = B.Context.for_cache(cases[0].k, W.SCALE)
    new = lambda c: (torch.full_like(c.q, float("nan")), torch.full((1, W.HQ, c.T), float("nan"), dtype=torch.float32, device=DEV))
    results, batched = [], []
    for rep in range(4):
        for c in cases:
            out, lse = new(c)
            B.sparrow_verify_attn(ctx, c.q, c.k, c.v, c.kv_len, c.parents, c.T, out, lse)
            results.append((out, lse))
        outs = [new(c) for c in cases]
        B.sparrow_verify_attn_batch(ctx, B.VerifyBatch([(c.q, c.k, c.v, c.kv_len, c.parents, c.T, o, l) for c, (o, l) in zip(cases, outs)]))
        batched.append(outs)
    torch.cuda.synchronize()
    assert ctx.last_device_status() == 0
    for i, (out, lse) in enumerate(results):
        check(out, lse, *refs[i % len(cases)])
    for outs in batched:
        for (o, l), (wo, wl), ref in zip(outs, batched[0], refs):
            check(o, l, *ref)
            assert torch.equal(o, wo) and torch.equal(l, wl)


@pytest.mark.parametrize("n_text,T,batch", [
    (56, 8, 1),                             # exactly one gathered tile
    (57, 8, 1),                             # two pieces
    (16 * 64 - 8, 8, 1),                    # sixteen pieces
    (16 * 64 - 7, 8, 1),                    # seventeen tiles
    (300, 40, 1),                           # three row groups, the last one short
    (200, 1, 3),
])
def test_anchored_pieces(n_text, T, batch):
    idx = list(range(40, 40 + n_text)) + list(range(2000, 2000 + T))
    case = W.make_anchor_case(7500 + n_text + T, idx, 0, T, batch, DEV)
    out, lse, _ = run_anchor(case)
    check(out, lse, *oracle_anchor(case))


@pytest.mark.parametrize("n_text,T_tree,T_new,window", [
    (0, 1, 1, 0),                           # a tile that is a tree of one node
    (63, 1, 1, 0),                          # a node in a tile's last column
    (64, 64, 64, 0),                        # a whole tile of nodes, from its first column
    (65, 64, 64, 0),                        # 63 nodes in one tile, one in the next
    (127, 64, 9, 40),                       # one node in a tile, 63 in the next; text of the tile before outside the window
    (100, 64, 33, 70),                      # nodes in two tiles, the window's end beside them
    (16 * 64 - 32, 64, 20, 300),            # seventeen tiles, merged by the combine kernel
    (30, 33, 2, 1),                         # a window that leaves no text
])
def test_gathered_trees_across_tiles(n_text, T_tree, T_new, window):
    """Gathered keys are masked by position in front of the draft tree and by ancestors from the column of its first node on."""
    idx = list(range(40, 40 + n_text)) + list(range(2000, 2000 + T_tree))
    case = W.make_anchor_case(7600 + n_text + T_tree, idx, window + 2000 - 40 - n_text if window else 0, T_tree, 2, DEV)
    parents = torch.tensor([W.random_tree_parents(7650 + b + n_text, 99, T_tree) for b in range(2)], dtype=torch.int32, device=DEV)
    q = case.q[:, T_tree - T_new:].contiguous()
    ctx = B.Context.for_cache(case.k, W.SCALE)
    out, lse = torch.full_like(q, float("nan")), torch.full((2, W.HQ, T_new), float("nan"), dtype=torch.float32, device=DEV)
    B.sparrow_anchor_attn_tree(ctx, q, case.k, case.v, case.anchor_idx, case.n_anchor, case.window, parents, T_tree, T_new, out, lse)
    torch.cuda.synchronize()
    assert ctx.last_device_status() == 0
    check(out, lse, *oracle.anchor_attn_tree(W.bf16_bits(q), W.bf16_bits(case.k), W.bf16_bits(case.v), case.anchor_idx.cpu().numpy(),
                                             case.window, parents.cpu().numpy(), W.SCALE))


@pytest.mark.parametrize("hq,hkv,kv_len,T", [
    (32, 8, [48 * 128 - 12] * 3, 12),       # one piece of 48 tiles a unit
    (32, 8, [48 * 128 - 11, 300, 6000], 12),  # ragged lengths, 49 tiles the longest
    (28, 4, [2000], 19),                    # two row blocks in items of one
    (28, 4, [30000], 36),                   # two row blocks in items of two
    (28, 4, [10000], 37),                   # three
    (16, 1, [900], 64),                     # eight
])
def test_split_of_calls_in_a_batch(hq, hkv, kv_len, T):
    """Two calls that overlap in a batch, where their pieces and row blocks are chosen differently from a lone call's."""
    cases = [W.make_verify_case(7700 + T + i, kv_len, T, "random", DEV, hq=hq, hkv=hkv) for i in range(2)]
    ctx = B.Context.for_cache(cases[0].k, W.SCALE, n_q_heads=hq)
    ctx.set_plan_policy(B.PLAN_THROUGHPUT)
    outs = [(torch.full_like(c.q, float("nan")), torch.full((len(kv_len), hq, T), float("nan"), dtype=torch.float32, device=DEV))
            for c in cases]
    B.sparrow_verify_attn_batch(ctx, B.VerifyBatch([(c.q, c.k, c.v, c.kv_len, c.parents, c.T, o, l) for c, (o, l) in zip(cases, outs)]))
    torch.cuda.synchronize()
    assert ctx.last_device_status() == 0
    for c, (o, l) in zip(cases, outs):
        check(o, l, *oracle_verify(c))
