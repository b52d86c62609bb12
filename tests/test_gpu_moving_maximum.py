"""Rows whose largest score keeps growing along the keys: the softmax's reference has to move in the middle of a piece,
in either half of a tile, with the halves of a row at different tiles, and by more than an fp32 exponent holds."""
import pytest
import torch

from paper_2602_15318_b200 import binding as B
from paper_2602_15318_b200 import workloads as W

from gpu_util import check, oracle_verify

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
KV = 1800

# Where one key holds a row's whole weight nothing averages out.  Its P is 1 and exact (the reference is its score), so what is left
# for |v| < 4 is the rounding of the output to bf16, 2^-7, and of a partial row to fp16, 2^-10: 8.8e-3 of TOL_OUT's 1e-2.
V_MOST = 4.0 - 2.0 ** -6


def _profile(kind, n):
    """Added to every key's first component; one unit is about 2^1 in the weight of a row with +8 there."""
    j = torch.arange(n)
    tile, low = j // 128, (j % 128) < 64
    if kind == "stairs": return 20.0 * tile                                # every tile, both halves at once
    if kind == "low": return torch.where(low, 24.0 * (tile // 2), 0.0)     # the lower halves only, every other tile
    if kind == "high": return torch.where(low, 0.0, 24.0 * (tile // 3))    # the upper halves only
    if kind == "turns": return torch.where(low, 18.0 * tile, 18.0 * tile + 9.0)
    if kind == "cliff": return torch.where(j == n - 300, 250.0, 0.0)       # one key, by more than 2^126
    if kind == "falls": return -20.0 * tile                                # (rows with the other sign climb)
    if kind == "late": return torch.where(j >= n - 20, 60.0, 0.0)          # among the last keys
    return torch.zeros(n)


def _case(T, hq, hkv):
    kinds = ["stairs", "low", "high", "turns", "cliff", "falls", "late", "none"]
    case = W.make_verify_case(8300 + T, [KV] * len(kinds), T, "random", DEV, hq=hq, hkv=hkv)
    for b, kind in enumerate(kinds):
        case.k[b, :, :KV + T, 0] = _profile(kind, KV + T).to(DEV, torch.bfloat16)
    sign = torch.tensor([8.0, 0.0, -8.0], device=DEV)
    rows = torch.arange(hq, device=DEV)[None, :] + torch.arange(T, device=DEV)[:, None]       # neighbours differ
    case.q[..., 0] = sign[rows % 3].to(torch.bfloat16)
    case.v.clamp_(-V_MOST, V_MOST)
    return case


def _new(case):
    return torch.full_like(case.q, float("nan")), torch.full((case.B, case.q.shape[2], case.T), float("nan"), dtype=torch.float32, device=DEV)


def _call(ctx, case, outs, alone):
    if alone:
        for out, lse in outs:
            B.sparrow_verify_attn(ctx, case.q, case.k, case.v, case.kv_len, case.parents, case.T, out, lse)
    else:                                                                  # (pieces of up to 15 tiles)
        B.sparrow_verify_attn_batch(ctx, B.VerifyBatch([(case.q, case.k, case.v, case.kv_len, case.parents, case.T, out, lse) for out, lse in outs]))
    torch.cuda.synchronize()
    assert ctx.last_device_status() == 0


@pytest.mark.parametrize("alone", [False, True])
@pytest.mark.parametrize("T,hq,hkv", [(16, 28, 4), (30, 28, 4), (3, 8, 8)])
def test_growing_scores(T, hq, hkv, alone):
    case = _case(T, hq, hkv)
    ctx = B.Context.for_cache(case.k, W.SCALE, n_q_heads=hq)
    ctx.set_plan_policy(B.PLAN_THROUGHPUT)
    out, lse = _new(case)
    _call(ctx, case, [(out, lse)], alone)
    check(out, lse, *oracle_verify(case))


@pytest.mark.parametrize("alone", [False, True])
@pytest.mark.parametrize("T,hq,hkv", [(16, 28, 4), (3, 8, 8)])
def test_growing_scores_repeat_bit_for_bit(T, hq, hkv, alone):
    """The warps that share a row come to its tiles in an order that differs from call to call; the bits do not."""
    case = _case(T, hq, hkv)
    ctx = B.Context.for_cache(case.k, W.SCALE, n_q_heads=hq)
    ctx.set_plan_policy(B.PLAN_THROUGHPUT)
    outs = [_new(case) for _ in range(24)]
    for _ in range(4):
        _call(ctx, case, outs, alone)
        for out, lse in outs[1:]:
            assert torch.equal(out.view(torch.int16), outs[0][0].view(torch.int16)) and torch.equal(lse, outs[0][1])


@pytest.mark.parametrize("alone", [False, True])
@pytest.mark.parametrize("T,hq,hkv", [(16, 28, 4), (30, 28, 4), (3, 8, 8)])
def test_one_key_far_above_the_rest(T, hq, hkv, alone):
    """One late key that exceeds everything before it by 2^9 to 2^15, by every fraction: it has a row's whole weight, and P
    must not round it."""
    n = 32
    case = W.make_verify_case(8400 + T, [KV] * n, T, "random", DEV, hq=hq, hkv=hkv)
    case.q.mul_(0.125)                                                     # (the other keys' scores: 2^(+- 0.6) of a row's largest)
    case.q[..., 0] = 8.0
    case.k[..., 0] = 0.0
    unit = 8.0 * W.SCALE * 1.4426950408889634                              # of the key's first component, in log2
    for b in range(n):
        at = 900 + 29 * b                                                  # (either half of a tile, any tile of a piece)
        case.k[b, :, at] = 0.0
        case.k[b, :, at, 0] = (9.6 + 6.0 * b / n) / unit
    case.v.clamp_(-V_MOST, V_MOST)
    ctx = B.Context.for_cache(case.k, W.SCALE, n_q_heads=hq)
    ctx.set_plan_policy(B.PLAN_THROUGHPUT)
    out, lse = _new(case)
    _call(ctx, case, [(out, lse)], alone)
    check(out, lse, *oracle_verify(case))
