"""Row movers and window bounds at the edges of their rules: few sequences (short launch arguments) and many,
anchor lists around one, two and three rounds of a 32-way search.  Copies and integers: bit-exact."""
import random

import pytest
import torch

from paper_2602_15318_b200 import binding as B

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _context(batch, hkv, capacity):
    return B.Context(batch, capacity, hkv * capacity * 128, capacity * 128, 0.1, n_q_heads=hkv, n_kv_heads=hkv)


@pytest.mark.parametrize("batch", [1, 4, 5, 64])
def test_rows_of_few_and_many_sequences(batch):
    hkv, cap, T = 3, 40, 7
    ctx = _context(batch, hkv, cap)
    g = torch.Generator(device=DEV).manual_seed(batch)
    normal = lambda *s: torch.randn(*s, generator=g, device=DEV).bfloat16()
    k, v, k_new, v_new = normal(batch, hkv, cap, 128), normal(batch, hkv, cap, 128), normal(batch, hkv, T, 128), normal(batch, hkv, T, 128)
    kv_len = [(5 * b) % (cap - T + 1) for b in range(batch)]
    want_k, want_v = k.clone(), v.clone()
    for b, n in enumerate(kv_len):
        want_k[b, :, n:n + T], want_v[b, :, n:n + T] = k_new[b], v_new[b]
    B.sparrow_kv_append(ctx, k_new, v_new, k, v, kv_len, T)
    torch.cuda.synchronize()
    assert torch.equal(k, want_k) and torch.equal(v, want_v)

    path = torch.tensor([[1, 3, 6, -1, -1, -1, -1]] * batch, dtype=torch.int32, device=DEV)
    n_accept = torch.tensor([b % 4 for b in range(batch)], dtype=torch.int32, device=DEV)
    for b, n in enumerate(kv_len):
        for i, src in enumerate([1, 3, 6][:b % 4]):
            want_k[b, :, n + i], want_v[b, :, n + i] = k_new[b, :, src], v_new[b, :, src]
    B.sparrow_kv_keep_accepted(ctx, k, v, kv_len, path, n_accept, T)

    idx = torch.tensor([sorted(random.Random(b).sample(range(cap), 11)) for b in range(batch)], dtype=torch.int32, device=DEV)
    kc, vc = torch.zeros(batch, hkv, 16, 128, dtype=torch.bfloat16, device=DEV), torch.zeros(batch, hkv, 16, 128, dtype=torch.bfloat16, device=DEV)
    B.sparrow_compact_anchors(ctx, k, v, idx, 11, kc, vc, 16, 3)
    torch.cuda.synchronize()
    assert ctx.last_device_status() == 0
    assert torch.equal(k, want_k) and torch.equal(v, want_v)
    for b in range(batch):
        rows = idx[b].long()
        assert torch.equal(kc[b, :, 3:14], want_k[b][:, rows]) and torch.equal(vc[b, :, 3:14], want_v[b][:, rows])
    assert not kc[:, :, :3].any() and not kc[:, :, 14:].any()


@pytest.mark.parametrize("n_text", [0, 1, 31, 32, 33, 448, 1024, 1025, 5000])
def test_window_bounds_search(n_text):
    rng = random.Random(n_text)
    T_tree, T_new, batch = 9, 5, 3
    lists = [sorted(rng.sample(range(20000), n_text)) + list(range(20000 + 7 * b, 20000 + 7 * b + T_tree)) for b in range(batch)]
    anchors = torch.tensor(lists, dtype=torch.int32, device=DEV)
    ctx = _context(batch, 1, 128)
    for window in (1, 12000, 20010, 30000, 0):
        first = torch.full((batch, T_new), -1, dtype=torch.int32, device=DEV)
        B.sparrow_window_first_visible_device(ctx, anchors, n_text + T_tree, window, T_tree, T_new, first)
        assert first.tolist() == [B.sparrow_window_first_visible(x, window, T_tree, T_new)[0] for x in lists]
