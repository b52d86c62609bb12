"""What is timed: the work that a speculative decoder for video LLMs has this library do.

A step of such a decoder is: the draft model grows a tree of candidate tokens, each growth step
attending to the text-anchored rows only (projection of its inputs, append of the new K/V rows,
window attention); the target model verifies the whole tree against its long video cache, one
attention call per decoder layer; the accepted path is found and its rows are kept.  Every case is
one of these pieces, called through the package's binding exactly as such a program calls it.

Sizes are those of the repository's five workload configurations, its tests and its benchmark
(28 / 4 heads of 128, caches of 2,048 to 32,768 rows, draft blocks of 8 to 64 tokens, 28 layers,
d = 3584, a vocabulary of 151,936), and draws are spread over the ranges around them.
"""
import math

import torch

from paper_2602_15318_b200 import binding as B
from paper_2602_15318_b200 import workloads as W

DEV = "cuda:0"
D = 128
POLICIES = {"latency": B.PLAN_LATENCY, "balanced": B.PLAN_BALANCED, "throughput": B.PLAN_THROUGHPUT}


# ---- the cases -------------------------------------------------------------------------------------

def listed():
    return [
        # the draft model's attention of one step straight on the full-length cache: 448 text anchors of a
        # 1024-position window and the 8 draft rows; the smallest call, all latency
        {"name": "anchor_n456_T8", "kind": "anchor", "hq": 28, "hkv": 4, "batch": 1, "rows": 26120, "n_text": 448,
         "window": 1024, "T_tree": 8, "T_new": 8, "tree": "chain"},
        # one drafting round on a compacted cache: the anchors are compacted once, then six growth steps of
        # eight nodes each, every one an append, the window bounds and the window attention
        {"name": "draft_round_n448_6x8", "kind": "draft", "hq": 28, "hkv": 4, "batch": 1, "rows": 26112, "n_text": 448,
         "window": 1024, "T_new": 8, "steps": 6},
        # one layer's verification in a short conversation: 2,048 rows, a chain of 8
        {"name": "verify_kv2048_T8", "kind": "verify", "hq": 28, "hkv": 4, "batch": 1, "kv": 2048, "T": 8,
         "tree": "chain", "policy": "balanced"},
        # one layer's verification of a long video: 26,112 rows, a chain of 16, the library's defaults
        {"name": "verify_kv26112_T16", "kind": "verify", "hq": 28, "hkv": 4, "batch": 1, "kv": 26112, "T": 16,
         "tree": "chain", "policy": "balanced"},
        # the largest draft tree, 64 nodes, one call at a time under the latency policy
        {"name": "verify_kv16384_T64_tree", "kind": "verify", "hq": 28, "hkv": 4, "batch": 1, "kv": 16384, "T": 64,
         "tree": "random", "policy": "latency"},
        # another head geometry, odd ragged lengths and an odd tree: three sequences, 32 / 8 heads
        {"name": "verify_b3_kv9001_T23_g4", "kind": "verify", "hq": 32, "hkv": 8, "batch": 3, "kv": 9001, "T": 23,
         "tree": "random", "policy": "balanced"},
        # a whole model's verification of a chain of 16, enqueued in one call: 28 layers, 26,112 rows each
        {"name": "layers28_kv26112_T16", "kind": "layers", "hq": 28, "hkv": 4, "batch": 1, "kv": 26112, "T": 16,
         "tree": "chain", "policy": "throughput", "layers": 28},
        # the same for eight ragged sequences with trees of 32: the largest work, 15 GB of cache
        {"name": "layers28_b8_kv32768_T32", "kind": "layers", "hq": 28, "hkv": 4, "batch": 8, "kv": 32768, "T": 32,
         "tree": "random", "policy": "throughput", "layers": 28},
        # one layer's verification for a caller with host buffers: pinned inputs in, results back, synchronised
        {"name": "step_host_kv26112_T16", "kind": "step_host", "hq": 28, "hkv": 4, "batch": 1, "kv": 26112, "T": 16,
         "tree": "chain", "policy": "latency"},
        # the draft model's input projection for a 48-node tree of a 7B-class model
        {"name": "hsr_M48_d3584", "kind": "hsr", "M": 48, "d": 3584, "d_out": 3584, "bias": True},
        # acceptance at temperature 1 of a 32-node tree over a full vocabulary
        {"name": "accept_T32_V151936", "kind": "accept", "batch": 1, "T": 32, "vocab": 151936},
        # what surrounds a verification at temperature 0: every layer's new rows are appended, the accepted
        # path is found, every layer keeps the accepted rows
        {"name": "commit_28_layers_T32", "kind": "commit", "hq": 28, "hkv": 4, "batch": 1, "kv": 2048, "T": 32, "layers": 28},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["anchor", "draft", "verify", "verify", "verify", "layers", "layers", "step_host", "hsr", "accept", "commit"])
    hq, hkv = rng.choice([(28, 4), (28, 4), (28, 4), (32, 8), (32, 4), (12, 4), (8, 8), (16, 1)])
    tree = rng.choice(["chain", "random"])
    if kind == "anchor":
        T_tree = rng.randint(1, 64)
        n_text = _log(rng, 40, 6000)
        return {"kind": kind, "hq": hq, "hkv": hkv, "batch": rng.randint(1, 4), "rows": 26112 + rng.randint(0, 2000), "n_text": n_text,
                "window": rng.choice([0, 512, 1024, 4096]), "T_tree": T_tree, "T_new": rng.randint(1, T_tree), "tree": "random"}
    if kind == "draft":
        T_new = rng.randint(1, 10)
        return {"kind": kind, "hq": hq, "hkv": hkv, "batch": rng.randint(1, 4), "rows": 26112 + rng.randint(0, 2000),
                "n_text": _log(rng, 40, 6000), "window": rng.choice([0, 512, 1024, 4096]), "T_new": T_new, "steps": rng.randint(2, 6)}
    if kind == "verify":
        return {"kind": kind, "hq": hq, "hkv": hkv, "batch": rng.randint(1, 8), "kv": _log(rng, 300, 32768), "T": rng.randint(1, 64),
                "tree": tree, "policy": rng.choice(["balanced", "balanced", "latency", "throughput"])}
    if kind == "layers":
        batch, layers = rng.choice([1, 1, 2, 4]), rng.randint(8, 28)
        most = min(32768, 18000000 // (batch * layers * hkv))         # no more than the largest listed case reads
        return {"kind": kind, "hq": hq, "hkv": hkv, "batch": batch, "kv": _log(rng, 1000, most), "T": rng.randint(1, 64),
                "tree": tree, "policy": rng.choice(["balanced", "latency", "throughput"]), "layers": layers}
    if kind == "step_host":
        return {"kind": kind, "hq": hq, "hkv": hkv, "batch": rng.randint(1, 4), "kv": _log(rng, 1000, 32768), "T": rng.randint(1, 64),
                "tree": tree, "policy": rng.choice(["balanced", "latency"])}
    if kind == "hsr":
        d = 64 * _log(rng, 12, 80)
        return {"kind": kind, "M": rng.randint(1, 64), "d": d, "d_out": rng.choice([128 * _log(rng, 8, 40), 128 * max(1, d // 128)]),
                "bias": rng.random() < 0.5}
    if kind == "accept":
        return {"kind": kind, "batch": rng.choice([1, 2, 3, 4, 8]), "T": rng.randint(4, 64), "vocab": _log(rng, 20000, 260000)}
    return {"kind": kind, "hq": hq, "hkv": hkv, "batch": rng.randint(1, 8), "kv": rng.randint(200, 1000), "T": rng.randint(1, 64),
            "layers": rng.randint(4, 28)}


# ---- inputs ----------------------------------------------------------------------------------------

def _lengths(case):
    """Prefix lengths: the longest first, the others spread between a quarter of it and all of it."""
    kv = case["kv"]
    return [kv - int((kv - kv // 4) * ((0.381966 * i) % 1.0)) for i in range(case["batch"])]


def _normal(g, *shape):
    return torch.empty(shape, dtype=torch.bfloat16, device=DEV).normal_(generator=g)


def _trees(seed, batch, T, tree):
    rows = [W.chain_parents(T) if tree == "chain" else W.random_tree_parents(seed + 31 * b, 4, T) for b in range(batch)]
    return torch.tensor(rows, dtype=torch.int32, device=DEV)


def _attention_inputs(case, g, capacity, lens, q_tokens):
    """q, K and V of one layer: normal values, and one in a hundred prefix keys drawn towards its head
    group's queries, as the few tokens that a real attention pattern concentrates on."""
    b, hq, hkv = case["batch"], case["hq"], case["hkv"]
    q = _normal(g, b, q_tokens, hq, D)
    k, v = _normal(g, b, hkv, capacity, D), _normal(g, b, hkv, capacity, D)
    n = max(1, min(lens) // 100)
    at = torch.randint(0, max(1, min(lens)), (b, hkv, n), generator=g, device=DEV)
    towards = q.float().view(b, q_tokens, hkv, hq // hkv, D).mean(dim=(1, 3))
    at = at[..., None].expand(b, hkv, n, D)
    k.scatter_(2, at, (k.gather(2, at).float() + 2.0 * towards[:, :, None, :]).to(torch.bfloat16))
    return q, k, v


def _outputs(b, T, hq):
    return (torch.zeros((b, T, hq, D), dtype=torch.bfloat16, device=DEV), torch.zeros((b, hq, T), dtype=torch.float32, device=DEV))


def _context(case, cache):
    return B.Context.for_cache(cache, W.SCALE, n_q_heads=case["hq"])


def _anchors(g, case, n_extra):
    """Text anchors (sorted positions of the prefix, dense at its end as under a window) and the rows after it."""
    rows, n = case["rows"] - 64, case["n_text"]
    out = []
    for _ in range(case["batch"]):
        near = torch.randperm(min(rows, 2 * n), generator=g, device=DEV)[:n] + max(0, rows - 2 * n)
        out.append(torch.cat([near.sort().values, torch.arange(rows, rows + n_extra, device=DEV)]))
    return torch.stack(out).to(torch.int32).contiguous()


def prepare(case, seed):
    g = torch.Generator(device=DEV).manual_seed(seed)
    s = {"kind": case["kind"], "case": case}
    kind = case["kind"]
    if kind in ("verify", "layers", "step_host"):
        lens, T = _lengths(case), case["T"]
        s["kv_len"], cap = lens, max(lens) + 64
        s["parents"] = _trees(seed, case["batch"], T, case["tree"])
        layers = [_attention_inputs(case, g, cap, lens, T) for _ in range(case.get("layers", 1))]
        s["ctx"] = _context(case, layers[0][1])
        s["ctx"].set_plan_policy(POLICIES[case["policy"]])
        s["layers"] = layers
        if kind == "step_host":
            q, k, v = layers[0]
            new = [torch.stack([x[b, :, n:n + T] for b, n in enumerate(lens)]).cpu().pin_memory() for x in (k, v)]
            s["q_host"], s["k_new"], s["v_new"] = q.cpu().pin_memory(), new[0], new[1]
            s["parents_host"] = s["parents"].cpu().pin_memory()
            s["out"], s["lse"] = (x.cpu().pin_memory() for x in _outputs(case["batch"], T, case["hq"]))
        else:
            s["outs"] = [_outputs(case["batch"], T, case["hq"]) for _ in layers]
            if kind == "layers":
                s["calls"] = B.VerifyBatch([(q, k, v, lens, s["parents"], T, o, l) for (q, k, v), (o, l) in zip(layers, s["outs"])])
    elif kind == "anchor":
        s["anchors"] = _anchors(g, case, case["T_tree"])
        s["n_anchor"] = case["n_text"] + case["T_tree"]
        s["q"], s["k"], s["v"] = _attention_inputs(case, g, case["rows"], [case["rows"]], case["T_new"])
        s["parents"] = _trees(seed, case["batch"], case["T_tree"], case["tree"])
        s["ctx"] = _context(case, s["k"])
        s["out"], s["lse"] = _outputs(case["batch"], case["T_new"], case["hq"])
    elif kind == "draft":
        b, n_text, T_new, steps = case["batch"], case["n_text"], case["T_new"], case["steps"]
        nodes = T_new * steps
        s["q"], s["k"], s["v"] = _attention_inputs(case, g, case["rows"], [case["rows"]], T_new)
        anchors = _anchors(g, case, nodes)
        parents = _trees(seed, b, nodes, "random")
        s["text"] = anchors[:, :n_text].contiguous()
        s["capacity"] = n_text + 64
        s["kc"], s["vc"] = (torch.zeros((b, case["hkv"], s["capacity"], D), dtype=torch.bfloat16, device=DEV) for _ in range(2))
        s["ctx"], s["draft_ctx"] = _context(case, s["k"]), _context(case, s["kc"])
        s["draft_ctx"].set_plan_policy(B.PLAN_LATENCY)
        s["steps"] = []
        for i in range(steps):
            grown = (i + 1) * T_new
            s["steps"].append({"grown": grown, "anchors": anchors[:, :n_text + grown].contiguous(), "parents": parents[:, :grown].contiguous(),
                               "q": s["q"] if i == 0 else _normal(g, b, T_new, case["hq"], D),
                               "k_new": _normal(g, b, case["hkv"], T_new, D), "v_new": _normal(g, b, case["hkv"], T_new, D),
                               "first": torch.zeros((b, T_new), dtype=torch.int32, device=DEV), "out": _outputs(b, T_new, case["hq"])})
    elif kind == "hsr":
        d, d_out = case["d"], case["d_out"]
        s["e"], s["h"] = _normal(g, case["M"], d), _normal(g, case["M"], d)
        s["w"] = _normal(g, d_out, 2 * d).mul_((2 * d) ** -0.5)
        s["bias"] = _normal(g, d_out) if case["bias"] else None
        s["z"] = torch.zeros((case["M"], d_out), dtype=torch.bfloat16, device=DEV)
        s["ctx"] = B.Context(1, 128, 4 * 128 * D, 128 * D, W.SCALE)
    elif kind == "accept":
        b, T, V = case["batch"], case["T"], case["vocab"]
        parents = _trees(seed, b, T, "random")
        logits = torch.empty((b, T + 1, V), device=DEV).normal_(generator=g).mul_(3.0)
        draft = logits + torch.empty_like(logits).normal_(generator=g).mul_(0.7)
        s["p"], s["q"] = torch.softmax(logits, -1), torch.softmax(draft, -1)
        # children of a node: distinct tokens drawn from its draft row, the i-th child the i-th of them
        noise = torch.empty_like(draft).exponential_(generator=g).log_().neg_()
        likely = (draft + noise).topk(4, dim=-1).indices.cpu()
        tokens, par = torch.zeros((b, T), dtype=torch.int32), parents.cpu()
        for i in range(b):
            born = {}
            for t, p in enumerate(par[i].tolist()):
                tokens[i, t] = likely[i, p + 1, born.get(p, 0)]
                born[p] = born.get(p, 0) + 1
        s["tokens"], s["parents"] = tokens.to(DEV), parents
        s["u_node"], s["u_bonus"] = (torch.randint(-2 ** 31, 2 ** 31, (b, n), generator=g, device=DEV, dtype=torch.int64).to(torch.int32)
                                     for n in (T, T + 1))
        s["ctx"] = B.Context(b, 128, 4 * 128 * D, 128 * D, W.SCALE)
        s["path"] = torch.zeros((b, T), dtype=torch.int32, device=DEV)
        s["n_accept"], s["bonus"] = (torch.zeros(b, dtype=torch.int32, device=DEV) for _ in range(2))
    else:
        b, T, n = case["batch"], case["T"], case["layers"]
        s["kv_len"] = _lengths(case)
        s["k"], s["v"] = (_normal(g, n, b, case["hkv"], case["kv"] + 64, D) for _ in range(2))
        s["k_new"], s["v_new"] = (_normal(g, n, b, case["hkv"], T, D) for _ in range(2))
        s["layers"] = list(zip(s["k"], s["v"], s["k_new"], s["v_new"]))
        s["ctx"] = _context(case, s["k"][0])
        parents = _trees(seed, b, T, "random")
        nxt = torch.randint(0, 151936, (b, T + 1), generator=g, device=DEV, dtype=torch.int32)
        right = nxt.gather(1, (parents + 1).long())                 # what the target says after each node's parent
        wrong = torch.rand((b, T), generator=g, device=DEV) < 0.35
        s["parents"], s["next"], s["tokens"] = parents, nxt, torch.where(wrong, right ^ 1, right).contiguous()
        s["path"] = torch.zeros((b, T), dtype=torch.int32, device=DEV)
        s["n_accept"], s["bonus"] = (torch.zeros(b, dtype=torch.int32, device=DEV) for _ in range(2))
    return s


# ---- one pass --------------------------------------------------------------------------------------

def run(s):
    kind, case = s["kind"], s["case"]
    if kind == "verify":
        (q, k, v), (out, lse) = s["layers"][0], s["outs"][0]
        B.sparrow_verify_attn(s["ctx"], q, k, v, s["kv_len"], s["parents"], case["T"], out, lse)
        return out, lse
    if kind == "layers":
        B.sparrow_verify_attn_batch(s["ctx"], s["calls"])
        return s["outs"]
    if kind == "step_host":
        _, k, v = s["layers"][0]
        B.sparrow_verify_step_host(s["ctx"], s["q_host"], s["k_new"], s["v_new"], k, v, s["kv_len"], s["parents_host"], case["T"],
                                   s["out"], s["lse"])
        return s["out"], s["lse"]
    if kind == "anchor":
        if case["tree"] == "chain":
            B.sparrow_anchor_attn(s["ctx"], s["q"], s["k"], s["v"], s["anchors"], s["n_anchor"], case["window"], case["T_new"], s["out"], s["lse"])
        else:
            B.sparrow_anchor_attn_tree(s["ctx"], s["q"], s["k"], s["v"], s["anchors"], s["n_anchor"], case["window"], s["parents"],
                                       case["T_tree"], case["T_new"], s["out"], s["lse"])
        return s["out"], s["lse"]
    if kind == "draft":
        b, n_text, T_new, ctx = case["batch"], case["n_text"], case["T_new"], s["draft_ctx"]
        B.sparrow_compact_anchors(s["ctx"], s["k"], s["v"], s["text"], n_text, s["kc"], s["vc"], s["capacity"], 0)
        for st in s["steps"]:
            B.sparrow_kv_append(ctx, st["k_new"], st["v_new"], s["kc"], s["vc"], [n_text + st["grown"] - T_new] * b, T_new)
            B.sparrow_window_first_visible_device(ctx, st["anchors"], n_text + st["grown"], case["window"], st["grown"], T_new, st["first"])
            B.sparrow_verify_attn_window(ctx, st["q"], s["kc"], s["vc"], [n_text] * b, st["parents"], st["grown"], T_new, st["first"], None,
                                         *st["out"])
        return [st["out"] for st in s["steps"]], s["kc"], s["vc"]
    if kind == "hsr":
        B.sparrow_hsr_fuse(s["ctx"], s["e"], s["h"], s["w"], s["bias"], s["z"])
        return s["z"]
    if kind == "accept":
        B.sparrow_accept_sample(s["ctx"], s["tokens"], s["parents"], s["p"], s["q"], s["u_node"], s["u_bonus"], case["vocab"], case["T"],
                                s["path"], s["n_accept"], s["bonus"])
        return s["path"], s["n_accept"], s["bonus"]
    ctx, T = s["ctx"], case["T"]
    for k, v, k_new, v_new in s["layers"]:
        B.sparrow_kv_append(ctx, k_new, v_new, k, v, s["kv_len"], T)
    B.sparrow_accept_greedy(ctx, s["tokens"], s["parents"], s["next"], T, s["path"], s["n_accept"], s["bonus"])
    for k, v, _, _ in s["layers"]:
        B.sparrow_kv_keep_accepted(ctx, k, v, s["kv_len"], s["path"], s["n_accept"], T)
    return s["k"], s["v"], s["path"], s["n_accept"], s["bonus"]


# ---- what a pass cannot do without -----------------------------------------------------------------

def _attention_work(case, keys, T):
    """keys: rows of K and V per KV head, summed over the sequences; T query tokens each."""
    io = case["batch"] * T * case["hq"] * (2 * D * 2 + 4)
    return {"bytes": keys * case["hkv"] * D * 2 * 2 + io, "flops": 4 * D * keys * case["hq"] * T}


def work(case):
    kind = case["kind"]
    if kind in ("verify", "layers", "step_host"):
        w = _attention_work(case, sum(_lengths(case)) + case["batch"] * case["T"], case["T"])
        return {m: x * case.get("layers", 1) for m, x in w.items()}
    if kind == "anchor":
        return _attention_work(case, case["batch"] * (case["n_text"] + case["T_tree"]), case["T_new"])
    if kind == "draft":
        per = [_attention_work(case, case["batch"] * (case["n_text"] + (i + 1) * case["T_new"]), case["T_new"]) for i in range(case["steps"])]
        rows = case["batch"] * case["hkv"] * D * 2 * 2 * 2 * (case["n_text"] + case["steps"] * case["T_new"])
        return {"bytes": rows + sum(w["bytes"] for w in per), "flops": sum(w["flops"] for w in per)}
    if kind == "hsr":
        M, d, d_out = case["M"], case["d"], case["d_out"]
        return {"bytes": 2 * (2 * d * d_out + 2 * M * d + M * d_out + d_out), "flops": 4 * M * d * d_out}
    if kind == "accept":
        # the target's and the draft's row at every node of the walk: two or three accepted nodes, and the stop
        return {"bytes": case["batch"] * 7 * 4 * case["vocab"], "flops": 0}
    # appended rows: read and written; kept rows (about a fifth of the tree): read and written
    row = case["batch"] * case["hkv"] * D * 2 * 2
    return {"bytes": case["layers"] * row * 2 * (case["T"] + case["T"] // 5), "flops": 0}


def tolerance(case):
    if case["kind"] in ("accept", "commit"):
        return "exact"
    if case["kind"] == "hsr":
        return {"rel": 6.5e-3, "max": 1.6e-2}       # one rounding of z to bf16: 1.6e-3 and 3.9e-3 against 64-bit sums
    # P and the output are rounded to bf16 (2^-9 relative each), the rest is 32-bit: 2.2e-3 to 2.4e-3, and 8e-3 to
    # 1e-2 for the largest, against the same sums in 64 bits
    return {"rel": 9e-3, "max": 4e-2}
