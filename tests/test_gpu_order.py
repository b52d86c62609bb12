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


# ---- a predecessor that lets its dependents start at once and writes an input of theirs late ------------------

def _normal(gen, *shape):
    return torch.empty(shape, dtype=torch.bfloat16, device=DEV).normal_(generator=gen)


def _ints(rows):
    return torch.tensor(rows, dtype=torch.int32, device=DEV)


def _problem(entry):
    """(context, inputs by name, prepare): prepare(inputs) allocates the outputs and returns them with the call itself,
    so that nothing else comes between the late kernel and the call.  Inputs are device tensors."""
    gen = torch.Generator(device=DEV).manual_seed(8600)
    T, kv, D, H, HK = 16, 3000, W.D, W.HQ, W.HKV
    cap = 3100
    k, v = _normal(gen, 1, HK, cap, D), _normal(gen, 1, HK, cap, D)
    ctx = B.Context.for_cache(k, W.SCALE)
    q = _normal(gen, 1, T, H, D)
    tree = _ints([W.random_tree_parents(8601, 3, T)])
    new_out = lambda: (torch.full((1, T, H, D), float("nan"), dtype=torch.bfloat16, device=DEV),
                       torch.full((1, H, T), float("nan"), dtype=torch.float32, device=DEV))
    anchors = _ints([list(range(40, 40 + 300)) + list(range(2000, 2000 + T))])
    n_anchor = 300 + T
    if entry in ("verify", "verify_short", "verify_window"):
        n = 900 if entry == "verify_short" else kv                       # in clusters; through the workspace
        first = _ints([[100 + 10 * t for t in range(T)]])
        ins = {"q": q, "k": k, "v": v, "parents": tree}
        if entry == "verify_window":
            ins["first"] = first

        def prepare(x):
            o, l = new_out()
            if entry == "verify_window":
                return (o, l), lambda: B.sparrow_verify_attn_window(ctx, x["q"], x["k"], x["v"], [n], x["parents"], T, T, x["first"], None, o, l)
            return (o, l), lambda: B.sparrow_verify_attn(ctx, x["q"], x["k"], x["v"], [n], x["parents"], T, o, l)
        return ctx, ins, prepare
    if entry == "step_host":
        k_new, v_new = (_normal(gen, 1, HK, T, D).cpu().pin_memory() for _ in range(2))
        q_host, par_host = q.cpu().pin_memory(), tree.cpu().pin_memory()

        def prepare(x):
            o = torch.full((1, T, H, D), float("nan"), dtype=torch.bfloat16).pin_memory()
            l = torch.full((1, H, T), float("nan")).pin_memory()
            return (o, l), lambda: B.sparrow_verify_step_host(ctx, q_host, k_new, v_new, x["k"], x["v"], [kv], par_host, T, o, l)
        return ctx, {"k": k, "v": v}, prepare
    if entry in ("anchor", "anchor_long"):                                # merged in a cluster; by the second kernel
        idx = anchors if entry == "anchor" else _ints([list(range(40, 40 + 2500)) + list(range(3000, 3000 + T))])

        def prepare(x):
            o, l = new_out()
            return (o, l), lambda: B.sparrow_anchor_attn_tree(ctx, x["q"], x["k"], x["v"], x["anchors"], idx.shape[1], 0, x["parents"], T, T, o, l)
        return ctx, {"q": q, "k": k, "v": v, "anchors": idx, "parents": tree}, prepare
    if entry == "compact":
        def prepare(x):
            kc, vc = (torch.zeros((1, HK, 400, D), dtype=torch.bfloat16, device=DEV) for _ in range(2))
            return (kc, vc), lambda: B.sparrow_compact_anchors(ctx, x["k"], x["v"], x["anchors"], n_anchor, kc, vc, 400, 3)
        return ctx, {"k": k, "v": v, "anchors": anchors}, prepare
    if entry == "window_bounds":
        def prepare(x):
            first = torch.full((1, T), -7, dtype=torch.int32, device=DEV)
            return (first,), lambda: B.sparrow_window_first_visible_device(ctx, x["anchors"], n_anchor, 1800, T, T, first)
        return ctx, {"anchors": anchors}, prepare
    if entry == "append":
        def prepare(x):
            kc, vc = k.clone(), v.clone()
            return (kc, vc), lambda: B.sparrow_kv_append(ctx, x["k_new"], x["v_new"], kc, vc, [kv], T)
        return ctx, {"k_new": _normal(gen, 1, HK, T, D), "v_new": _normal(gen, 1, HK, T, D)}, prepare
    if entry == "keep":
        def prepare(x):
            return (x["k"], x["v"]), lambda: B.sparrow_kv_keep_accepted(ctx, x["k"], x["v"], [kv], x["path"], x["n_accept"], T)
        return ctx, {"k": k, "v": v, "path": _ints([[1, 4, 5, 9] + [-1] * (T - 4)]), "n_accept": _ints([4])}, prepare
    if entry == "hsr":
        def prepare(x):
            z = torch.full((9, 512), float("nan"), dtype=torch.bfloat16, device=DEV)
            return (z,), lambda: B.sparrow_hsr_fuse(ctx, x["e"], x["h"], x["w"], x["bias"], z)
        return ctx, {"e": _normal(gen, 9, 256), "h": _normal(gen, 9, 256), "w": _normal(gen, 512, 512), "bias": _normal(gen, 512)}, prepare
    V = 20000
    tokens = torch.randint(0, V, (1, T), generator=gen, device=DEV, dtype=torch.int32)
    new_path = lambda: (torch.full((1, T), -9, dtype=torch.int32, device=DEV), _ints([-9]), _ints([-9]))
    if entry == "accept_greedy":
        nxt = torch.randint(0, V, (1, T + 1), generator=gen, device=DEV, dtype=torch.int32)
        right = nxt.gather(1, (tree + 1).long())
        tokens = torch.where(torch.arange(T, device=DEV)[None] % 3 == 2, right ^ 1, right).contiguous()

        def prepare(x):
            r = new_path()
            return r, lambda: B.sparrow_accept_greedy(ctx, x["tokens"], x["parents"], x["next"], T, *r)
        return ctx, {"tokens": tokens, "parents": tree, "next": nxt}, prepare
    assert entry == "accept_sample"
    p = torch.softmax(torch.randn((1, T + 1, V), generator=gen, device=DEV) * 3, -1)
    pd = torch.softmax(torch.randn((1, T + 1, V), generator=gen, device=DEV) * 3, -1)
    tokens[0, 0] = int(p[0, 0].argmax())                                  # (a root that is accepted more often than not)
    u = torch.randint(0, 2 ** 31 - 1, (1, 2 * T + 1), generator=gen, device=DEV, dtype=torch.int32)

    def prepare(x):
        r = new_path()
        return r, lambda: B.sparrow_accept_sample(ctx, x["tokens"], x["parents"], x["p"], x["pd"], x["u_node"], x["u_bonus"], V, T, *r)
    return ctx, {"tokens": tokens, "parents": tree, "p": p, "pd": pd, "u_node": u[:, :T].contiguous(), "u_bonus": u[:, T:].contiguous()}, prepare


def _poison(t):
    """Values that any reader may meet but that give another result: zeros, -1, the first rows for a list of anchors."""
    if t.dtype != torch.int32 or t.numel() == 1:
        return torch.zeros_like(t)
    if t.shape[-1] > 100:
        return torch.arange(t.shape[-1], dtype=torch.int32, device=DEV).expand_as(t).contiguous()
    return torch.full_like(t, -1)


def _padded(t):
    """A copy in a buffer of whole 16-byte words, as the copying kernel wants it: (buffer, the tensor in it)."""
    n = t.numel() * t.element_size()
    buf = torch.zeros((n + 15) // 16 * 16, dtype=torch.uint8, device=DEV)
    view = buf[:n].view(t.dtype).view(t.shape)
    view.copy_(t)
    return buf, view


ENTRIES = ["verify", "verify_short", "verify_window", "step_host", "anchor", "anchor_long", "compact", "window_bounds", "append", "keep",
           "hsr", "accept_greedy", "accept_sample"]


@pytest.mark.parametrize("entry", ENTRIES)
def test_late_inputs_of_every_entry_point(entry):
    """Each device input in turn is written by the kernel directly before the call, which lets its dependents start
    at once and writes 0, 50 or 400 us later.  The results have to be the bits of a call on inputs that lie there."""
    ctx, inputs, prepare = _problem(entry)

    def run(x, before=None):
        outs, call = prepare(x)
        torch.cuda.synchronize()
        if before:
            before()
        call()
        torch.cuda.synchronize()
        return [o.clone() for o in outs]

    want = run({n: t.clone() for n, t in inputs.items()})
    assert ctx.last_device_status() == 0
    for name, true in inputs.items():
        src, _ = _padded(true)
        wrong = run({n: _poison(t) if n == name else t.clone() for n, t in inputs.items()})
        ctx.last_device_status()
        if name not in ("u_node", "u_bonus"):                           # (one draw need not change with its uniform)
            assert any(not torch.equal(a, b) for a, b in zip(wrong, want)), f"{name} does not matter"
        for delay in (0, 50, 400):
            x = {n: t.clone() for n, t in inputs.items() if n != name}
            buf, x[name] = _padded(_poison(true))
            got = run(x, lambda: B.sparrow_debug_early_trigger_copy(ctx, src, buf, buf.numel(), delay))
            for a, b in zip(got, want):
                assert torch.equal(a, b), f"{name} written {delay} us late"
    assert ctx.last_device_status() == 0
