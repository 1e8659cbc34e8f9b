"""Kernels whose CTAs are set up while the preceding grid ends (concatenation, merge, the SIMT attention): random
sequences of them and of calls that start early, over shared buffers and without a synchronisation, give to the bit what
they give with one behind every call; so does a replayed graph."""
import numpy as np
import pytest
import torch

from helpers import fa

pytestmark = pytest.mark.gpu


def run(dtype, d, hq, hkv, seed, mode, n_ops=40):
    m, N, L, K = fa(), 3, 96, 40
    dt = torch.bfloat16 if dtype == "bf16" else torch.float32
    T = N * L
    shape = m.Shape(N, hq, hkv, d, m.BF16 if dtype == "bf16" else m.F32)
    ctx = m.Context(shape, T, T)
    g = torch.Generator(device="cuda").manual_seed(5)

    def new(*s):
        return torch.randn(s, generator=g, device="cuda").to(dt)

    q, k, v, k2, v2 = new(T, hq, d), new(T, hkv, d), new(T, hkv, d), new(T, hkv, d), new(T, hkv, d)
    o = [torch.zeros_like(q) for _ in range(3)]
    lse = [torch.zeros(T, hq, device="cuda") for _ in range(3)]
    pos, cu, od = torch.zeros(T, dtype=torch.int32, device="cuda"), [0, L, 2 * L, T], torch.zeros(N, hq, d, dtype=dt, device="cuda")
    kt, vt = torch.zeros(hkv, N * K, d, dtype=dt, device="cuda"), torch.zeros(hkv, N * K, d, dtype=dt, device="cuda")
    post, cut, sel = (torch.zeros(s, dtype=torch.int32, device="cuda") for s in ((hkv, N * K), (N + 1,), (hkv, N * K)))
    lens, total = torch.full((N,), L, dtype=torch.int32, device="cuda"), torch.tensor([T], dtype=torch.int32, device="cuda")
    snaps = torch.zeros(n_ops, 3, T, hq, d, dtype=dt, device="cuda")

    def split(x):
        return [x[cu[i]:cu[i + 1]] for i in range(N)]

    calls = [
        lambda: m.fedattn_local(ctx, shape, q, k, v, cu, o[0], lse[0]),
        lambda: m.fedattn_aggregate_kv(ctx, shape, m.AGG_CONCAT, split(k), split(v), [L] * N, None, None, k2, v2, pos, None, None),
        lambda: m.fedattn_sync(ctx, shape, q, None, k2, v2, None, T, False, o[1], lse[1]),
        lambda: m.fedattn_merge(ctx, shape, T, o[0], lse[0], o[1], lse[1], o[2], lse[2]),
        lambda: m.fedattn_merge(ctx, shape, T, o[2], lse[2], o[0], lse[0], o[1], lse[1]),
        # what the next calls read, written by a merge, an attention and a concatenation
        lambda: m.fedattn_decode(ctx, shape, m.DECODE_LOCAL, o[2][:N], k2, v2, L * hkv * d, lens, L, od),
        lambda: m.fedattn_decode(ctx, shape, m.DECODE_SYNC, o[0][:N], k2, v2, 0, total, T, o[1][:N]),
        lambda: m.fedattn_aggregate_kv(ctx, shape, m.AGG_TOPK_KNORM, split(k2), split(v2), [L] * N, [K] * N, None, kt, vt, post, cut, sel),
        lambda: m.fedattn_aggregate_kv(ctx, shape, m.AGG_INDEXED, split(k), split(v2), [L] * N, [K] * N, sel, kt, vt, post, cut, None),
        lambda: m.fedattn_sync(ctx, shape, q, None, kt, vt, post, N * K, True, o[0], lse[0]),
    ]
    calls[7]()
    order = np.random.default_rng(seed).integers(0, len(calls), n_ops)
    torch.cuda.synchronize()

    def walk():
        for i, c in enumerate(order):
            calls[c]()
            if mode == "synchronised":
                torch.cuda.synchronize()
            if i % 8 == 7:
                for j in range(3):
                    snaps[i, j].copy_(o[j])

    if mode == "graph":
        stream = torch.cuda.Stream()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            walk()
        graph.replay()
    else:
        walk()
    torch.cuda.synchronize()
    assert ctx.poll() == 0
    return [snaps, od, kt, vt, post, *o, *lse]


@pytest.mark.parametrize("dtype,d,hq,hkv", [("f32", 64, 4, 4), ("f32", 128, 8, 2), ("bf16", 64, 4, 2), ("bf16", 128, 8, 2)])
@pytest.mark.parametrize("seed", range(3))
def test_sequences_without_synchronisation(dtype, d, hq, hkv, seed):
    want = run(dtype, d, hq, hkv, seed, "synchronised")
    for mode in ("free", "graph"):
        for a, b in zip(run(dtype, d, hq, hkv, seed, mode), want):
            assert torch.equal(a, b), mode


def test_empty_selection_lets_nothing_overtake_a_decode():
    """A grid of which no thread waits would end before the decode in front of it, and the merge behind would read the
    decode's output too soon: an empty indexed selection without cu_kv launches nothing."""
    m, N, L, hq, hkv, d = fa(), 8, 4096, 32, 8, 128
    shape = m.Shape(N, hq, hkv, d, m.BF16)
    ctx = m.Context(shape, N * L, N * L)
    g = torch.Generator(device="cuda").manual_seed(6)
    q, k, v = (torch.randn(s, generator=g, device="cuda").to(torch.bfloat16) for s in ((N, hq, d), (N * L, hkv, d), (N * L, hkv, d)))
    parts, lens = list(k.split(L)), torch.full((N,), L, dtype=torch.int32, device="cuda")
    none = torch.zeros(0, dtype=torch.int32, device="cuda")

    def rounds(synchronised):
        res = []
        for i in range(6):
            o, lse, out = torch.zeros_like(q), torch.zeros(N, hq, device="cuda"), torch.zeros_like(q)
            for c in (lambda: m.fedattn_decode(ctx, shape, m.DECODE_LOCAL, q * (i + 1), k, v, L * hkv * d, lens, L, o, lse),
                      lambda: m.fedattn_aggregate_kv(ctx, shape, m.AGG_INDEXED, parts, parts, [L] * N, [0] * N, none),
                      lambda: m.fedattn_merge(ctx, shape, N, o, lse, o, lse, out)):
                c()
                if synchronised:
                    torch.cuda.synchronize()
            res.append(out)
        torch.cuda.synchronize()
        return res

    before = ctx.launch_count()
    m.fedattn_aggregate_kv(ctx, shape, m.AGG_INDEXED, parts, parts, [L] * N, [0] * N, none)
    assert ctx.launch_count() == before
    cu_kv = torch.full((N + 1,), -1, dtype=torch.int32, device="cuda")
    m.fedattn_aggregate_kv(ctx, shape, m.AGG_INDEXED, parts, parts, [L] * N, [0] * N, none, None, None, None, cu_kv)
    assert ctx.launch_count() == before + 1 and not cu_kv.any()
    for a, b in zip(rounds(False), rounds(True)):
        assert torch.equal(a, b)
    assert ctx.poll() == 0


def test_captured_branches_that_join():
    """A graph of two branches: one selects, the other decodes, joins it and gathers by what it selected.  The gather's
    launch gets a programmatic edge from the other branch's selection too."""
    m, N, L, K, hq, hkv, d = fa(), 16, 1024, 256, 8, 4, 128
    shape = m.Shape(N, hq, hkv, d, m.BF16)
    ctx, ctx2 = m.Context(shape, N * L, N * L), m.Context(shape, N * L, N * L)
    g = torch.Generator(device="cuda").manual_seed(7)
    q, k, v, w = (torch.randn(s, generator=g, device="cuda").to(torch.bfloat16)
                  for s in ((N, hq, d), (N * L, hkv, d), (N * L, hkv, d), (N * L, hkv, d)))
    lens, rows = torch.full((N,), 64, dtype=torch.int32, device="cuda"), torch.arange(K, dtype=torch.int32, device="cuda").repeat(hkv, N)
    ks, vs, kg, vg = (torch.zeros(hkv, N * K, d, dtype=torch.bfloat16, device="cuda") for _ in range(4))
    sel, o = rows.clone(), torch.zeros_like(q)

    def branches(one, two):
        m.fedattn_decode(ctx2, shape, m.DECODE_LOCAL, q, k, v, L * hkv * d, lens, 64, o, stream=two)
        m.fedattn_aggregate_kv(ctx, shape, m.AGG_TOPK_KNORM, list(k.split(L)), list(v.split(L)), [L] * N, [K] * N, None, ks, vs, None, None,
                               sel, stream=one)
        two.wait_stream(one)
        m.fedattn_aggregate_kv(ctx2, shape, m.AGG_INDEXED, list(w.split(L)), list(v.split(L)), [L] * N, [K] * N, sel, kg, vg, None, None,
                               None, stream=two)

    one, two, graph = torch.cuda.Stream(), torch.cuda.Stream(), torch.cuda.CUDAGraph()
    branches(one, two)
    torch.cuda.synchronize()
    want = [x.clone() for x in (ks, vs, kg, vg, sel, o)]
    with torch.cuda.graph(graph, stream=one):
        two.wait_stream(one)
        branches(one, two)
        one.wait_stream(two)
    for _ in range(10):
        for x in (ks, vs, kg, vg, o):
            x.zero_()
        sel.copy_(rows)
        graph.replay()
        torch.cuda.synchronize()
        assert ctx.poll() == 0 and ctx2.poll() == 0
        for a, b in zip((ks, vs, kg, vg, sel, o), want):
            assert torch.equal(a, b)


def run_ragged(dtype, d, hq, hkv, seed, mode, n_ops=48):
    """Random calls of two contexts over ragged segments (empty ones and one of a single token among them; the bf16
    attention gets more items than there are SMs): explicit query positions, whose tables share the scratch with the
    decode partials, both masks, remote-only attention, whole tokens, empty selections, no keys at all."""
    m, lens = fa(), [0, 1, 700, 257, 1300, 0]
    N, T = len(lens), sum(lens)
    cu, keep = np.concatenate([[0], np.cumsum(lens)]).tolist(), [min(x, 90) for x in lens]
    K, dt = sum(keep), torch.bfloat16 if dtype == "bf16" else torch.float32
    shape, both = (m.Shape(N, hq, hkv, d, m.BF16 if dtype == "bf16" else m.F32, causal) for causal in (1, 0))
    contexts = [m.Context(shape, T, T) for _ in range(2)]
    g = torch.Generator(device="cuda").manual_seed(9)

    def new(*s):
        return torch.randn(s, generator=g, device="cuda").to(dt)

    def ints(*s):
        return torch.zeros(s, dtype=torch.int32, device="cuda")

    q, k, v, k2, v2 = new(T, hq, d), new(T, hkv, d), new(T, hkv, d), new(T, hkv, d), new(T, hkv, d)
    o, lse = [torch.zeros_like(q) for _ in range(3)], [torch.zeros(T, hq, device="cuda") for _ in range(3)]
    od, od2, cap = torch.zeros(N, hq, d, dtype=dt, device="cuda"), torch.zeros(N, hq, d, dtype=dt, device="cuda"), T // N
    kt, vt, post, sel, cut = *(torch.zeros(hkv, K, d, dtype=dt, device="cuda") for _ in range(2)), ints(hkv, K), ints(hkv, K), ints(N + 1)
    kw, vw, posw, selw = *(torch.zeros(K, hkv, d, dtype=dt, device="cuda") for _ in range(2)), ints(K), ints(K)
    q_pos = torch.randperm(T, generator=g, device="cuda").int()
    kv_pos = torch.arange(T, dtype=torch.int32, device="cuda")
    n_loc, n_all = torch.full((N,), cap, dtype=torch.int32, device="cuda"), torch.tensor([T], dtype=torch.int32, device="cuda")
    none = ints(0)
    state = [*o, *lse, od, od2, kt, vt, post, sel, cut, kw, vw, posw, selw, k2, v2]

    def split(x):
        return [x[cu[i]:cu[i + 1]] for i in range(N)]

    calls = [
        lambda c, s: m.fedattn_local(c, shape, q, k, v, cu, o[0], lse[0], stream=s),
        lambda c, s: m.fedattn_local(c, both, q, k, v2, cu, o[1], lse[1], stream=s),
        lambda c, s: m.fedattn_aggregate_kv(c, shape, m.AGG_CONCAT, split(k), split(v), lens, None, None, k2, v2, None, None, None, stream=s),
        lambda c, s: m.fedattn_sync(c, shape, q, None, k2, v2, None, T, False, o[1], lse[1], stream=s),
        lambda c, s: m.fedattn_sync(c, both, q, None, kw, vw, posw, K, False, o[2], lse[2], stream=s),
        lambda c, s: m.fedattn_sync(c, shape, q, q_pos, k2, v2, kv_pos, T, False, o[0], lse[0], stream=s),
        lambda c, s: m.fedattn_sync(c, shape, q, q_pos, kt, vt, post, K, True, o[1], lse[1], stream=s),
        lambda c, s: m.fedattn_sync(c, shape, q, None, None, None, None, 0, False, o[2], lse[2], stream=s),
        lambda c, s: m.fedattn_sync_remote(c, shape, q, cu, kt, vt, post, K, True, o[1], lse[1], stream=s),
        lambda c, s: m.fedattn_sync_remote(c, both, q, cu, kw, vw, posw, K, False, o[2], lse[2], stream=s),
        lambda c, s: m.fedattn_merge(c, shape, T, o[0], lse[0], o[1], lse[1], o[2], lse[2], stream=s),
        lambda c, s: m.fedattn_merge(c, shape, T, o[2], lse[2], o[1], lse[1], o[1], lse[1], stream=s),
        lambda c, s: m.fedattn_decode(c, shape, m.DECODE_LOCAL, o[2][:N], k2, v2, cap * hkv * d, n_loc, cap, od, stream=s),
        lambda c, s: m.fedattn_decode(c, shape, m.DECODE_SYNC, od, k2, v2, 0, n_all, T, o[0][:N], stream=s),
        lambda c, s: m.fedattn_decode(c, shape, m.DECODE_SYNC, o[1][:N], k2, v2, 0, n_all, 1 << 20, od2, stream=s),   # two launches
        lambda c, s: m.fedattn_aggregate_kv(c, shape, m.AGG_TOPK_KNORM, split(k2), split(v2), lens, keep, None, kt, vt, post, cut, sel, stream=s),
        lambda c, s: m.fedattn_aggregate_kv(c, shape, m.AGG_TOPK_TOKEN, split(k2), split(v), lens, keep, None, kw, vw, posw, cut, selw, stream=s),
        lambda c, s: m.fedattn_aggregate_kv(c, shape, m.AGG_INDEXED, split(k), split(v2), lens, keep, sel, kt, vt, post, cut, None, stream=s),
        lambda c, s: m.fedattn_aggregate_kv(c, shape, m.AGG_INDEXED, split(k2), split(v2), lens, [0] * N, none, stream=s),
        lambda c, s: m.fedattn_aggregate_kv(c, shape, m.AGG_TOPK_KNORM, split(k2), split(v2), lens, [0] * N, None, None, None, None, cut, stream=s),
    ]
    if dtype == "bf16" and d == 128:
        calls.append(lambda c, s: m.fedattn_decode_noalloc(shape, m.DECODE_SYNC, od2, k2, v2, 0, n_all, T, o[2][:N], stream=s))
    for i in (15, 16, 0, 3):                                    # what a first call sets up, and selections to start from
        calls[i](contexts[0], None)
    r = np.random.default_rng(seed)
    order, who = r.integers(0, len(calls), n_ops), r.integers(0, 2, n_ops)
    snaps = [[torch.zeros_like(x) for x in (*o, od, kt)] for _ in range(n_ops // 8)]
    start = [x.clone() for x in state]
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]

    def walk(two):
        turn = r.integers(0, 2, n_ops)
        for i, c in enumerate(order):
            s = streams[turn[i] if two else 0]
            if two:
                s.wait_stream(streams[1 - turn[i]])
            calls[c](contexts[who[i]], s)
            if mode == "synchronised":
                torch.cuda.synchronize()
            if i % 8 == 7:
                with torch.cuda.stream(s):
                    for a, b in zip(snaps[i // 8], (*o, od, kt)):
                        a.copy_(b)
        if two:
            streams[0].wait_stream(streams[1])

    if mode.startswith("graph"):
        for i in (5, 6, 8, 9, 10, 12, 13, 14, 17, len(calls) - 1):
            calls[i](contexts[0], None)
        for a, b in zip(state, start):
            a.copy_(b)
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=streams[0]):
            if mode == "graph of two streams":
                streams[1].wait_stream(streams[0])
            walk(mode == "graph of two streams")
        graph.replay()
    else:
        walk(mode == "two streams")
    torch.cuda.synchronize()
    assert all(c.poll() == 0 for c in contexts)
    return [x for s in snaps for x in s] + state


@pytest.mark.parametrize("dtype,d,hq,hkv", [("f32", 64, 4, 2), ("bf16", 64, 8, 4), ("bf16", 128, 32, 8)])
@pytest.mark.parametrize("seed", range(3))
def test_ragged_sequences_without_synchronisation(dtype, d, hq, hkv, seed):
    want = run_ragged(dtype, d, hq, hkv, seed, "synchronised")
    for mode in ("free", "graph", "two streams", "graph of two streams"):
        for i, (a, b) in enumerate(zip(run_ragged(dtype, d, hq, hkv, seed, mode), want)):
            assert torch.equal(a, b), (mode, i)
