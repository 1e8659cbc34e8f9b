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
