"""Which launches are set up while the preceding grid ends, read off the edges of a capture (nothing is launched): every
kernel but the bf16 attention behind one that releases its dependents early, whoever put that on the stream."""
import ctypes as C

import pytest
import torch

from helpers import fa

pytestmark = pytest.mark.gpu


class EdgeData(C.Structure):
    _fields_ = [("from_port", C.c_ubyte), ("to_port", C.c_ubyte), ("type", C.c_ubyte), ("reserved", C.c_ubyte * 5)]


def captured_edges(body):
    """Programmatic (1) or full (0): the edge in front of every captured kernel but the first, in order."""
    cu, stream = C.CDLL("libcuda.so.1"), torch.cuda.Stream()
    s, graph, n = C.c_void_p(stream.cuda_stream), C.c_void_p(), C.c_size_t(0)
    assert cu.cuStreamBeginCapture_v2(s, 2) == 0
    try:
        body(stream)
    finally:
        assert cu.cuStreamEndCapture(s, C.byref(graph)) == 0
    assert cu.cuGraphGetEdges_v2(graph, None, None, None, C.byref(n)) == 0
    src, dst, data = (C.c_void_p * n.value)(), (C.c_void_p * n.value)(), (EdgeData * n.value)()
    assert cu.cuGraphGetEdges_v2(graph, src, dst, data, C.byref(n)) == 0
    assert cu.cuGraphDestroy(graph) == 0
    follows = {a: (b, e.type) for a, b, e in zip(src, dst, data)}
    assert len(follows) == n.value                              # a chain
    at, types = (set(src) - set(dst)).pop(), []
    while at in follows:
        at, t = follows[at]
        types.append(t)
    return types


@pytest.fixture(scope="module")
def calls():
    m, N, L, K, hq, hkv, d = fa(), 2, 256, 64, 4, 2, 128
    T, bf = N * L, torch.bfloat16
    shape = m.Shape(N, hq, hkv, d, m.BF16)
    ctx, other = m.Context(shape, T, T), m.Context(shape, T, T)
    q, k, v = (torch.zeros(T, h, d, dtype=bf, device="cuda") for h in (hq, hkv, hkv))
    o, o2, lse = torch.zeros_like(q), torch.zeros_like(q), torch.zeros(T, hq, device="cuda")
    kc, vc, ka, va = torch.zeros_like(k), torch.zeros_like(v), *(torch.zeros(hkv, N * K, d, dtype=bf, device="cuda") for _ in range(2))
    rows, pos = torch.arange(K, dtype=torch.int32, device="cuda").repeat(hkv, N), torch.arange(T, dtype=torch.int32, device="cuda")
    lens = torch.full((N,), L, dtype=torch.int32, device="cuda")
    parts = list(k.split(L)), list(v.split(L)), [L] * N
    small = m.Context(m.Shape(1, hkv, hkv, 64, m.F32), 1, 1)     # a workspace that a decode cannot use

    def refused(s):
        with pytest.raises(m.FedAttnError):
            m.fedattn_decode(small, shape, m.DECODE_LOCAL, q[:N], k, v, L * hkv * d, lens, L, o, stream=s)

    def make(c):
        return {
            "local": lambda s: m.fedattn_local(c, shape, q, k, v, [0, L, T], o, lse, stream=s),
            "positions": lambda s: m.fedattn_sync(c, shape, q, pos, k, v, pos, T, False, o, lse, stream=s),
            "concat": lambda s: m.fedattn_aggregate_kv(c, shape, m.AGG_CONCAT, *parts, None, None, kc, vc, stream=s),
            "topk": lambda s: m.fedattn_aggregate_kv(c, shape, m.AGG_TOPK_KNORM, *parts, [K] * N, None, ka, va, stream=s),
            "indexed": lambda s: m.fedattn_aggregate_kv(c, shape, m.AGG_INDEXED, *parts, [K] * N, rows, ka, va, stream=s),
            "merge": lambda s: m.fedattn_merge(c, shape, T, o, lse, o, lse, o2, stream=s),
            "decode": lambda s: m.fedattn_decode(c, shape, m.DECODE_LOCAL, q[:N], k, v, L * hkv * d, lens, L, o, stream=s),
            "noalloc": lambda s: m.fedattn_decode_noalloc(shape, m.DECODE_LOCAL, q[:N], k, v, L * hkv * d, lens, L, o, stream=s),
            "refused": refused,
        }

    table = {**make(ctx), **{"other " + name: f for name, f in make(other).items()}}
    for f in table.values():                                    # what a first call sets up is not for a capture
        f(None)
    torch.cuda.synchronize()
    return table


@pytest.mark.parametrize("names,edges", [
    ("local local", [1]), ("concat local", [1]), ("merge local", [1]),
    ("topk local", [0]), ("indexed local", [0]), ("decode local", [0]),
    ("other topk, local", [0]), ("noalloc local", [0]),         # (released by another context, by none)
    ("topk merge local", [1, 1]), ("topk local local", [0, 1]), ("topk, other concat, local", [1, 1]),
    ("topk positions", [0, 1]),                                 # (the tables' kernel is an ordinary launch, and in front)
    ("merge refused local", [1]),                               # (a call that was rejected is not in front)
    ("topk merge", [1]), ("topk concat", [1]), ("decode merge", [1]), ("topk topk", [1]), ("local topk", [1])])
def test_launch_forms(calls, names, edges):
    seq = names.split(", ") if "," in names else names.split()
    assert captured_edges(lambda s: [calls[x](s) for x in seq]) == edges


def test_another_stream_has_a_front_of_its_own(calls):
    aside = torch.cuda.Stream()

    def body(s):
        calls["merge"](s)
        calls["topk"](aside)                                    # (not part of the capture)
        calls["local"](s)

    assert captured_edges(body) == [1]
    torch.cuda.synchronize()
