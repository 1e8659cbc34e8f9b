"""A call that the CUDA runtime refuses reports it and leaves nothing behind: the next call is accepted, and right.  The
refusal is the host's: the call's stream is in a capture that has been invalidated, so nothing is enqueued."""
import ctypes as C

import pytest
import torch

from helpers import fa

pytestmark = pytest.mark.gpu


class InvalidCapture:
    """A stream whose capture has been invalidated by a synchronisation, which a capture refuses."""

    def __enter__(self):
        self.cu = C.CDLL("libcuda.so.1")
        self.stream = torch.cuda.Stream()
        s = C.c_void_p(self.stream.cuda_stream)
        assert self.cu.cuStreamBeginCapture_v2(s, 2) == 0        # relaxed: other streams and threads are not concerned
        assert self.cu.cuStreamSynchronize(s) != 0
        return self.stream

    def __exit__(self, *_):
        graph = C.c_void_p()
        assert self.cu.cuStreamEndCapture(C.c_void_p(self.stream.cuda_stream), C.byref(graph)) != 0 and not graph.value


FORMS = [("f32", 64), ("bf16", 64), ("bf16", 128)]
CALLS = ["local", "concat", "topk", "indexed", "sync", "sync_positions", "merge", "decode", "decode_long", "selftest", "poll"]


@pytest.mark.parametrize("call,dtype,d", [(c, *f) for c in CALLS for f in FORMS] + [("noalloc", "bf16", 128)])
def test_refused_call_leaves_nothing_behind(call, dtype, d):
    m, N, L, K, hq, hkv = fa(), 2, 1024, 64, 4, 2
    dt, T = torch.bfloat16 if dtype == "bf16" else torch.float32, N * L
    shape = m.Shape(N, hq, hkv, d, m.BF16 if dtype == "bf16" else m.F32)
    ctx = m.Context(shape, T, T)
    g = torch.Generator(device="cuda").manual_seed(8)
    q, k, v = (torch.randn(s, generator=g, device="cuda").to(dt) for s in ((T, hq, d), (T, hkv, d), (T, hkv, d)))
    o, lse, od = torch.zeros_like(q), torch.zeros(T, hq, device="cuda"), torch.zeros(N, hq, d, dtype=dt, device="cuda")
    ka, va = (torch.zeros(hkv, N * K, d, dtype=dt, device="cuda") for _ in range(2))
    kc, vc = torch.zeros_like(k), torch.zeros_like(v)
    rows = torch.arange(K, dtype=torch.int32, device="cuda").repeat(hkv, N)
    pos, lens = torch.arange(T, dtype=torch.int32, device="cuda"), torch.full((N,), L, dtype=torch.int32, device="cuda")
    parts = list(k.split(L)), list(v.split(L)), [L] * N
    calls = {
        "local": lambda s: m.fedattn_local(ctx, shape, q, k, v, [0, L, T], o, lse, stream=s),
        "concat": lambda s: m.fedattn_aggregate_kv(ctx, shape, m.AGG_CONCAT, *parts, None, None, kc, vc, stream=s),
        "topk": lambda s: m.fedattn_aggregate_kv(ctx, shape, m.AGG_TOPK_KNORM, *parts, [K] * N, None, ka, va, stream=s),
        "indexed": lambda s: m.fedattn_aggregate_kv(ctx, shape, m.AGG_INDEXED, *parts, [K] * N, rows, ka, va, stream=s),
        "sync": lambda s: m.fedattn_sync(ctx, shape, q, None, k, v, None, T, False, o, lse, stream=s),
        "sync_positions": lambda s: m.fedattn_sync(ctx, shape, q, pos, k, v, pos, T, False, o, lse, stream=s),
        "merge": lambda s: m.fedattn_merge(ctx, shape, T, q, lse, q, lse, o, None, stream=s),
        "decode": lambda s: m.fedattn_decode(ctx, shape, m.DECODE_LOCAL, q[:N], k, v, L * hkv * d, lens, 160, od, stream=s),
        "decode_long": lambda s: m.fedattn_decode(ctx, shape, m.DECODE_LOCAL, q[:N], k, v, L * hkv * d, lens, 1 << 20, od, stream=s),
        "noalloc": lambda s: m.fedattn_decode_noalloc(shape, m.DECODE_LOCAL, q[:N], k, v, L * hkv * d, lens, L, od, stream=s),
        "selftest": lambda s: ctx.selftest_wait_timeout(stream=s),
        "poll": lambda s: None,
    }
    outputs = (o, lse, od, ka, va, kc, vc)

    def result():
        for x in outputs:
            x.zero_()
        if call != "selftest":
            calls[call](None)
        calls["merge"](None)
        torch.cuda.synchronize()
        return [x.clone() for x in outputs]

    lens.fill_(160)                                             # (within every max_kv_len above)
    want = result()
    with InvalidCapture() as s:
        if call == "poll":
            assert ctx.poll(s) == 4
        else:
            with pytest.raises(m.FedAttnError) as e:
                calls[call](s)
            assert e.value.code == 4
    for a, b in zip(result(), want):
        assert torch.equal(a, b)
    assert ctx.poll() == 0
