"""The work that users of this package have it do, as timed cases.

Every case is one pass through the public entry points on buffers that a program would hold anyway: a Transformer
block's attention (local, synchronised, with a sparsified exchange, with general positions), the exchange step by
itself, and decode steps.  Sizes are those of the repository's workloads and tests, or generic; inputs are i.i.d.
N(0, 1) rounded to the storage type, which gives N(0, 1) logits under the default scale.
"""
import math

import torch

import paper_2511_02647_b200 as fa

CFG3_LENS = "1467,650,1400,1484,2698,4093,845,996"      # eight lengths uniform on [256, 4096], 13 633 tokens


def listed():
    return [
        # one fp32 layer of two short participants: every call is a few microseconds, latency and launches count
        dict(name="round_f32_2x128", kind="round", lens="128,128", hq=4, hkv=4, d=64, dtype="f32", causal=True),
        # a local and a synchronised block of a model with 64 channels per head, ragged prompts
        dict(name="round_bf16_d64_ragged", kind="round", lens="300,517,64,700,129,450", hq=16, hkv=4, d=64, dtype="bf16",
             causal=True),
        # the block that runs most often: every participant attends its own 2048 tokens
        dict(name="local_4x2048", kind="local", lens="2048,2048,2048,2048", hq=32, hkv=8, d=128, dtype="bf16", causal=True),
        # the block that costs most: dense aggregation, then 8192 queries over 8192 keys
        dict(name="sync_4x2048", kind="sync", lens="2048,2048,2048,2048", hq=32, hkv=8, d=128, dtype="bf16", causal=True),
        # one communication round (a local block, a synchronised block) of prompts of very different length: the largest
        dict(name="round_8xragged", kind="round", lens=CFG3_LENS, hq=32, hkv=8, d=128, dtype="bf16", causal=True),
        # synchronised block over a sparsified exchange: the top quarter of every participant's keys per KV head
        dict(name="sparse_16x1024_top256", kind="sparse", lens=",".join(["1024"] * 16), keep=0.25, select="topk", hq=32, hkv=8,
             d=128, dtype="bf16", causal=True),
        # the own segment stays complete, the others' keys are a random quarter: two attentions and their merge
        dict(name="exchange_16x1024_random", kind="exchange", lens=",".join(["1024"] * 16), keep=0.25, select="random", hq=32,
             hkv=8, d=128, dtype="bf16", causal=True),
        # the same block of an encoder (no causal mask) over whole selected tokens, short ragged segments, odd group size
        dict(name="exchange_bidir_token_ragged", kind="exchange", lens="300,517,64,700,129,450", keep=0.3, select="token",
             hq=24, hkv=8, d=128, dtype="bf16", causal=False),
        # only half of the participants exchange: explicit positions for them, local attention for the rest
        dict(name="subset_8xragged", kind="subset", lens=CFG3_LENS, order="contiguous", hq=32, hkv=8, d=128, dtype="bf16",
             causal=True),
        # the exchange step by itself (what the aggregating side runs): selection and gather, no attention
        dict(name="aggregate_16x1024_top256", kind="aggregate", lens=",".join(["1024"] * 16), keep=0.25, select="topk", hq=32,
             hkv=8, d=128, dtype="bf16", causal=True),
        # four blocks of a decode step, the fourth synchronised (H = 4): full caches, bound by memory
        dict(name="decode_round_8x4096", kind="decode", n=8, cap=4096, low=1.0, hq=32, hkv=8, d=128, dtype="bf16"),
        # one synchronised decode block after some generation: shared cache, private suffixes, merge; small and ragged
        dict(name="decode_suffix_4x700", kind="suffix", n=4, total=2800, cap=160, low=0.1, hq=32, hkv=8, d=128, dtype="bf16"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _lens(rng, lo_total, hi_total, most_parts, longest):
    """Segment lengths: equal or ragged, odd ones among them."""
    total = _log_int(rng, lo_total, hi_total)
    n = rng.randint(2, most_parts)
    n = max(2, n, -(-total // longest) * 2)
    if rng.random() < 0.4:
        return ",".join([str(max(1, min(longest, total // n)))] * n)
    w = [rng.uniform(0.2, 1.8) for _ in range(n)]
    return ",".join(str(max(1, min(longest, int(total * x / sum(w))))) for x in w)


def draw(rng):
    kind = rng.choice(["round", "round", "local", "sync", "sparse", "exchange", "subset", "aggregate", "decode", "decode", "suffix"])
    hkv, g = rng.choice([(8, 4), (8, 4), (8, 3), (8, 2), (4, 4), (2, 7), (8, 1)])
    c = dict(kind=kind, hq=hkv * g, hkv=hkv, d=128, dtype="bf16")
    if kind in ("decode", "suffix"):
        c["n"] = rng.randint(1, 16)
        c["low"] = rng.choice([1.0, 0.7, 0.1])                       # shortest cache over the longest
        most = 8 * 4096
        if rng.random() < 0.3:                                       # other types and head sizes, at moderate lengths
            c["dtype"], c["d"] = rng.choice([("f32", 64), ("bf16", 64), ("f32", 128)])
            most = 4096
        if kind == "decode":
            c["cap"] = _log_int(rng, 64, max(64, min(8192, most // c["n"])))
        else:
            c["total"] = _log_int(rng, 256, most)
            c["cap"] = _log_int(rng, 8, 512)
        return c
    c["causal"] = kind == "subset" or rng.random() < 0.75
    lo, hi = 256, 13600
    if kind in ("round", "exchange") and rng.random() < 0.4:         # other types and head sizes
        c["dtype"], c["d"] = rng.choice([("f32", 64), ("f32", 128), ("bf16", 64), ("bf16", 96)])
        c["hq"], c["hkv"] = rng.choice([(4, 4), (8, 2), (16, 4)])
        lo, hi = 64, 2048
    elif kind in ("sparse", "exchange", "aggregate"):
        hi = 16384
    if not c["causal"]:
        hi = min(hi, 8192)                                           # every pair counts: twice the work per token
    c["lens"] = _lens(rng, lo, hi, 16 if kind in ("sparse", "exchange", "aggregate") else 8, 4096)
    if kind in ("sparse", "exchange", "aggregate"):
        c["keep"] = rng.choice([0.1, 0.25, 0.5])
        c["select"] = rng.choice(["topk", "token", "random"])
    if kind == "subset":
        c["order"] = rng.choice(["contiguous", "interleaved"])
    return c


# ---- what a program has in hand ------------------------------------------------------------------------

def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _dtype(case):
    return torch.bfloat16 if case["dtype"] == "bf16" else torch.float32


def _lens_of(case):
    return [int(x) for x in case["lens"].split(",")]


def _kept(case):
    return [max(1, int(case["keep"] * n)) for n in _lens_of(case)]


def _offsets(lens):
    cu = [0]
    for n in lens:
        cu.append(cu[-1] + n)
    return cu


def prepare(case, seed):
    gen, dt = _gen(seed), _dtype(case)
    hq, hkv, d, kind = case["hq"], case["hkv"], case["d"], case["kind"]
    code = fa.BF16 if dt == torch.bfloat16 else fa.F32

    def normal(*shape):
        return torch.randn(shape, generator=gen, device="cuda", dtype=torch.float32).to(dt)

    def empty(*shape, dtype=dt):
        return torch.empty(shape, dtype=dtype, device="cuda")

    if kind in ("decode", "suffix"):
        return _prepare_decode(case, gen, code, normal, empty)
    lens = _lens_of(case)
    n, cu = len(lens), _offsets(lens)
    L = cu[-1]
    s = dict(case=case, lens=lens, cu=cu, L=L)
    s["shape"] = fa.Shape(n, hq, hkv, d, code, causal=1 if case["causal"] else 0)
    s["k"], s["v"] = normal(L, hkv, d), normal(L, hkv, d)
    s["k_parts"] = [s["k"][cu[i]:cu[i + 1]] for i in range(n)]
    s["v_parts"] = [s["v"][cu[i]:cu[i + 1]] for i in range(n)]
    if kind != "aggregate":
        s["q"], s["o"] = normal(L, hq, d), empty(L, hq, d)
        s["o_local"] = empty(L, hq, d)
    kept, T = None, L
    if "select" in case:
        kept = _kept(case)
        T = sum(kept)
        s["kept"], s["T"] = kept, T
        token = case["select"] == "token"
        s["mode"] = {"topk": fa.AGG_TOPK_KNORM, "token": fa.AGG_TOPK_TOKEN, "random": fa.AGG_INDEXED}[case["select"]]
        rows = (T, hkv, d) if token else (hkv, T, d)
        s["k_agg"], s["v_agg"] = empty(*rows), empty(*rows)
        s["kv_pos"] = empty(*(rows[:1] if token else rows[:2]), dtype=torch.int32)
        s["cu_kv"] = empty(n + 1, dtype=torch.int32)
        s["sel"], s["drawn"] = torch.empty_like(s["kv_pos"]), None
        if case["select"] == "random":                               # a seeded draw per participant and KV head, ascending
            s["drawn"] = torch.cat([torch.rand((hkv, m), generator=gen, device="cuda").argsort(1)[:, :k].sort(1).values
                                    for m, k in zip(lens, kept)], 1).to(torch.int32).contiguous()
    elif kind in ("sync", "round"):
        s["k_agg"], s["v_agg"], s["kv_pos"] = empty(L, hkv, d), empty(L, hkv, d), empty(L, dtype=torch.int32)
    if kind == "exchange":
        s["o_remote"] = empty(L, hq, d)
        s["lse_local"], s["lse_remote"] = empty(L, hq, dtype=torch.float32), empty(L, hq, dtype=torch.float32)
    if kind == "subset":
        half = n // 2
        Lm = cu[half]
        s.update(half=half, Lm=Lm, cu_rest=[c - Lm for c in cu[half:]])
        s["shape_members"] = fa.Shape(half, hq, hkv, d, code)
        s["shape_rest"] = fa.Shape(n - half, hq, hkv, d, code)
        s["k_agg"], s["v_agg"] = empty(Lm, hkv, d), empty(Lm, hkv, d)
        # the members' rows hold contiguous stretches of the global sequence, or alternate tokens of it
        pos = torch.arange(Lm, device="cuda")
        if case["order"] == "interleaved":
            owner = torch.repeat_interleave(torch.arange(half, device="cuda"), torch.tensor(lens[:half], device="cuda"))
            within = pos - torch.tensor(cu[:half], device="cuda")[owner]
            pos = torch.empty_like(pos).scatter_(0, torch.argsort(within * half + owner), pos)
        s["pos"] = pos.to(torch.int32)
    s["ctx"] = fa.Context(s["shape"], L, max(T, L))
    return s


def _prepare_decode(case, gen, code, normal, empty):
    n, hq, hkv, d, cap = case["n"], case["hq"], case["hkv"], case["d"], case["cap"]
    T = n * cap if case["kind"] == "decode" else case["total"]
    s = dict(case=case, shape=fa.Shape(n, hq, hkv, d, code))
    s["ctx"] = fa.Context(s["shape"], n * cap, T)
    ctx, shape, stride = s["ctx"], s["shape"], cap * hkv * d
    lens = (cap * (case["low"] + (1 - case["low"]) * torch.rand(n, generator=gen, device="cuda"))).round().clamp(1, cap)
    s["lens"] = lens.to(torch.int32)
    s["total"] = torch.tensor([T], dtype=torch.int32, device="cuda")
    f32 = torch.float32
    s["calls"], s["out"] = [], []

    def local(lse=None):
        q, k, v, o = normal(n, hq, d), normal(n, cap, hkv, d), normal(n, cap, hkv, d), empty(n, hq, d)
        s["calls"].append(fa.prepare_decode(ctx, shape, fa.DECODE_LOCAL, q, k, v, stride, s["lens"], cap, o, lse))
        return q, o

    def sync(q, lse=None):
        k, v, o = normal(T, hkv, d), normal(T, hkv, d), empty(n, hq, d)
        s["calls"].append(fa.prepare_decode(ctx, shape, fa.DECODE_SYNC, q, k, v, 0, s["total"], T, o, lse))
        return o

    if case["kind"] == "decode":                                     # blocks 1..4 of a model with H = 4
        s["out"] = [local()[1] for _ in range(3)] + [sync(normal(n, hq, d))]
    else:                                                            # one query over the suffix and the shared cache
        lse_a, lse_b = empty(n, hq, dtype=f32), empty(n, hq, dtype=f32)
        q, o_a = local(lse_a)
        o_b = sync(q, lse_b)
        o, lse = empty(n, hq, d), empty(n, hq, dtype=f32)
        s["calls"].append(fa.prepare_merge(ctx, shape, n, o_b, lse_b, o_a, lse_a, o, lse))
        s["out"] = [o, lse]
    return s


# ---- one pass ---------------------------------------------------------------------------------------------

def run(s):
    kind = s["case"]["kind"]
    if kind in ("decode", "suffix"):
        for call in s["calls"]:
            call()
        return s["out"]
    ctx, shape = s["ctx"], s["shape"]
    out = {}
    if kind in ("local", "round"):
        fa.fedattn_local(ctx, shape, s["q"], s["k"], s["v"], s["cu"], s["o_local"])
        out["o_local"] = s["o_local"]
    if kind in ("sync", "round"):
        fa.fedattn_aggregate_kv(ctx, shape, fa.AGG_CONCAT, s["k_parts"], s["v_parts"], s["lens"], None, None, s["k_agg"],
                                s["v_agg"], s["kv_pos"], None, None)
        fa.fedattn_sync(ctx, shape, s["q"], None, s["k_agg"], s["v_agg"], s["kv_pos"], s["L"], False, s["o"])
        out.update(k_agg=s["k_agg"], v_agg=s["v_agg"], kv_pos=s["kv_pos"], o=s["o"])
    if kind in ("sparse", "exchange", "aggregate"):
        fa.fedattn_aggregate_kv(ctx, shape, s["mode"], s["k_parts"], s["v_parts"], s["lens"], s["kept"], s["drawn"], s["k_agg"],
                                s["v_agg"], s["kv_pos"], s["cu_kv"], s["sel"])
        out.update(k_agg=s["k_agg"], v_agg=s["v_agg"], kv_pos=s["kv_pos"], cu_kv=s["cu_kv"], sel=s["sel"])
    head_major = s["case"].get("select") != "token"
    if kind == "sparse":
        fa.fedattn_sync(ctx, shape, s["q"], None, s["k_agg"], s["v_agg"], s["kv_pos"], s["T"], head_major, s["o"])
        out["o"] = s["o"]
    if kind == "exchange":
        fa.fedattn_local(ctx, shape, s["q"], s["k"], s["v"], s["cu"], s["o_local"], s["lse_local"])
        fa.fedattn_sync_remote(ctx, shape, s["q"], s["cu"], s["k_agg"], s["v_agg"], s["kv_pos"], s["T"], head_major,
                               s["o_remote"], s["lse_remote"])
        fa.fedattn_merge(ctx, shape, s["L"], s["o_local"], s["lse_local"], s["o_remote"], s["lse_remote"], s["o"])
        out.update(o_local=s["o_local"], lse_local=s["lse_local"], o_remote=s["o_remote"], lse_remote=s["lse_remote"], o=s["o"])
    if kind == "subset":
        half, Lm = s["half"], s["Lm"]
        fa.fedattn_aggregate_kv(ctx, s["shape_members"], fa.AGG_CONCAT, s["k_parts"][:half], s["v_parts"][:half],
                                s["lens"][:half], None, None, s["k_agg"], s["v_agg"], None, None, None)
        fa.fedattn_sync(ctx, s["shape_members"], s["q"][:Lm], s["pos"], s["k_agg"], s["v_agg"], s["pos"], Lm, False,
                        s["o"][:Lm])
        fa.fedattn_local(ctx, s["shape_rest"], s["q"][Lm:], s["k"][Lm:], s["v"][Lm:], s["cu_rest"], s["o"][Lm:])
        out.update(k_agg=s["k_agg"], v_agg=s["v_agg"], o=s["o"])
    return out


# ---- what a pass cannot do without ---------------------------------------------------------------------

def _pairs_local(lens, causal):
    return sum(n * (n + 1) // 2 if causal else n * n for n in lens)


def _pairs_sparse(lens, kept, causal, remote):
    """(query, kept key) pairs; a participant's kept keys lie evenly along its segment."""
    total, before, T = 0.0, 0, sum(kept)
    for n, k in zip(lens, kept):
        if remote:
            total += n * (before if causal else T - k)
        else:
            total += n * before + k * (n + 1) / 2 if causal else n * T
        before += k
    return total


def work(case):
    hq, hkv, d, kind = case["hq"], case["hkv"], case["d"], case["kind"]
    e = 2 if case["dtype"] == "bf16" else 4
    if kind in ("decode", "suffix"):
        n, cap = case["n"], case["cap"]
        T = n * cap if kind == "decode" else case["total"]
        mean = cap * (1 + case["low"]) / 2
        blocks = 3 if kind == "decode" else 1
        kv_local, kv_sync = blocks * n * mean * hkv * d * 2 * e, T * hkv * d * 2 * e
        q_o = n * hq * d * e * (2 * (blocks + 1) if kind == "decode" else 2)
        return {"bytes": kv_local + kv_sync + q_o, "flops": 4.0 * d * hq * n * (blocks * mean + T)}
    lens = _lens_of(case)
    L, causal = sum(lens), case["causal"]
    qo, kv = L * hq * d * e, L * hkv * d * 2 * e                       # Q or O once; K and V once
    nbytes, pairs = 0.0, 0.0
    if kind in ("local", "round"):
        nbytes += 2 * qo + kv
        pairs += _pairs_local(lens, causal)
    if kind in ("sync", "round"):
        nbytes += 2 * qo + 2 * kv + 4 * L                             # K and V read, and written once as the aggregate
        pairs += L * (L + 1) // 2 if causal else L * L
        if kind == "round":
            nbytes -= qo + kv                                         # the same inputs serve both blocks
    if kind in ("sparse", "exchange", "aggregate"):
        kept = _kept(case)
        T = sum(kept)
        row = hkv * d * e
        # all keys are read for the scores, or for the own segments; values only where they are used
        whole = kind == "exchange"
        nbytes += L * row if case["select"] != "random" or whole else T * row
        nbytes += L * row if whole else T * row
        nbytes += 2 * T * row + 8 * T * (1 if case["select"] == "token" else hkv)
        if kind == "sparse":
            nbytes += 2 * qo
            pairs += _pairs_sparse(lens, kept, causal, False)
        if kind == "exchange":
            nbytes += 4 * qo + 8 * L * hq
            pairs += _pairs_local(lens, causal) + _pairs_sparse(lens, kept, causal, True)
    if kind == "subset":
        half = len(lens) // 2
        Lm = sum(lens[:half])
        nbytes += 2 * qo + kv + Lm * hkv * d * 2 * e
        pairs += Lm * (Lm + 1) // 2 + _pairs_local(lens[half:], True)
    return {"bytes": nbytes, "flops": 4.0 * d * hq * pairs}


def tolerance(case):
    if case["kind"] == "aggregate":
        return "exact"                                                # rows, positions and indices: copies and an exact order
    # Four times what the path shows against the same sums in 64 bits: fp32 2.4e-7 at 256 keys (a few times that
    # where more keys are summed), bf16 2.3e-3 (2.8e-3 merged; the rounding of P and of the output), largest
    # difference 2.4e-6 and 4.5e-2 of the root mean square.
    if case["dtype"] == "f32":
        return {"rel": 3e-6, "max": 3e-5}
    return {"rel": 1e-2, "max": 0.2}
