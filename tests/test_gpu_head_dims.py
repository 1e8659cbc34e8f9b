"""The prefill calls at every storage type and head_dim that the bf16 head_dim-128 kernel does not serve: bf16 with
fewer channels (tensor cores, weights in three bf16 parts) and fp32 (tiled SIMT), against an fp64 evaluation of the
same inputs.  The weights keep more bits than the output has, so the bf16 bound is the rounding of the output: half
a unit in the last of 8 significant bits is at most 2^-8 |o|, plus 2^-14 for weights and sums; fp32 sums of at most
a few hundred O(1) terms stay within 2^-24 * sqrt(terms) * a small factor, 1e-5 is generous."""
import numpy as np
import pytest
import torch

import fedattn_inputs as fi
from helpers import LSE_TOL, Runner, dev, fa, host

pytestmark = pytest.mark.gpu

KINDS = [("bf16", 4, 2, 8), ("bf16", 3, 1, 40), ("bf16", 8, 2, 64), ("bf16", 5, 5, 72), ("bf16", 6, 2, 96), ("bf16", 2, 1, 120),
         ("f32", 4, 4, 64), ("f32", 6, 2, 40), ("f32", 7, 1, 128), ("f32", 3, 3, 72), ("f32", 2, 2, 8)]


def gen(seed, lens, hq, hkv, d, dtype):
    return fi.Workload("t", seed, tuple(int(x) for x in lens), hq, hkv, d, dtype, 1.0).qkv()


def reference(q, k, v, visible):
    """fp64 attention; visible: [rows, keys] or [heads of K, rows, keys]; k, v: [keys, hkv, d]."""
    rows, hq, d = q.shape
    g = hq // k.shape[1]
    o, lse = np.zeros((rows, hq, d)), np.full((rows, hq), -np.inf)
    for h in range(hq):
        vis = visible if visible.ndim == 2 else visible[h // g]
        s = np.where(vis, q[:, h].astype(np.float64) @ k[:, h // g].astype(np.float64).T / np.sqrt(d), -np.inf)
        some = vis.any(1)
        m = np.where(some, s.max(1, initial=-np.inf), 0.0)
        p = np.exp(s - m[:, None])
        z = p.sum(1)
        # excluded keys take no part, whatever their value rows hold
        vh = v[:, h // g].astype(np.float64)
        pv = p @ vh if np.isfinite(vh).all() else np.array([p[i, vis[i]] @ vh[vis[i]] for i in range(rows)])
        o[some, h] = pv[some] / z[some, None]
        lse[some, h] = m[some] + np.log(z[some])
    return o, lse


def check(got, want, dtype, what):
    (o, lse), (wo, wl) = got, want
    assert np.isfinite(o).all(), what
    tol = 2.0 ** -8 * np.abs(wo) + 2.0 ** -14 if dtype == "bf16" else 1e-5
    assert (np.abs(o - wo) <= tol).all(), (what, np.abs(o - wo).max())
    empty = np.isneginf(wl)
    assert np.array_equal(np.isneginf(lse), empty), what
    assert empty.all() or np.abs(lse[~empty] - wl[~empty]).max() <= 1e-5, what


def owners(lens):
    return np.repeat(np.arange(len(lens)), lens)


@pytest.mark.parametrize("lens", [[1], [127, 1, 0, 128], [129, 300, 64], [33, 257, 5, 512]])
@pytest.mark.parametrize("causal", [True, False])
@pytest.mark.parametrize("dtype,hq,hkv,d", KINDS)
def test_local_and_sync_by_row_index(dtype, hq, hkv, d, causal, lens):
    q, k, v = gen(7, lens, hq, hkv, d, dtype)
    L, own = sum(lens), owners(lens)
    r = Runner(len(lens), hq, hkv, d, dtype, L, causal=causal)
    below = np.tri(L, dtype=bool) if causal else np.ones((L, L), bool)
    check(r.local(q, k, v, lens), reference(q, k, v, below & (own[:, None] == own)), dtype, "local")
    check(r.sync(q, k, v), reference(q, k, v, below), dtype, "sync")
    T = max(1, L - 3)                                             # fewer keys than queries, head-major
    kh, vh = (np.ascontiguousarray(np.transpose(x[:T], (1, 0, 2))) for x in (k, v))
    check(r.sync(q, kh, vh, head_major=True), reference(q, k[:T], v[:T], below[:, :T]), dtype, "sync, head-major")


@pytest.mark.parametrize("dtype,hq,hkv,d", KINDS)
def test_positions_in_any_order(dtype, hq, hkv, d):
    """Key positions that go up and down, per head, with and without explicit query positions; the first tiles of
    the walk may hold no visible key of a row whose later logits are far below zero."""
    lens = [200, 131, 390]
    L = sum(lens)
    q, k, v = gen(8, lens, hq, hkv, d, dtype)
    q = q * 3.0 if dtype == "f32" else q
    rng = np.random.default_rng(3)
    pos = np.stack([rng.permutation(L + 40)[:L] for _ in range(hkv)]).astype(np.int32)
    qp = rng.permutation(L).astype(np.int32)
    kh, vh = (np.ascontiguousarray(np.transpose(x, (1, 0, 2))) for x in (k, v))
    r = Runner(len(lens), hq, hkv, d, dtype, L)
    check(r.sync(q, kh, vh, kv_pos=pos, head_major=True), reference(q, k, v, pos[:, None, :] <= np.arange(L)[None, :, None]),
          dtype, "row index against kv_pos")
    check(r.sync(q, kh, vh, kv_pos=pos, q_pos=qp, head_major=True), reference(q, k, v, pos[:, None, :] <= qp[None, :, None]),
          dtype, "q_pos against kv_pos")
    check(r.sync(q, k, v, q_pos=qp), reference(q, k, v, np.arange(L)[None] <= qp[:, None]), dtype, "q_pos alone")
    asc = np.sort(pos[0])
    check(r.sync(q, k, v, kv_pos=asc), reference(q, k, v, asc[None] <= np.arange(L)[:, None]), dtype, "ascending kv_pos")


@pytest.mark.parametrize("causal", [True, False])
@pytest.mark.parametrize("dtype,hq,hkv,d", KINDS)
def test_remote_only(dtype, hq, hkv, d, causal):
    lens = [140, 0, 90, 260, 33]
    L, own = sum(lens), owners(lens)
    q, k, v = gen(9, lens, hq, hkv, d, dtype)
    cu = np.concatenate([[0], np.cumsum(lens)])
    m = fa()
    r = Runner(len(lens), hq, hkv, d, dtype, L, causal=causal)
    kept = np.sort(np.random.default_rng(4).permutation(L)[:301]).astype(np.int32)
    for pos, what in ((kept, "ascending"), (kept[::-1].copy(), "descending"), (None, "all rows")):
        keys = np.arange(L) if pos is None else pos
        qd, kd, vd = dev(q, dtype), dev(k[keys], dtype), dev(v[keys], dtype)
        o = torch.full_like(qd, float("nan"))
        lse = torch.full((L, hq), float("nan"), device="cuda")
        m.fedattn_sync_remote(r.ctx, r.shape, qd, cu, kd, vd, None if pos is None else torch.from_numpy(pos).cuda(), len(keys),
                              False, o, lse)
        assert r.poll() == 0
        before, after = keys[None] < cu[:-1][own][:, None], keys[None] >= cu[1:][own][:, None]
        check((host(o), host(lse)), reference(q, k[keys], v[keys], before if causal else before | after), dtype, what)


def low_logits(seed, L, hq, hkv, d, dtype):
    """q, k, v whose logits all lie near -300."""
    q, k, v = gen(seed, [L], hq, hkv, d, dtype)
    q = np.full_like(q, 4.0)
    k = k * 0.25 if dtype == "f32" else np.round(k * 4) / 16
    k -= 75.0 / np.sqrt(d)
    if dtype == "bf16":
        k = torch.from_numpy(k).to(torch.bfloat16).float().numpy()
    return q, k, v


def check_low(got, want, dtype, d):
    # head_dim 128 takes a part of its exponentials to 7.5e-5 (LSE_TOL has the bound that follows for its lse)
    assert want[1].max() < -200
    assert np.abs(got[1] - want[1]).max() <= (LSE_TOL["bf16"] if dtype == "bf16" and d == 128 else 1e-4)
    assert np.abs(got[0] - want[0]).max() <= (2e-2 if dtype == "bf16" else 1e-3)


# head_dim 128 in bf16 too: items of one head whose KV tiles two sub-tiles share, and (36 heads) of two heads
@pytest.mark.parametrize("dtype,hq,hkv,d", KINDS + [("bf16", 8, 8, 128), ("bf16", 2, 1, 128), ("bf16", 72, 36, 128)])
def test_rows_that_see_no_logit_near_zero(dtype, hq, hkv, d):
    """A row whose first key tiles are all excluded and whose visible logits are near -300: its weights must not be
    taken against a reference of 0."""
    L = 400
    q, k, v = low_logits(10, L, hq, hkv, d, dtype)
    rows = np.arange(L, dtype=np.int32)
    r = Runner(1, hq, hkv, d, dtype, L)
    pos = rows[::-1].copy()                                       # row 0 sees the last key only
    check_low(r.sync(q, k, v, kv_pos=pos, q_pos=rows), reference(q, k, v, pos[None] <= rows[:, None]), dtype, d)
    # every row sees keys of the first tile and of the last one, but only late rows see those between
    pos = np.concatenate([rows[:128] // 4, 300 + rows[128:256] % 64, 280 + rows[256:384] % 64, rows[384:] - 384]).astype(np.int32)
    check_low(r.sync(q, k, v, kv_pos=pos, q_pos=rows), reference(q, k, v, pos[None] <= rows[:, None]), dtype, d)


@pytest.mark.parametrize("dtype,hq,hkv,d", [("bf16", 8, 8, 128), ("bf16", 32, 8, 128), ("bf16", 6, 2, 96)])
def test_interleaved_members_with_low_logits(dtype, hq, hkv, d):
    """Two members that hold alternate tokens of the sequence: a query tile sees a stretch of each member's KV tiles,
    and its rows differ in the last one of either."""
    L = 2000
    q, k, v = low_logits(12, L, hq, hkv, d, dtype)
    pos = np.concatenate([np.arange(0, L, 2), np.arange(1, L, 2)]).astype(np.int32)
    r = Runner(2, hq, hkv, d, dtype, L)
    check_low(r.sync(q, k, v, kv_pos=pos, q_pos=pos), reference(q, k, v, pos[None] <= pos[:, None]), dtype, d)


@pytest.mark.parametrize("dtype,hq,hkv,d", KINDS)
def test_excluded_rows_may_hold_anything(dtype, hq, hkv, d):
    """Inf and NaN in value rows (and NaN in key rows) that the mask excludes do not reach the output; rows that do
    see them come out non-finite."""
    lens = [150, 130, 100]
    L, own = sum(lens), owners(lens)
    q, k, v = gen(11, lens, hq, hkv, d, dtype)
    v[140], v[149, 0, 1], k[279], v[160:170] = np.inf, np.nan, np.nan, -np.inf
    visible = np.tri(L, dtype=bool) & (own[:, None] == own)
    spoilt = visible[:, [140, 149, 279] + list(range(160, 170))].any(1)
    r = Runner(len(lens), hq, hkv, d, dtype, L)
    for (o, lse), vis in ((r.local(q, k, v, lens), visible), (r.sync(q, k, v), np.tri(L, dtype=bool))):
        spoilt = vis[:, [140, 149, 279] + list(range(160, 170))].any(1)
        with np.errstate(invalid="ignore"):
            wo, wl = reference(q, k, v, vis)
        check((o[~spoilt], lse[~spoilt]), (wo[~spoilt], wl[~spoilt]), dtype, "excluded Inf and NaN")
        assert not np.isfinite(o[spoilt][:, 0]).all(1).any()


@pytest.mark.parametrize("d", [8, 64, 96, 120])
def test_weights_keep_more_bits_than_the_output(d):
    """bf16 below 128 channels: two weights that differ by 2^-12 of themselves, on values 1 and -1, beside a third of any
    size on value 0.  Each weight is off by no more than the exponential's and the reference's rounding, 2^-22 each; 16 bits
    would show as 2^-17."""
    rows = 400
    rng = np.random.default_rng(14)
    bf = lambda x: torch.from_numpy(np.asarray(x)).to(torch.bfloat16).float().numpy()
    q, k, v = np.zeros((rows, 1, d)), np.zeros((rows, 1, d)), np.zeros((rows, 1, d))
    q[:, 0, 0], q[:, 0, 1], q[:, 0, 2] = 1.0, bf(rng.uniform(1, 2, rows)), bf(rng.uniform(0.1, 2, rows) * np.sqrt(d))
    k[0, 0, :2], k[1, 0, :2], k[2, 0, 2] = [1.0, 0.0], [1.0, bf(2.0 ** -12 * np.sqrt(d))], 1.0
    v[0], v[1] = -1.0, 1.0
    r = Runner(1, 1, 1, d, "bf16", rows, causal=False)
    q, k, v = (x.astype(np.float32) for x in (q, k[:3], v[:3]))
    o, _ = r.sync(q, k, v)
    wo, _ = reference(q, k, v, np.ones((rows, 3), bool))
    assert (np.abs(wo) < 2.0 ** -9).all() and (np.abs(o - wo) <= 2.0 ** -8 * np.abs(wo) + 2.0 ** -21).all()


@pytest.mark.parametrize("hq,hkv,d,L", [(16, 4, 64, 1000), (8, 2, 96, 1000), (4, 4, 120, 433), (4, 4, 8, 833)])
def test_lse_has_no_bias(hq, hkv, d, L):
    """The mean error of lse over thousands of rows of N(0, 1) logits: fp32 FMA chains stay below 3e-8; sums that are
    cut off instead of rounded, and not corrected for, show as 1e-7 to 2e-7."""
    q, k, v = gen(15, [L], hq, hkv, d, "bf16")
    _, lse = Runner(1, hq, hkv, d, "bf16", L).sync(q, k, v)
    err = lse - reference(q, k, v, np.tri(L, dtype=bool))[1]
    assert abs(err.mean()) <= 9e-8 and err.std() <= 2.5e-7


@pytest.mark.parametrize("lens", [[400], [300, 517, 129]])
@pytest.mark.parametrize("dtype,hq,hkv,d", [("bf16", 8, 2, 64), ("bf16", 6, 2, 96), ("bf16", 32, 32, 40), ("f32", 4, 4, 64)])
def test_logits_whose_last_place_exceeds_one(dtype, hq, hkv, d, lens):
    """Logits around 10^12, a unit of which is 2^16: a row's largest logit takes it all, and its weight must not depend on
    how the reference was rounded."""
    L, own = sum(lens), owners(lens)
    q, k, v = gen(16, lens, hq, hkv, d, dtype)
    q, k = q * 2.0 ** 20, k * 2.0 ** 20
    r = Runner(len(lens), hq, hkv, d, dtype, L)
    visible = np.tri(L, dtype=bool)
    for (o, lse), vis in ((r.local(q, k, v, lens), visible & (own[:, None] == own)), (r.sync(q, k, v), visible)):
        wo, wl = reference(q, k, v, vis)
        # a logit is a sum of d terms around 2^40 / sqrt(d) that may cancel: d / 2 roundings of up to 2^-24 of sqrt(d) 2^40
        assert np.abs(o - wo).max() <= 1e-6 and np.abs(lse - wl).max() <= d / 2 * 2.0 ** -24 * np.sqrt(d) * 2.0 ** 40


@pytest.mark.parametrize("positions", [False, True])
def test_as_many_keys_as_an_int_counts(positions):
    """2^31 - 1 keys of one head of 8 channels (34 GB, K and V in one buffer): the last tile ends where 32-bit sums would
    wrap.  All keys are zero but the last 1000, whose logits are large enough to decide the output."""
    T, d, tail = 2 ** 31 - 1, 8, 1000
    if torch.cuda.mem_get_info()[0] < 60 << 30:
        pytest.skip("needs 60 GB of free device memory")
    rng = np.random.default_rng(13)
    last = torch.from_numpy(rng.standard_normal((tail, d))).to(torch.bfloat16)
    q = torch.from_numpy(16.0 + rng.standard_normal((2, 1, d))).to(torch.bfloat16)
    kv = torch.zeros((T, 1, d), dtype=torch.bfloat16, device="cuda")
    kv[T - tail:, 0] = last.cuda()
    seen = np.ones((2, tail), bool)
    pos = None
    if positions:
        pos = torch.zeros(T, dtype=torch.int32, device="cuda")
        pos[T - tail:] = torch.arange(tail, dtype=torch.int32, device="cuda")
        seen = np.arange(tail)[None] <= np.array([500, tail])[:, None]
    m = fa()
    r = Runner(1, 1, 1, d, "bf16", 2, 1)
    qp = torch.tensor([500, tail] if positions else [T, T], dtype=torch.int32, device="cuda")
    o, lse = torch.full((2, 1, d), float("nan"), dtype=torch.bfloat16, device="cuda"), torch.full((2, 1), float("nan"), device="cuda")
    m.fedattn_sync(r.ctx, r.shape, q.cuda(), qp, kv, kv, pos, T, False, o, lse)
    assert r.poll() == 0
    s = np.where(seen, host(q)[:, 0] @ host(last).T / np.sqrt(d), -np.inf)
    z = np.exp(s).sum(1) + (T - tail)
    wo = (np.exp(s) @ host(last) / z[:, None])[:, None]
    check((host(o), host(lse)), (wo, np.log(z)[:, None]), "bf16", "2^31 - 1 keys")
