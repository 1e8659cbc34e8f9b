"""The forms of a work item of the bf16 prefill kernel: two heads of a query tile; the last heads of an odd group of two
neighbouring query tiles; one head whose KV tiles two sub-tiles share (calls with few items, so all the small ones).
Segments around one and two tiles, walks of one, two and three tiles, tiles whose walks differ in length (also the
second one's being the shorter), rows that see nothing; head_dim 128 and one below it."""
import numpy as np
import pytest
import torch

from helpers import LSE_TOL, TOL, Runner, check_close, dev, fa, host
from test_gpu_head_dims import check as check_rows, gen, owners, reference

pytestmark = pytest.mark.gpu

GROUPS = [(1, 1, 128), (3, 1, 128), (10, 2, 128), (7, 1, 128), (5, 5, 64)]
LENS = [[1, 128, 129], [256, 257, 0, 385], [640, 100, 512]]


def check(got, want, what):
    check_close(got[0], want[0], TOL["bf16"], what)
    check_close(got[1], want[1], LSE_TOL["bf16"], what + " lse")


MANY = [(24, 8, 128), (32, 32, 128), (28, 4, 128), (32, 8, 128), (24, 8, 64)]       # enough items for the other forms


@pytest.mark.parametrize("hq,hkv,d,lens", [(*g, n) for g in GROUPS for n in LENS] + [(*g, [300, 517, 64, 700, 129]) for g in MANY])
@pytest.mark.parametrize("causal", [True, False])
def test_local_sync_and_remote(hq, hkv, d, lens, causal):
    q, k, v = gen(21, lens, hq, hkv, d, "bf16")
    L, own = sum(lens), owners(lens)
    r = Runner(len(lens), hq, hkv, d, "bf16", L, causal=causal)
    below = np.tri(L, dtype=bool) if causal else np.ones((L, L), bool)
    check(r.local(q, k, v, lens), reference(q, k, v, below & (own[:, None] == own)), "local")
    check(r.sync(q, k, v), reference(q, k, v, below), "sync")
    # a sparse ascending aggregate whose first key lies late: the first query tile sees nothing
    kept = np.sort(np.random.default_rng(5).permutation(np.arange(L // 3, L))[:max(1, L // 4)]).astype(np.int32)
    check(r.sync(q, k[kept], v[kept], kv_pos=kept),
          reference(q, k[kept], v[kept], kept[None] <= np.arange(L)[:, None] if causal else np.ones((L, len(kept)), bool)), "sparse")
    cu = np.concatenate([[0], np.cumsum(lens)])
    qd, kd, vd = dev(q, "bf16"), dev(k[kept], "bf16"), dev(v[kept], "bf16")
    o, lse = torch.full_like(qd, float("nan")), torch.full((L, hq), float("nan"), device="cuda")
    fa().fedattn_sync_remote(r.ctx, r.shape, qd, cu, kd, vd, torch.from_numpy(kept).cuda(), len(kept), False, o, lse)
    assert r.poll() == 0
    before, after = kept[None] < cu[:-1][own][:, None], kept[None] >= cu[1:][own][:, None]
    check((host(o), host(lse)), reference(q, k[kept], v[kept], before if causal else before | after), "remote")


@pytest.mark.parametrize("hq,hkv,d,L", [(*g, 700) for g in GROUPS] + [(24, 8, 128, 2000), (24, 8, 128, 2400), (32, 8, 128, 2000)])
def test_positions_that_fall_along_the_rows(hq, hkv, d, L):
    """Query positions in falling order: the second query tile of a pair walks fewer KV tiles than the first."""
    q, k, v = gen(22, [L], hq, hkv, d, "bf16")
    r = Runner(1, hq, hkv, d, "bf16", L)
    qp = np.arange(L, dtype=np.int32)[::-1] - 5                   # the last rows see nothing
    check(r.sync(q, k, v, q_pos=qp.copy()), reference(q, k, v, np.arange(L)[None] <= qp[:, None]), "falling q_pos")
    pos = np.random.default_rng(6).permutation(L).astype(np.int32)
    check(r.sync(q, k, v, kv_pos=pos, q_pos=qp.copy()), reference(q, k, v, pos[None] <= qp[:, None]), "falling q_pos, any kv_pos")


@pytest.mark.parametrize("T", [256 * 128, 300 * 128 + 20])
def test_walks_that_skip_tiles_and_walks_too_long_to_list(T):
    """Explicit positions, every other KV tile beyond what the rows see: 128 tiles are listed, 150 and more are walked up
    to the last visible one."""
    rows = 130
    q, k, v = gen(23, [T], 2, 1, 128, "bf16")
    q = q[:rows]
    rng = np.random.default_rng(7)
    tile, within = np.arange(T) // 128, np.arange(T) % 128
    pos = np.where(tile % 2 == 0, (tile // 2) * 128 + within, T + tile).astype(np.int32)
    qp = np.concatenate([[0], rng.integers(0, T // 2, rows - 2), [T - 1]]).astype(np.int32)
    r = Runner(1, 2, 1, 128, "bf16", rows, T)
    check(r.sync(q, k, v, kv_pos=pos, q_pos=qp), reference(q, k, v, pos[None] <= qp[:, None]), "%d keys" % T)


@pytest.mark.parametrize("hq,hkv,d", [(16, 4, 128), (8, 8, 128), (16, 4, 64), (16, 4, 96)])
def test_repeated_calls_agree_to_the_bit(hq, hkv, d):
    """Calls whose items are shared by two warpgroups: every output has one writer."""
    lens = [700, 500]
    L, T = sum(lens), 400
    cu = np.concatenate([[0], np.cumsum(lens)])
    q, k, v = (dev(x, "bf16") for x in gen(24, lens, hq, hkv, d, "bf16"))
    pos = torch.arange(0, L, 3, dtype=torch.int32, device="cuda")
    r = Runner(2, hq, hkv, d, "bf16", L)
    seen = None
    for _ in range(20):
        o, lse = [torch.full_like(q, float("nan")) for _ in range(3)], [torch.full((L, hq), float("nan"), device="cuda") for _ in range(3)]
        fa().fedattn_local(r.ctx, r.shape, q, k, v, cu, o[0], lse[0])
        fa().fedattn_sync(r.ctx, r.shape, q, None, k, v, None, L, False, o[1], lse[1])
        fa().fedattn_sync_remote(r.ctx, r.shape, q, cu, k[:T], v[:T], pos, T, False, o[2], lse[2])
        assert r.poll() == 0
        seen = seen or (o, lse)
        assert all(torch.equal(a, b) for a, b in zip(o + lse, seen[0] + seen[1]))


@pytest.mark.parametrize("hq,hkv,d", [(16, 4, 96), (3, 3, 120), (16, 4, 64), (8, 8, 72)])
def test_one_warpgroup_redoes_a_row(hq, hkv, d):
    """Items shared by two warpgroups, each of which writes half of the columns: a value that is not finite in one
    channel of an excluded row, below and above column 64, leaves every row that does not see it as it is."""
    lens = [700, 500]
    L, own = sum(lens), owners(lens)
    q, k, v = gen(25, lens, hq, hkv, d, "bf16")
    v[690, :, 3], v[1190, 0, d - 5] = np.inf, np.nan
    visible = np.tri(L, dtype=bool) & (own[:, None] == own)
    spoilt = visible[:, [690, 1190]].any(1)
    r = Runner(2, hq, hkv, d, "bf16", L)
    with np.errstate(invalid="ignore"):
        want = reference(q, k, v, visible)
    seen = None
    for _ in range(10):
        o, lse = r.local(q, k, v, lens)
        check_rows((o[~spoilt], lse[~spoilt]), (want[0][~spoilt], want[1][~spoilt]), "bf16", "excluded")
        assert np.abs(lse - want[1]).max() <= 1e-5 and not np.isfinite(o[690:700, :, 3]).any() and not np.isfinite(o[1190:, 0, d - 5]).any()
        seen = seen or (o, lse)
        assert np.array_equal(o, seen[0], equal_nan=True) and np.array_equal(lse, seen[1])
