"""bf16 head_dim-128 decode on either side of the line between one launch (clusters merge in shared memory) and two
(partials through the scratch): caches of no, one and a few 64-key tiles, splits that stay empty, 1, 2, 4 and 8 splits,
4 to 96 stacked query rows per KV head (one, two and several row tiles), an odd group."""
import numpy as np
import pytest

import fedattn_inputs as fi
from helpers import LSE_TOL, TOL, Runner, check_close

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,hq,hkv,cap,lens,launches", [
    (1, 4, 1, 64, [1], 1), (1, 8, 8, 40, [0], 1), (3, 8, 2, 130, [130, 0, 65], 1), (2, 7, 1, 700, [700, 63], 1),
    (5, 32, 8, 300, [300, 1, 128, 64, 257], 1), (2, 8, 2, 2100, [2100, 129], 1), (2, 8, 2, 3200, [3200, 129], 2),
    (12, 8, 1, 200, [200, 3, 64, 65, 127, 128, 129, 0, 190, 191, 192, 193], 1), (1, 40, 1, 500, [499], 1),
    (4, 8, 4, 2600, [2600, 64, 0, 1999], 2), (9, 12, 4, 1000, [1000, 1, 999, 64, 65, 0, 500, 128, 960], 2)])
def test_decode_around_one_and_two_launches(oracle, n, hq, hkv, cap, lens, launches):
    d = 128
    w = fi.Workload("d1", 61, (cap,) * n, hq, hkv, d, "bf16")
    _, k, v = w.qkv()
    q = w.decode_q(0)
    kc, vc = k.reshape(n, cap, hkv, d), v.reshape(n, cap, hkv, d)
    r = Runner(n, hq, hkv, d, "bf16", n * cap)
    before = r.ctx.launch_count()
    o, lse = r.decode(q, kc, vc, lens, False, max_kv_len=cap)
    assert r.ctx.launch_count() - before == launches
    oo, ol = oracle.decode(q, kc, vc, lens, False)
    check_close(o, oo, TOL["bf16"], "local")
    check_close(lse, ol, LSE_TOL["bf16"], "local lse")
    for T in sorted({n * cap, max(lens), 1, 0}):
        o, lse = r.decode(q, k, v, [T], True, max_kv_len=n * cap)
        oo, ol = oracle.decode(q, k, v, [T], True)
        check_close(o, oo, TOL["bf16"], "sync %d" % T)
        check_close(lse, ol, LSE_TOL["bf16"], "sync lse %d" % T)
