"""Values and gate logits past the range of their type stay where they belong: an infinite value reaches the columns of the rows
that attend to it and no others, a key that is not finite makes NaN of the rows that attend to it, and a gate logit of -inf is a
probability of zero."""
import math

import numpy as np
import pytest

from oracle import seer_oracle as O
from paper_2410_13276_b200 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("chunk", [False, True])
@pytest.mark.parametrize("lengths", [(1, 2, 3), (3, 4, 5), (5, 6, 7, 9)])
def test_infinite_values(lengths, chunk):
    from paper_2410_13276_b200 import binding as B
    from paper_2410_13276_b200.prefill import Prefill
    nb, hq, first = 20, 4, 10
    w = W.make_small(seed=220, seqlens=[nb * 64 - 7], hq=hq, hkv=2)
    v = w.v.copy()
    inf = np.uint16(0x7f80)
    v[3 * 64 + 5, 0, 7] = inf                            # blocks 3 and 8 of either KV head
    v[3 * 64 + 63, 1, 100] = inf | np.uint16(0x8000)
    v[8 * 64, 0, 64] = inf
    r = np.random.default_rng(sum(lengths))
    rows = []
    for h in range(hq):
        for i in range(nb):
            n = min(lengths[(h + i) % len(lengths)], i) if i >= first else 0
            row = sorted(r.choice(i, n, replace=False).tolist()) if n else []      # (no diagonal: every row sees every listed key)
            if n and i % 2:                                  # an infinite value in the last block of the list
                row = sorted(r.choice(8, n - 1, replace=False).tolist() + [8]) if n <= 9 else row
            rows.append(row)
    rp, col = np.concatenate([[0], np.cumsum([len(x) for x in rows])]).astype(np.int32), np.array([j for x in rows for j in x], np.int32)
    p = Prefill(w.cu_seqlens, hq, 2, cu_seqlens_q=np.array([0, (nb - first) * 64 - 7], np.int32) if chunk else None)
    p.set_inputs(w.q[first * 64:] if chunk else w.q, w.k, v, w.wq, w.wk)
    p.set_lists(rp, col)
    p.attn()
    assert p.status() == 0
    want, _ = O.sparse_attention(w.q, w.k, v, w.cu_seqlens, rp, col, hq, 2, 64, 1 / math.sqrt(128))
    got = p.o_host().astype(np.float64)
    got, want = got if chunk else got[first * 64:], want[first * 64:]
    assert np.isinf(want).any() and not np.isnan(want).any() and np.isfinite(want).mean() > 0.9
    off = ~np.isfinite(want)
    assert np.array_equal(got[off], want[off]) and np.isfinite(got[~off]).all()
    assert np.all(np.abs(got[~off] - want[~off]) <= 2e-2 + 1e-2 * np.abs(want[~off]))   # the attention's tolerance


# keys of a block by their place: exponentials run on either of two pipes
@pytest.mark.parametrize("what", [float("nan"), float("inf")])
def test_keys_that_are_not_finite(what):
    from paper_2410_13276_b200 import binding as B
    from paper_2410_13276_b200.prefill import Prefill
    nb, hq = 70, 2
    w = W.make_small(seed=221, seqlens=[nb * 64], hq=hq, hkv=1)
    q, k = w.q.copy(), w.k.copy()
    q[:, :, 3] = np.where(np.arange(nb * 64) % 5 == 0, 0xbf80, 0x3f80)[:, None]   # -1 or 1: an infinite key scores +inf or -inf
    for j in range(64):
        k[j * 64 + j, 0, 3] = 0x7fc0 if np.isnan(what) else 0x7f80              # block j: its key j
    rows = [[] for _ in range(hq * nb)]
    r = np.random.default_rng(4)
    for h in range(hq):
        for i in range(64, nb):
            n = (i - 64 + h) % 5 + 1
            rows[h * nb + i] = sorted(r.choice(64, n, replace=False).tolist()) if i % 2 else [64] * (i > 64) + [65] * (i > 65)
    rows[64], rows[66] = list(range(64)), [0, 17, 64]
    rp, col = np.concatenate([[0], np.cumsum([len(x) for x in rows])]).astype(np.int32), np.array([j for x in rows for j in x], np.int32)
    p = Prefill(w.cu_seqlens, hq, 1)
    p.set_inputs(q, k, w.v, w.wq, w.wk)
    p.set_lists(rp, col)
    p.attn()
    assert p.status() == 0
    got = p.o_host().astype(np.float64)
    clean = np.where((k & 0x7f80) == 0x7f80, 0, k).astype(np.uint16)             # (the key of -inf scores is replaced below)
    for h in range(hq):
        for i in range(64, nb):
            row = rows[h * nb + i]
            bad = any(j < 64 for j in row)
            for t in range(i * 64, i * 64 + 64, 7):
                if bad and (np.isnan(what) or t % 5):
                    assert np.isnan(got[t, h]).all(), (h, i, t)
                elif row:
                    keys = [x for j in row for x in range(j * 64, j * 64 + 64) if not (j < 64 and x == j * 65)]   # 2^(-inf) = 0
                    s = O.bf16_bits_to_f64(clean[keys, 0]) @ O.bf16_bits_to_f64(q[t, h]) / math.sqrt(128)
                    e = np.exp(s - s.max())
                    want = e @ O.bf16_bits_to_f64(w.v[keys, 0]) / e.sum()
                    assert np.all(np.abs(got[t, h] - want) <= 2e-2 + 1e-2 * np.abs(want)), (h, i, t)   # the attention's tolerance


# blocks whose logits lie below the range of fp32, alone among a row's columns of a 32-column group, at the edges of groups, tiles
# and 256-column segments; by one launch and by two
@pytest.mark.parametrize("nb,two", [(300, False), (640, True)])
def test_logits_below_the_range(nb, two):
    from paper_2410_13276_b200 import binding as B
    from paper_2410_13276_b200.prefill import Prefill
    low = [31, 32, 64, 95, 96, 128, 255, 256, 257, 288, nb - 1]
    q, k = np.zeros((nb * 64, 1, 128), np.float32), np.zeros((nb * 64, 1, 128), np.float32)
    q[:, 0, 0] = 2.0 ** 64                                   # (powers of two: pooling, projection and products are exact)
    q[:, 0, 1] = 1.0
    k[:, 0, 1] = np.repeat(np.arange(nb) % 7, 64)
    for j in low:
        k[j * 64:(j + 1) * 64, 0, 0] = -2.0 ** 100           # a logit of -2^164 / sqrt(128)
    eye = np.eye(128, dtype=np.float32)[None]
    bits = [W.f32_to_bf16_bits(x) for x in (q, k)]
    p = Prefill(np.array([0, nb * 64], np.int32), 1, 1, want_lse=False)
    p.set_inputs(bits[0], bits[1], bits[1], eye, eye)
    p.scores.zero_()
    n0 = B.seer_launch_count(p.ctx)
    p.gate()
    assert p.status() == 0 and B.seer_launch_count(p.ctx) - n0 == (3 if two else 2)
    got = O.unflatten_scores(p.scores_host(), p.cu, 64, 1)[0][0].astype(np.float64)
    want = O.gate_scores(bits[0], bits[1], eye, eye, p.cu, 64)[0][0]
    tri = np.tril(np.ones((nb, nb), bool))
    assert all((want[j:, j] == 0).all() for j in low)
    assert np.all(np.abs(got - want)[tri] <= 1e-3 * want[tri])      # the gate's tolerance
    # lists from those scores by one call
    params = B.make_mask_params(B.SEER_TOPK_RATIO, keep_num=1, keep_den=3, flags=3)
    p.mask(params)
    lists = [x.copy() for x in p.lists_host()]
    p.row_ptr.fill_(-1)
    p.gate_mask(params, band_bytes=1 << 20)
    assert p.status() == 0 and all(np.array_equal(a, b) for a, b in zip(lists, p.lists_host()))
