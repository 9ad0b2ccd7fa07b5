"""Edges of the gate's and the mask's dispatch: scores by one launch or by two (statistics of column segments first, 256 columns
up to 2048-block sequences and 1024 beyond), pooling by 2 or by 16 blocks per CTA, TopK rows by one, four or eight warps or
by the general kernel, and the packed score bands of a chunk."""
import numpy as np
import pytest

from oracle import seer_oracle as O
from paper_2410_13276_b200 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rt():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("no CUDA device: the gpu tests must run on a B200")
    from paper_2410_13276_b200 import binding as B
    from paper_2410_13276_b200.prefill import Prefill
    ctx = B.Context(0)
    yield B, Prefill, ctx
    ctx.close()


def check_rows(got, ref, rows):
    """Scores of causal blocks within 1e-3 relative (logits from three bf16 planes a factor, fp32 sums: about 2^-17 of a logit of
    magnitude 10, then the exponential)."""
    for g, r in zip(got, ref):
        for i in rows:
            if i < r.shape[-1]:
                a, b = g[:, i, :i + 1].astype(np.float64), r[:, i, :i + 1]
                assert np.all(np.abs(a - b) <= np.where(b < 1e-30, 1e-33, 1e-3 * b)), i


# blocks: 577 = the shortest row split for one head; 2048 / 2049: the last of 256-column segments, the first of 1024-column ones
@pytest.mark.parametrize("lens,hq,hkv", [([577 * 64], 1, 1), ([640 * 64 - 63], 3, 1), ([2048 * 64], 1, 1), ([2048 * 64 + 1], 1, 1),
                                         ([100, 700 * 64 + 5, 0, 65, 650 * 64 - 1], 2, 2)])
def test_two_launches_equal_one(rt, lens, hq, hkv):
    import torch
    B, Prefill, ctx = rt
    w = W.make_small(seed=55_000 + len(lens), seqlens=lens, hq=hq, hkv=hkv, q_gain=2.0)
    p = Prefill(w.cu_seqlens, hq, hkv, ctx=ctx, want_lse=False)
    p.set_inputs(w.q, w.k, w.v, w.wq, w.wk)
    n0 = B.seer_launch_count(ctx)
    p.gate()
    n1 = B.seer_launch_count(ctx)
    got = p.scores_host().copy()
    p.ws = torch.empty(B.seer_workspace_bytes(p.shape), dtype=torch.uint8, device="cuda")   # no room for the statistics
    p.scores.fill_(float("nan"))
    p.gate()
    assert p.status() == 0 and (n1 - n0, B.seer_launch_count(ctx) - n1) == (3, 2)
    a, b = (O.unflatten_scores(x, w.cu_seqlens, 64, hq) for x in (got, p.scores_host()))
    edges = [0, 1, 63, 64, 65, 255, 256, 257, 576, 639, 1023, 1024, 1025, 2047, 2048]
    for x, y in zip(a, b):
        tri = np.tril(np.ones(x.shape[-2:], bool))
        assert np.array_equal(x[:, tri], y[:, tri])
    check_rows(a, O.gate_scores(w.q, w.k, w.wq, w.wk, w.cu_seqlens, 64), edges)


# 16 heads (12 + 4): 37 groups of 16 blocks are 592 CTAs (pooled two blocks a CTA), 38 are 608 (sixteen)
@pytest.mark.parametrize("block", [64, 128])
@pytest.mark.parametrize("extra", [[], [1]])
def test_pooling_group_sizes(rt, block, extra):
    B, Prefill, ctx = rt
    lens = [300 * block - 5, 291 * block + 1] + extra
    w = W.make_small(seed=55_100, seqlens=lens, hq=12, hkv=4, block=block)
    p = Prefill(w.cu_seqlens, 12, 4, ctx=ctx, want_lse=False, block=block)
    p.set_inputs(w.q, w.k, w.v, w.wq, w.wk)
    p.gate()
    assert p.status() == 0
    check_rows(O.unflatten_scores(p.scores_host(), w.cu_seqlens, block, 12),
               O.gate_scores(w.q, w.k, w.wq, w.wk, w.cu_seqlens, block), [0, 1, 15, 16, 17, 150, 290, 291, 298, 299])


@pytest.mark.parametrize("nb", [2048, 2049, 8192, 8193, 16384, 16385])
def test_topk_row_lengths(rt, nb):
    import torch
    B, Prefill, ctx = rt
    cu = np.array([0, nb * 64 - 3], np.int32)
    for kw in (dict(mode=O.MODE_TOPK_COUNT, k=257, flags=3), dict(mode=O.MODE_TOPK_RATIO, keep_num=1, keep_den=9, flags=1)):
        p = Prefill(cu, 1, 1, ctx=ctx, want_lse=False, col_capacity=sum(O.keep_count(i + 1, kw["mode"], kw.get("keep_num", 1), kw.get("keep_den", 1),
                                                                                     kw.get("k", 0)) for i in range(nb)))
        gen = torch.Generator(device="cuda").manual_seed(nb)
        s = p.scores.view(nb, nb)
        s.copy_(torch.rand(nb, nb, generator=gen, device="cuda") ** 8)
        s[::3] = torch.randint(0, 40, (s[::3].shape[0], nb), generator=gen, device="cuda") / 64.0   # many ties
        s[5::7] = 0.25                                                                              # nothing but ties
        s[4::9, ::5] = float("nan")
        p.mask(B.make_mask_params(kw["mode"], keep_num=kw.get("keep_num", 1), keep_den=kw.get("keep_den", 1), k=kw.get("k", 0),
                                  flags=kw["flags"]))
        assert p.status() == 0
        rp, col = p.lists_host()
        for i in sorted({0, 1, 256, 257, 1023, 1024, 1030, 1034, 2040, 2046, 2047, nb // 2, nb // 2 + 1, nb - 9, nb - 8, nb - 7, nb - 6, nb - 5,
                         nb - 4, nb - 3, nb - 2, nb - 1}):
            assert col[rp[i]:rp[i + 1]].tolist() == O.select_row(s[i, :i + 1].cpu().numpy(), i, **kw), (nb, i, kw)


@pytest.mark.parametrize("heads_per_band", [1, 2, 3, 4])
@pytest.mark.parametrize("mode", [dict(mode=O.MODE_TOPK_RATIO, keep_num=1, keep_den=5, flags=3), dict(mode=O.MODE_THRESHOLD, threshold=0.01, flags=1)])
def test_packed_chunk_bands(rt, heads_per_band, mode):
    B, Prefill, ctx = rt
    lens, starts = [9000, 333, 4000], [4032, 64, 3968]
    w = W.make_small(seed=55_200, seqlens=lens, hq=4, hkv=2, q_gain=2.0)
    cu, q, cu_q = w.cu_seqlens, [], [0]
    for b, st in enumerate(starts):
        q.append(w.q[cu[b] + st:cu[b + 1]])
        cu_q.append(cu_q[-1] + len(q[-1]))
    p = Prefill(cu, 4, 2, ctx=ctx, want_lse=False, cu_seqlens_q=np.array(cu_q, np.int32))
    p.set_inputs(np.concatenate(q), w.k, w.v, w.wq, w.wk)
    params = B.make_mask_params(mode["mode"], keep_num=mode.get("keep_num", 1), keep_den=mode.get("keep_den", 1),
                                threshold=mode.get("threshold", 0.0), flags=mode["flags"])
    p.gate()
    p.mask(params)
    want = [x.copy() for x in p.lists_host()]
    packed = lambda i: 4096 * ((i // 64) * (i // 64 + 1) // 2) + (i % 64) * 64 * (i // 64 + 1)   # columns rounded up to 64
    rows_bytes = (packed(141) - packed(starts[0] // 64)) * 4
    # with room for the statistics behind the projected vectors (4 heads x 210 blocks x 2 segments x 8 bytes) and without
    for room in (0, 13568):
        p.row_ptr.fill_(-1)
        p.gate_mask(params, band_bytes=max(heads_per_band * rows_bytes + 16, 64 * 141 * 4 + 16) + room)
        assert p.status() == 0
        for x, y in zip(p.lists_host(), want):
            assert np.array_equal(x, y)


# 641 blocks and 16 KV heads: chunks of sixteen blocks; two heads: of two.  The question starts around the edges of both.
@pytest.mark.parametrize("heads", [16, 2])
@pytest.mark.parametrize("lens,starts", [([641 * 64 - 9], [b]) for b in (0, 1, 2, 15, 16, 17, 31, 623, 624, 639, 640)] +
                         [([300 * 64, 65, 341 * 64 - 9], s) for s in ([299, 0, 340], [17, 1, 340], [300, 1, 0], [0, 2, 16])])
def test_pooling_of_chunks(rt, heads, lens, starts):
    import torch
    B, Prefill, ctx = rt
    cu = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
    gen = torch.Generator(device="cuda").manual_seed(7)
    q, k = (torch.randn(int(cu[-1]), heads, 128, generator=gen, device="cuda").bfloat16() for _ in range(2))
    wq, wk = (torch.randn(heads, 128, 128, generator=gen, device="cuda") / 11.3 for _ in range(2))
    part = [q[min(int(cu[b]) + 64 * s, int(cu[b + 1])):int(cu[b + 1])] for b, s in enumerate(starts)]
    cu_q = np.concatenate([[0], np.cumsum([len(x) for x in part])]).astype(np.int32)
    scores = []
    for qq, cuq in ((q, None), (torch.cat(part), cu_q)):
        p = Prefill(cu, heads, heads, ctx=ctx, want_lse=False, cu_seqlens_q=cuq)
        p.q, p.k, p.wq, p.wk = qq, k, wq, wk
        p.scores.fill_(float("nan"))
        p.gate()
        assert p.status() == 0
        scores.append(p.scores)
    at = 0
    for n, s in zip(lens, starts):
        nb = (n + 63) // 64
        a, b = (x[at:at + heads * nb * nb].view(heads, nb, nb)[:, s:] for x in scores)
        tri = torch.ones(nb, nb, dtype=torch.bool, device="cuda").tril()[s:]
        assert torch.equal(a[:, tri], b[:, tri]) and not torch.isnan(a[:, tri]).any()
        at += heads * nb * nb


# rows of the mask: one tile of the scan (8192), a tile and a row, a cluster's eight tiles, and beyond
@pytest.mark.parametrize("hq,seqs", [(1, 1), (2, 4095), (2, 4096), (3, 2731), (17, 3855), (16, 4096), (18, 3641), (40, 3500)])
def test_scan_sizes(rt, hq, seqs):
    B, Prefill, ctx = rt
    p = Prefill(np.arange(seqs + 1, dtype=np.int32), hq, 1, ctx=ctx, want_lse=False)   # a block each: lists of no or one entry
    p.scores.uniform_()
    p.mask(B.make_mask_params(B.SEER_THRESHOLD, threshold=0.7, flags=0))
    assert p.status() == 0
    rp, col = p.lists_host()
    kept = p.scores_host().reshape(-1)[:hq * seqs] > np.float32(0.7)
    assert np.array_equal(rp, np.concatenate([[0], np.cumsum(kept)])) and int(p.nnz.item()) == kept.sum() and not col[:kept.sum()].any()
