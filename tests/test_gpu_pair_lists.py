"""Attention where query blocks 2u and 2u + 1 list the same blocks: o and lse equal those of the launch without a work counter, which takes every
query block by itself, bit for bit (the same rows, sums in the same order).  The words behind the counter say which kernel ran: the
check of the lists answers there."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def problem(lens, hq, hkv, block=64, qlens=None, seed=0):
    import torch
    from paper_2410_13276_b200.prefill import Prefill
    cu = lambda x: np.concatenate([[0], np.cumsum(x)]).astype(np.int32)
    p = Prefill(cu(lens), hq, hkv, block=block, cu_seqlens_q=None if qlens is None else cu(qlens))
    g = torch.Generator(device="cuda"); g.manual_seed(seed + sum(lens))
    draw = lambda *s: torch.randn(*s, generator=g, device="cuda")
    p.q, p.k, p.v = (2 * draw(p.Tq, hq, 128)).bfloat16(), draw(p.T, hkv, 128).bfloat16(), draw(p.T, hkv, 128).bfloat16()
    p.wq, p.wk = draw(hq, 128, 128) / 11.3, draw(hkv, 128, 128) / 11.3
    p.scores.zero_()
    return p


def both_ways(p, by_pairs):
    import torch
    from paper_2410_13276_b200 import binding as B
    outs = []
    answer = p.ws[4:256].view(torch.int32)                         # behind the work counter: one word for each block of the check
    for left in (None, 0, 0x7f7f7f7f):                             # without a workspace; with one that something has been left in
        p.o.fill_(7.0); p.lse.fill_(7.0)
        if left is not None:
            answer.fill_(left)
        before = B.seer_launch_count(p.ctx)
        p.attn(dynamic=left is not None)
        torch.cuda.synchronize()
        assert p.status() == 0
        if left is not None:
            # the check, the kernel for single blocks and the one for pairs, of which one returns at once; every word is this call's
            assert B.seer_launch_count(p.ctx) - before == 3
            said = set(answer.tolist())
            assert 0x7f7f7f7f not in said and (0 not in said) == by_pairs and (len(said) == 1 or not by_pairs)
        outs.append((p.o.clone().view(torch.int16), p.lse.clone().view(torch.int32)))
    for o, lse in outs[1:]:
        assert torch.equal(outs[0][0], o) and torch.equal(outs[0][1], lse)


def maxima_by_pairs(p):
    """Whether CTA 0 takes its share of the block maxima by pairs: it loses its first copy, so entries of its items stay as they were.  By pairs those are
    both lists of a pair of query blocks; otherwise the blocks of a pair go to a stream each, and one stream loses the copy, while the other is through
    with its items long before the wait runs out."""
    import torch
    from paper_2410_13276_b200 import binding as B
    p.bmax = torch.full((max(p.col_idx.numel(), 1),), -1.0, device="cuda")
    B.seer_debug_lost_wait(p.ctx, 5_000, 0)
    try:
        before = B.seer_launch_count(p.ctx)
        p.block_max()
        assert B.seer_launch_count(p.ctx) - before == 1
        assert B.STATUS_NAMES[B.seer_poll_device_status(p.ctx)] == "SEER_ERR_TIMEOUT"
    finally:
        B.seer_debug_lost_wait(p.ctx, 2_000_000, -1)
    rp, _ = p.lists_host()
    left = (p.bmax[:int(rp[-1])] == -1.0).cpu().numpy()
    rows = set(np.unique(np.searchsorted(rp, np.flatnonzero(left), side="right") - 1).tolist())
    nbs = (np.diff(p.cu) + 63) // 64
    base, both, lone = 0, 0, 0
    for n, nq in zip(nbs, nbs if p.cu_q is None else np.diff(p.cu_q)):
        first = n - ((nq + 63) // 64 if p.cu_q is not None else n)
        for h in range(p.hq):
            for i in range(0, n, 2):
                here = [r in rows for r, j in ((base + h * n + i, i), (base + h * n + i + 1, i + 1)) if first <= j < n and rp[r + 1] > rp[r]]
                if len(here) == 2:
                    both, lone = both + all(here), lone + (sum(here) == 1)
        base += p.hq * n
    assert both + lone > 0 and (both == 0 or lone == 0)
    return both > 0


def maxima_of_groups(p, by_pairs=None):
    """Block maxima: equal to those of each KV head's problem by itself, which is below the size from which shares are pairs of query blocks."""
    import torch
    from paper_2410_13276_b200 import binding as B
    from paper_2410_13276_b200.prefill import Prefill
    p.attn()
    took = maxima_by_pairs(p)
    assert by_pairs is None or took == by_pairs
    p.bmax.fill_(-1.0)
    got = p.block_max()
    rp, col = p.lists_host()
    nbs, group = (np.diff(p.cu) + 63) // 64, p.hq // p.hkv
    for g in range(p.hkv):
        part = Prefill(p.cu, group, 1, cu_seqlens_q=p.cu_q, ctx=p.ctx)
        part.q, part.k, part.lse = p.q[:, g * group:(g + 1) * group].contiguous(), p.k[:, g:g + 1].contiguous(), p.lse[g * group:(g + 1) * group].contiguous()
        base, spans = 0, []
        for nb in nbs:
            spans.append((base + g * group * nb, base + (g + 1) * group * nb))
            base += p.hq * nb
        lens = np.concatenate([np.diff(rp[a:b + 1]) for a, b in spans])
        part.set_lists(np.concatenate([[0], np.cumsum(lens)]).astype(np.int32), np.concatenate([col[rp[a]:rp[b]] for a, b in spans]).astype(np.int32))
        want = part.block_max()[:int(lens.sum())]
        assert torch.equal(torch.cat([got[int(rp[a]):int(rp[b])] for a, b in spans]).view(torch.int32), want.view(torch.int32)), g
    assert p.status() == 0


# every causal block: odd and even block counts, ragged ends, batches in any order with sequences of one block, chunks from odd and even blocks
@pytest.mark.parametrize("lens,qlens,hq,hkv", [([16421], None, 32, 8), ([700, 1, 12032, 64, 4100], None, 64, 16), ([16500, 9000], [16500 - 64 * 33, 9000 - 64 * 58], 40, 8)])
def test_dense_lists(lens, qlens, hq, hkv):
    from paper_2410_13276_b200 import binding as B
    p = problem(lens, hq, hkv, qlens=qlens)
    p.mask(B.make_mask_params(B.SEER_TOPK_COUNT, k=1 << 20, flags=B.SEER_FORCE_DIAG))
    both_ways(p, True)
    maxima_of_groups(p, True)


@pytest.mark.parametrize("lens,qlens", [([23500], None), ([16400, 127, 11000], None), ([23500, 2000], [23500 - 128 * 57, 2000 - 128])])
def test_lists_of_128_token_blocks(lens, qlens):
    from paper_2410_13276_b200 import binding as B
    p = problem(lens, 32, 8, block=128, qlens=qlens)
    p.gate()
    p.mask(B.make_mask_params(B.SEER_TOPK_RATIO, keep_num=1, keep_den=5, flags=B.SEER_FORCE_DIAG | B.SEER_FORCE_SINK))
    both_ways(p, True)


# lists in any order, of no block to all, the second block with one more (its own, or an earlier one) or not; values and keys that are not finite
@pytest.mark.parametrize("spoilt", [False, True])
def test_hand_made_lists(spoilt):
    import torch
    lens, hq = [16400, 3000], 32
    p = problem(lens, hq, 8)
    r = np.random.default_rng(11)
    rows, at = [], 0
    for n in lens:
        nb = (n + 63) // 64
        for h in range(hq):
            for i in range(0, nb, 2):
                shared = r.permutation(i)[:r.choice([0, 0, 1, 2, 3, 5, 30, i])].tolist()
                if r.random() < 0.7:
                    shared.append(i)
                more = r.choice(3)
                rows.append(shared)
                if i + 1 < nb:
                    at = max(at, len(rows) - 1, key=lambda k: len(rows[k]))
                    rows.append(shared + ([] if more == 0 else [i + 1] if more == 1 else [int(r.integers(0, i + 2))]))
    if spoilt:
        p.v[64 * 101 + 5, 0, 3] = float("inf"); p.v[64 * 40, 2, 100] = float("nan"); p.v[16400 + 64 * 7 + 63, 5, 0] = float("-inf")
        p.k[64 * 77 + 9, 1, 4] = float("inf"); p.k[64 * 30 + 2, 3] *= 60; p.q[64 * 90:64 * 96] *= 20
    p.set_lists(np.concatenate([[0], np.cumsum([len(x) for x in rows])]).astype(np.int32), np.array([j for x in rows for j in x], np.int32))
    both_ways(p, True)
    maxima_of_groups(p, True)
    # a single pair that differs, by an entry or by a length, or whose own block is not its last entry: each query block by itself
    for change in (lambda x: x[1:], lambda x: [x[1], x[0]] + x[2:], lambda x: x + x[:2]):
        other = [change(x) if k == at else x for k, x in enumerate(rows)]
        p.set_lists(np.concatenate([[0], np.cumsum([len(x) for x in other])]).astype(np.int32), np.array([j for x in other for j in x], np.int32))
        both_ways(p, False)
    maxima_of_groups(p)                                            # (the CTA with that pair takes its share block by block, the others theirs by pairs)


# neighbouring query blocks list different blocks
@pytest.mark.parametrize("lens,qlens,hq,hkv", [([8192], None, 32, 8), ([700, 1, 12032, 64, 4100], None, 64, 16), ([16500, 9000], [16500 - 64 * 33, 9000 - 64 * 58], 40, 8)])
def test_maxima_of_lists_that_differ(lens, qlens, hq, hkv):
    from paper_2410_13276_b200 import binding as B
    p = problem(lens, hq, hkv, qlens=qlens)
    p.gate()
    p.mask(B.make_mask_params(B.SEER_TOPK_RATIO, keep_num=1, keep_den=10, flags=B.SEER_FORCE_DIAG))
    maxima_of_groups(p, False)


@pytest.mark.parametrize("lost_tile", [0, 130, 300])
def test_a_lost_copy(lost_tile):
    """A V copy that CTA 0 never issues: the call returns with the status, the rows of the items it had in hand stay as they were, all others are
    right, and the next call is normal."""
    import torch
    from paper_2410_13276_b200 import binding as B
    p = problem([16384], 32, 8)
    p.mask(B.make_mask_params(B.SEER_TOPK_COUNT, k=1 << 20, flags=B.SEER_FORCE_DIAG))
    both_ways(p, True)
    o, lse = p.o.clone(), p.lse.clone()
    B.seer_debug_lost_wait(p.ctx, 5_000, lost_tile)
    try:
        p.o.fill_(float("nan")); p.lse.fill_(float("nan"))
        p.attn()
        status = B.seer_poll_device_status(p.ctx)
    finally:
        B.seer_debug_lost_wait(p.ctx, 2_000_000, -1)
    assert B.STATUS_NAMES[status] == "SEER_ERR_TIMEOUT"
    missing = torch.isnan(p.lse)                                   # [heads, tokens]: whole items of 128 rows
    assert torch.equal(torch.isnan(p.o.float()).all(-1).T, missing) and torch.equal(torch.isnan(p.o.float()).any(-1).T, missing)
    items = missing.view(32, -1, 128)
    assert torch.equal(items.all(-1), items.any(-1)) and 1 <= int(items.any(-1).sum()) <= 5
    assert torch.equal(p.lse[~missing], lse[~missing]) and torch.equal(p.o.permute(1, 0, 2)[~missing], o.permute(1, 0, 2)[~missing])
    both_ways(p, True)
    assert torch.equal(p.o, o) and torch.equal(p.lse, lse)
