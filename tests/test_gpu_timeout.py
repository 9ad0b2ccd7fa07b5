"""The bounded waits of the tcgen05 attention kernel, exercised without faulting anything (needs a B200).

seer_debug_lost_wait makes exactly one wait run out: the first stream of CTA 0 never issues the V copy of one of its
tiles (the block maxima: the K copy), so the MMA issuer's wait for that copy expires after the (shortened) limit.  What must then hold: the device
status is SEER_ERR_TIMEOUT, the kernel has returned (the call and the poll come back), every row that does not belong
to the stream that lost its copy equals the normal run bit for bit, and the context goes on working: the next call
without the hook gives the normal result (so the tensor memory of the aborted CTA was freed and no barrier is left
half-armed).
"""
import numpy as np
import pytest

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
    B.seer_debug_lost_wait(ctx, 2_000_000, -1)
    ctx.close()


@pytest.mark.parametrize("lost_tile", [0, 3])
def test_a_lost_copy_raises_timeout_and_the_context_survives(rt, lost_tile):
    import torch
    B, Prefill, ctx = rt
    hq, hkv, S = 8, 2, 4096
    w = W.make_small(seed=4242, seqlens=[S], hq=hq, hkv=hkv)
    p = Prefill(w.cu_seqlens, hq, hkv, ctx=ctx, want_lse=True)
    p.set_inputs(w.q, w.k, w.v, w.wq, w.wk)
    params = B.make_mask_params(B.SEER_TOPK_RATIO, keep_num=1, keep_den=2, flags=B.SEER_FORCE_DIAG | B.SEER_FORCE_SINK)
    p.gate(); p.mask(params)
    p.attn(dynamic=False); torch.cuda.synchronize()
    assert p.status() == 0
    o_ref, lse_ref = p.o.clone(), p.lse.clone()

    # rows (head, query block) of the first stream of CTA 0: work items 0, 2 * grid, ... in the kernel's order
    # (KV head, query block from the last to the first, head within the group), two streams per CTA
    nb = S // 64
    rows = hq * nb
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    grid = min(sms, (rows + 1) // 2)
    group = hq // hkv
    lost_rows = set()
    for wi in range(0, rows, 2 * grid):
        g, rem = divmod(wi, nb * group)
        lost_rows.add((g * group + rem % group, nb - 1 - rem // group))

    B.seer_debug_lost_wait(ctx, 2_000, lost_tile)                  # 2 ms instead of 2 s
    try:
        p.o.fill_(float("nan")); p.lse.fill_(float("nan"))
        p.attn(dynamic=False)                                      # static deal: the rows of the stream that loses its copy are known
        status = B.seer_poll_device_status(ctx)                    # synchronises: the kernel has returned
    finally:
        B.seer_debug_lost_wait(ctx, 2_000_000, -1)
    assert B.STATUS_NAMES[status] == "SEER_ERR_TIMEOUT"
    o_bad, lse_bad = p.o.clone(), p.lse.clone()
    keep = torch.ones((hq, nb), dtype=torch.bool)
    for h, i in lost_rows:
        keep[h, i] = False
    keep_tok = keep.repeat_interleave(64, dim=1).cuda()            # [hq, S]
    assert torch.equal(o_bad.permute(1, 0, 2)[keep_tok], o_ref.permute(1, 0, 2)[keep_tok]), "a row of another stream changed"
    assert torch.equal(lse_bad[keep_tok], lse_ref[keep_tok])
    # the item that lost its copy cannot have been written
    h0, i0 = 0, nb - 1
    assert torch.isnan(o_bad[i0 * 64:(i0 + 1) * 64, h0].float()).all()

    # the context still works and the result is the normal one
    p.o.fill_(float("nan")); p.lse.fill_(float("nan"))
    p.attn(); torch.cuda.synchronize()                             # (with the work counter: the same result bit for bit)
    assert p.status() == 0
    assert torch.equal(p.o, o_ref) and torch.equal(p.lse, lse_ref)


@pytest.mark.parametrize("keep,lost_tile,lost_item", [(32, 15, 0), (2, 0, 0), (2, 1, 1), (3, 1, 0), (3, 3, 1), (1, 0, 0), (1, 1, 1)])
def test_a_lost_last_copy_leaves_the_items_rows_unwritten(rt, keep, lost_tile, lost_item):
    """The copy of an item's last tile: the group finds out at the item's merge, when everything but O is settled.  Neither o nor lse of any of the
    item's rows is written (lists of two blocks or more are merged by pairs of warps, a list of one block by one), items that the stream
    had finished are, and nothing of another stream changes."""
    import torch
    B, Prefill, ctx = rt
    hq, hkv, S = 8, 2, 4096
    w = W.make_small(seed=4243, seqlens=[S], hq=hq, hkv=hkv)
    p = Prefill(w.cu_seqlens, hq, hkv, ctx=ctx, want_lse=True)
    p.set_inputs(w.q, w.k, w.v, w.wq, w.wk)
    p.gate(); p.mask(B.make_mask_params(B.SEER_TOPK_COUNT, k=keep, flags=B.SEER_FORCE_DIAG))
    p.attn(dynamic=False); torch.cuda.synchronize()
    assert p.status() == 0
    o_ref, lse_ref = p.o.clone(), p.lse.clone()
    nb, group = S // 64, hq // hkv
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    rows = []                                                      # (head, query block) of the items of CTA 0's first stream, in order
    for wi in range(0, hq * nb, 2 * min(sms, hq * nb // 2)):
        g, rem = divmod(wi, nb * group)
        rows.append((g * group + rem % group, nb - 1 - rem // group))
    assert lost_item < len(rows) and all(i + 1 >= keep for _, i in rows[:lost_item + 1])   # every list so far has `keep` blocks
    B.seer_debug_lost_wait(ctx, 2_000, lost_tile)
    try:
        p.o.fill_(float("nan")); p.lse.fill_(float("nan"))
        p.attn(dynamic=False)
        status = B.seer_poll_device_status(ctx)
    finally:
        B.seer_debug_lost_wait(ctx, 2_000_000, -1)
    assert B.STATUS_NAMES[status] == "SEER_ERR_TIMEOUT"
    for n, (h, i) in enumerate(rows):
        o, lse = p.o[i * 64:(i + 1) * 64, h], p.lse[h, i * 64:(i + 1) * 64]
        if n < lost_item:
            assert torch.equal(o, o_ref[i * 64:(i + 1) * 64, h]) and torch.equal(lse, lse_ref[h, i * 64:(i + 1) * 64])
        elif n == lost_item:
            assert torch.isnan(o.float()).all() and torch.isnan(lse).all()
        p.o[i * 64:(i + 1) * 64, h] = o_ref[i * 64:(i + 1) * 64, h]
        p.lse[h, i * 64:(i + 1) * 64] = lse_ref[h, i * 64:(i + 1) * 64]
    assert torch.equal(p.o, o_ref) and torch.equal(p.lse, lse_ref), "a row of another stream changed"
    p.o.fill_(float("nan")); p.lse.fill_(float("nan"))
    p.attn(); torch.cuda.synchronize()
    assert p.status() == 0 and torch.equal(p.o, o_ref) and torch.equal(p.lse, lse_ref)


@pytest.mark.parametrize("S,hq,hkv,lost_tile", [(4096, 8, 2, 0), (4096, 8, 2, 37), (8192, 32, 8, 0), (8192, 32, 8, 31), (8192, 32, 8, 32), (8192, 32, 8, 333)])
def test_a_lost_copy_of_the_block_maxima(rt, S, hq, hkv, lost_tile):
    """A K copy that CTA 0 never issues, query block by query block (4096 tokens) and by pairs (8192: 2^18 causal blocks): the call returns with the
    status, entries of CTA 0's share are right or as they were, all others are right, and the next call is normal."""
    import torch
    B, Prefill, ctx = rt
    w = W.make_small(seed=4244, seqlens=[S], hq=hq, hkv=hkv)
    p = Prefill(w.cu_seqlens, hq, hkv, ctx=ctx, want_lse=True)
    p.set_inputs(w.q, w.k, w.v, w.wq, w.wk)
    p.scores.zero_()
    p.mask(B.make_mask_params(B.SEER_TOPK_COUNT, k=1 << 20, flags=B.SEER_FORCE_DIAG))
    p.attn()
    want = p.block_max().clone()
    assert p.status() == 0
    B.seer_debug_lost_wait(ctx, 5_000, lost_tile)
    try:
        p.bmax.fill_(-1.0)
        p.block_max()
        status = B.seer_poll_device_status(ctx)
    finally:
        B.seer_debug_lost_wait(ctx, 2_000_000, -1)
    assert B.STATUS_NAMES[status] == "SEER_ERR_TIMEOUT"
    missing = p.bmax == -1.0
    assert torch.equal(p.bmax[~missing], want[~missing])
    rows = torch.searchsorted(p.row_ptr.long(), torch.nonzero(missing)[:, 0], right=True).unique().numel()
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert 1 <= rows <= 2 * (-(-hq * (S // 64) // (2 * sms)) + 1)
    p.bmax.fill_(-1.0)
    p.block_max()
    assert p.status() == 0 and torch.equal(p.bmax, want)


def test_lost_wait_hook_rejects_a_zero_limit(rt):
    B, _, ctx = rt
    with pytest.raises(B.SeerError):
        B.seer_debug_lost_wait(ctx, 0, -1)
