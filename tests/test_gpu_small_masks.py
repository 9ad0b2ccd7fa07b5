"""Masks of few short rows, counted and scanned by one CTA: around its limits (TopK 384 rows of up to 48 blocks or 256 of up to 64, thresholds
512 rows of up to 32 or 384 of up to 64; beyond, two kernels), with ties,
NaN, forced blocks, dense tails, chunks, a capacity that does not suffice, and scores that begin on any element."""
import numpy as np
import pytest

from oracle import seer_oracle as O

pytestmark = pytest.mark.gpu

KW = [dict(mode=O.MODE_TOPK_RATIO, keep_num=1, keep_den=3, flags=3), dict(mode=O.MODE_TOPK_COUNT, k=4, flags=0), dict(mode=O.MODE_THRESHOLD, threshold=0.5, flags=2)]


@pytest.mark.parametrize("lens,hq", [([5], 1), ([64 * 64], 8), ([64 * 64, 1], 8), ([64 * 64 + 1], 2), ([700, 0, 64, 4000, 65], 4), ([130] * 43, 4), ([64] * 511, 1), ([64] * 512, 1),
                                     ([64] * 513, 1), ([64 * 64], 4), ([64 * 49, 64 * 15, 1], 4), ([64 * 48], 8), ([64 * 48, 1], 8), ([64 * 64], 6), ([64 * 64, 1], 6),
                                     ([64 * 49], 8), ([64 * 32], 16), ([64 * 33 - 5, 64 * 31], 6), ([64 * 33, 64 * 31], 8), ([64 * 32] * 2 + [64], 8)])
@pytest.mark.parametrize("tail", [0, 2])
def test_lists_of_few_short_rows(lens, hq, tail):
    import torch
    from paper_2410_13276_b200 import binding as B
    from paper_2410_13276_b200.prefill import Prefill
    rng = np.random.default_rng(len(lens) + hq)
    cu = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
    blocks = [(n + 63) // 64 for n in lens]
    rows = hq * sum(blocks)

    def few(mode):
        if mode == O.MODE_THRESHOLD:
            return rows <= (512 if max(blocks) <= 32 else 384 if max(blocks) <= 64 else 0)
        return rows <= (384 if max(blocks) <= 48 else 256 if max(blocks) <= 64 else 0)

    full = [np.round(rng.random((hq, nb, nb)), 1).astype(np.float32) for nb in blocks]
    for s in full:
        s[rng.random(s.shape) < 0.1] = np.nan
    half = [min(n, n - 64 * (nb // 2)) for n, nb in zip(lens, blocks)]   # the later blocks of each sequence as a chunk
    for chunk in (False, True):
        p = Prefill(cu, hq, 1, want_lse=False, cu_seqlens_q=np.concatenate([[0], np.cumsum(half)]).astype(np.int32) if chunk else None)
        for shift in (0, 1):
            p.scores = torch.full((sum(s.size for s in full) + 1,), float("nan"), device="cuda")[shift:]
            p.set_scores(O.flatten_scores(full))
            for kw in KW:
                if chunk:
                    rp, col = O.block_mask_chunk([s[:, nb - (h + 63) // 64:] for s, nb, h in zip(full, blocks, half)], dense_tail=tail, **kw)
                else:
                    rp, col = O.block_mask(full, dense_tail=tail, **kw)
                params = B.make_mask_params(kw["mode"], keep_num=kw.get("keep_num", 1), keep_den=kw.get("keep_den", 1), k=kw.get("k", 0),
                                            threshold=kw.get("threshold", 0.0), flags=kw["flags"], dense_tail=tail)
                p.row_ptr.fill_(-7)
                p.nnz.fill_(-7)
                before = B.seer_launch_count(p.ctx)
                p.mask(params)
                assert p.status() == 0 and B.seer_launch_count(p.ctx) - before == (2 if few(kw["mode"]) else 3)
                got_rp, got = p.lists_host()
                assert np.array_equal(got_rp, rp) and np.array_equal(got[:len(col)], col) and int(p.nnz.item()) == len(col)
                if len(col) > 1:
                    p.col_capacity = len(col) - 1
                    p.mask(params)
                    assert p.status() == 4 and int(p.nnz.item()) == len(col)   # SEER_ERR_CAPACITY
                    p.col_capacity = p.col_idx.numel()
