"""Scores by one launch: a CTA whose rows touch one or two column tiles keeps their logits between its two sweeps, one with three multiplies them twice.
Around that edge, with a first column tile that is even or odd, in packed batches and chunks: scores equal to the oracle's on every causal
block, nothing written beyond them, and the lists of the one-call form, which takes one sweep whatever the number of tiles."""
import numpy as np
import pytest

from oracle import seer_oracle as O
from paper_2410_13276_b200 import workloads as W

pytestmark = pytest.mark.gpu

# blocks of a row tile of 128 rows: its column tiles (of 64) are those from its first row's sequence start to its last row
CASES = [([64], None),                  # one tile
         ([65], None), ([128], None),   # two, even first
         ([129], None), ([192], None),  # row tile 1: three
         ([100, 60], None),             # row tile 1 (rows 128 to 159, columns from 100): two, odd first
         ([100, 64], None), ([100, 92], None),
         ([100, 93], None), ([100, 100], None),   # three, odd first
         ([128, 70], None), ([127, 65, 3], None), ([64, 64, 64, 64], None), ([1] * 200, None), ([3] * 50, None),
         ([130], [60]), ([100, 60], [1, 60]), ([70, 130], [70, 3])]


@pytest.mark.parametrize("blocks,qblocks", CASES)
def test_scores_around_two_column_tiles(blocks, qblocks):
    from paper_2410_13276_b200 import binding as B
    from paper_2410_13276_b200.prefill import Prefill
    hq, hkv = 2, 1
    lens = [64 * nb - (5 * n) % 64 for n, nb in enumerate(blocks)]
    w = W.make_small(seed=8100 + len(blocks) + blocks[-1], seqlens=lens, hq=hq, hkv=hkv, q_gain=2.0)
    q, cu_q = w.q, None
    if qblocks is not None:
        qlens = [n - 64 * (nb - nq) for n, nb, nq in zip(lens, blocks, qblocks)]
        cu_q = np.concatenate([[0], np.cumsum(qlens)]).astype(np.int32)
        q = np.concatenate([w.q[int(w.cu_seqlens[b + 1]) - qlens[b]:int(w.cu_seqlens[b + 1])] for b in range(len(lens))])
    p = Prefill(w.cu_seqlens, hq, hkv, want_lse=False, cu_seqlens_q=cu_q)
    p.set_inputs(q, w.k, w.v, w.wq, w.wk)
    p.scores.fill_(-7.0)
    before = B.seer_launch_count(p.ctx)
    p.gate()
    assert p.status() == 0 and B.seer_launch_count(p.ctx) - before == 2   # pooling and one launch of scores
    got = O.unflatten_scores(p.scores_host(), w.cu_seqlens, 64, hq)
    ref = O.gate_scores(w.q, w.k, w.wq, w.wk, w.cu_seqlens, 64)
    for b, (g, r) in enumerate(zip(got, ref)):
        nb = blocks[b]
        written = np.tril(np.ones((nb, nb), bool))
        written[:nb - (nb if qblocks is None else qblocks[b])] = False
        x, y = g[:, written].astype(np.float64), r[:, written]
        # logits from three bf16 planes a factor, fp32 sums: about 2^-17 of a logit of magnitude 10, then the exponential
        assert np.all(np.abs(x - y) <= np.where(y < 1e-30, 1e-33, 1e-3 * y))
        assert np.all(g[:, ~written] == -7.0)
    params = B.make_mask_params(B.SEER_TOPK_RATIO, keep_num=1, keep_den=5, flags=3)
    p.mask(params)
    rp, col = p.lists_host()
    p.gate_mask(params)
    assert p.status() == 0
    rp1, col1 = p.lists_host()
    assert np.array_equal(rp, rp1) and np.array_equal(col, col1)
