"""Attention over lists of every small length: tiles of two blocks, so lists of one block (no second half), of odd and of even
length, across the two score buffers and the four item slots, with the diagonal first, last or absent, an entry that is
rejected in either half, and rows of different lengths next to one another; against the fp64 oracle.  The block maxima of the
same lists, whose pipeline has four score buffers and five key units."""
import math

import numpy as np
import pytest

from oracle import seer_oracle as O
from paper_2410_13276_b200 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lengths,bad", [((1,), None), ((2,), None), ((3,), None), ((4,), None), ((5,), None), ((0, 1, 2, 3, 4, 5, 6, 7, 8, 9), None),
                                         ((1, 9, 0, 0, 2), None), ((16, 17, 33), None), ((4,), 0), ((4,), 1), ((3,), 2), ((1,), 0)])
def test_list_lengths(lengths, bad):
    from paper_2410_13276_b200 import binding as B
    from paper_2410_13276_b200.prefill import Prefill
    nb, hq = 40, 4
    w = W.make_small(seed=140, seqlens=[nb * 64 - 7], hq=hq, hkv=2, q_gain=2.0)
    r = np.random.default_rng(sum(lengths))
    rp, col = [0], []
    for h in range(hq):
        for i in range(nb):
            n = min(lengths[(h * nb + i) % len(lengths)], i + 1)
            row = sorted(r.choice(i + 1, n, replace=False).tolist())
            if n and (i + h) % 3:
                row = row[:-1] + [i] if i not in row else row
            if bad is not None and len(row) > bad and i % 5 == 2:
                row[bad] = nb + 3                            # not causal: skipped, and the status says so
            col += row
            rp.append(len(col))
    rp, col = np.array(rp, np.int32), np.array(col, np.int32)
    p = Prefill(w.cu_seqlens, hq, 2)
    p.set_inputs(w.q, w.k, w.v, w.wq, w.wk)
    p.set_lists(rp, col)
    p.o.fill_(float("nan"))
    p.attn()
    assert p.status() == (0 if bad is None else 5)
    o_ref, lse_ref = O.sparse_attention(w.q, w.k, w.v, w.cu_seqlens, rp, col, hq, 2, 64, 1 / math.sqrt(128))
    x = p.o_host().astype(np.float64)
    live = np.linalg.norm(o_ref, axis=-1) > 0
    assert np.all(x[~live] == 0)
    # bf16 probabilities and results: 2^-9 each, averaged over the keys; per row within 1e-2 in the 2-norm
    err = np.linalg.norm(x - o_ref, axis=-1)[live] / np.linalg.norm(o_ref, axis=-1)[live]
    assert err.max() <= 1e-2, err.max()
    lse = p.lse_host().astype(np.float64)
    fin = np.isfinite(lse_ref)
    assert np.array_equal(fin, np.isfinite(lse)) and np.all(np.abs(lse[fin] - lse_ref[fin]) <= 4e-4 + 2.0 ** -20 * np.abs(lse_ref[fin]))
    if bad is None:
        got = p.block_max().cpu().numpy()[:len(col)].astype(np.float64)
        assert p.status() == 0
        ref = O.maxpool_listed_blocks(w.q, w.k, w.cu_seqlens, rp, col, hq, 2, 64, 1 / math.sqrt(128))
        # bf16 operands, fp32 sums of magnitude 10, the lse within its own bound
        assert np.all(np.abs(got - ref) <= 1e-2 * np.abs(ref) + 1e-7)
