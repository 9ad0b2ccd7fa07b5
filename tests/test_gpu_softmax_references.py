"""Softmax references of the tcgen05 attention kernel: scores that rise, tile by tile, by amounts around the distance at
which a row's reference has to move (a tile sum of 2^60 relative to the first block's maximum, so scores 2^54 to 2^60 above
it), and around the ends of the range of fp32 (2^126, 2^128), upwards and downwards, against the fp64 oracle."""
import math

import numpy as np
import pytest

from oracle import seer_oracle as O
from paper_2410_13276_b200 import workloads as W

pytestmark = pytest.mark.gpu

LOG2_PER_UNIT = 16.0 / math.sqrt(128) / math.log(2.0)   # a key level of 1 moves the scores by this many powers of two


@pytest.mark.parametrize("where", ["later", "first", "stairs"])
@pytest.mark.parametrize("rise", [6, 32, 52, 54, 56, 58, 60, 62, 92, 120, 126, 130, 300])
def test_scores_that_rise_by_powers_of_two(rise, where):
    import torch
    from paper_2410_13276_b200 import binding as B
    from paper_2410_13276_b200.prefill import Prefill
    S = 500                                              # 8 blocks, the last one ragged: four tiles in the last rows
    r = np.random.default_rng(77)
    q = r.standard_normal((S, 2, 128), dtype=np.float32) * 0.3
    k = r.standard_normal((S, 1, 128), dtype=np.float32) * 0.3
    v = r.standard_normal((S, 1, 128), dtype=np.float32)
    q[:, 0, 0], q[:, 1, 0] = 16.0, np.where(np.arange(S) % 3 == 0, -16.0, 16.0)   # head 1: some columns fall instead
    level = np.zeros(8)
    if where == "later":
        level[5] = rise
    elif where == "first":
        level[0] = -rise                                 # the keys the first references are taken from are the low ones
    else:
        level[:] = rise * np.arange(8) / 3.0
    k[:, 0, 0] = np.repeat(level / LOG2_PER_UNIT, 64)[:S]
    k[::37, 0, 0] *= 0.5                                 # not every key of a block moves
    cu = np.array([0, S], np.int32)
    bits = [W.f32_to_bf16_bits(x) for x in (q, k, v)]
    p = Prefill(cu, 2, 1)
    p.set_inputs(*bits)
    rp, col = O.full_causal_lists(cu, 64, 2)
    p.set_lists(rp, col)
    p.o.fill_(float("nan"))
    p.attn()
    assert p.status() == 0
    o_ref, lse_ref = O.sparse_attention(*bits, cu, rp, col, 2, 1, 64, 1 / math.sqrt(128))
    x = p.o_host().astype(np.float64)
    # bf16 probabilities and results: 2^-9 each, averaged over the keys; per row within 1e-2 in the 2-norm
    err = np.linalg.norm(x - o_ref, axis=-1) / np.linalg.norm(o_ref, axis=-1)
    assert err.max() <= 1e-2, err.max()
    # lse: fp32 scores of magnitude |s| carry 2^-22 |s| from their 128-term sums, the sum of probabilities 2e-4 (ex2, cubic)
    lse = p.lse_host()
    assert np.all(np.abs(lse - lse_ref) <= 4e-4 + 2.0 ** -20 * np.abs(lse_ref)), np.abs(lse - lse_ref).max()
