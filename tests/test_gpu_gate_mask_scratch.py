"""The one-call gate + mask in a scratch that the statistics of its rows crowd: no more bands than the scores alone need in one band, at most twice
as many otherwise, and the lists of the two separate calls whatever the scratch."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# (lens, chunk, query heads, KV heads)
SHAPES = [([700], None, 32, 8), ([256] * 300, None, 32, 8), ([64, 700, 130, 0, 2000], None, 8, 2), ([2048], None, 4, 1), ([3000, 64, 64, 64] * 4, None, 8, 8),
          ([4096] * 3 + [90], [64, 4096, 200, 90], 8, 2), ([9000, 300, 300], None, 4, 2), ([700, 65], [60, 65], 4, 4)]


@pytest.mark.parametrize("lens,qlens,hq,hkv", SHAPES)
@pytest.mark.parametrize("share", [1.0, 1.05, 0.97, 0.6, 0.25])
def test_launches_and_lists_of_a_narrow_scratch(lens, qlens, hq, hkv, share):
    import torch
    from paper_2410_13276_b200 import binding as B
    from paper_2410_13276_b200.prefill import Prefill
    gen = torch.Generator(device="cuda").manual_seed(len(lens) + hq)
    rand = lambda *s: torch.randn(*s, generator=gen, device="cuda")
    cu = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
    if qlens is not None:                              # a chunk starts on a block
        qlens = [n - 64 * ((n - q) // 64) for n, q in zip(lens, qlens)]
    cu_q = None if qlens is None else np.concatenate([[0], np.cumsum(qlens)]).astype(np.int32)
    p = Prefill(cu, hq, hkv, want_lse=False, cu_seqlens_q=cu_q)
    p.q, p.k = (2.0 * rand(p.Tq, hq, 128)).bfloat16(), rand(p.T, hkv, 128).bfloat16()
    p.wq, p.wk = rand(hq, 128, 128) / 2, rand(hkv, 128, 128) / 2
    elems = B.seer_scores_elems(p.shape)
    blocks = [(n + 63) // 64 for n in lens]
    band = max(int(4 * elems * share) + 16, 64 * 4 * max(blocks) + 16)
    # bands that scores alone take in this scratch: whole sequences, else whole heads of one (packed), else 64-row tiles
    cap = (B.seer_gate_mask_workspace_bytes(p.shape, band) - B.seer_workspace_bytes(p.shape)) // 4 - 4
    packed = lambda i: 4096 * (i // 64 * (i // 64 + 1) // 2) + (i % 64) * 64 * (i // 64 + 1)
    bands, open_elems = 0, None
    for b, nb in enumerate(blocks):
        first = 0 if qlens is None else (lens[b] - qlens[b]) // 64 if qlens[b] else nb
        if hq * nb * nb <= cap:
            if open_elems is None or open_elems + hq * nb * nb > cap:
                bands, open_elems = bands + 1, 0
            open_elems += hq * nb * nb
            continue
        open_elems = None
        per_head = packed(nb) - packed(first)
        bands += -(-hq // (cap // per_head)) if 0 < per_head <= cap else 1 if per_head == 0 else hq * -(-(-(-nb // 64)) // (cap // (64 * nb)))
    for params in (B.make_mask_params(B.SEER_TOPK_RATIO, keep_num=1, keep_den=4, flags=3), B.make_mask_params(B.SEER_THRESHOLD, threshold=0.05, flags=1)):
        p.gate()
        p.mask(params)
        assert p.status() == 0
        rp, n = p.row_ptr.clone(), int(p.nnz.item())
        col = p.col_idx[:n].clone()
        p.row_ptr.fill_(-7)
        p.col_idx.fill_(-7)
        before = B.seer_launch_count(p.ctx)
        p.gate_mask(params, band_bytes=band)
        launches = B.seer_launch_count(p.ctx) - before
        assert p.status() == 0
        assert torch.equal(p.row_ptr, rp) and torch.equal(p.col_idx[:n], col) and int(p.nnz.item()) == n
        # pooling and statistics, then scores, counts, scan and lists of every band
        assert launches <= 2 + 4 * (bands if bands == 1 else 2 * bands), (launches, bands)
