"""The one-call gate + mask forms a row's scores where it selects, from logits and the statistics of the row's segments: lists equal to those
of the two separate calls around the edges of the segments (256 columns, 1024 beyond 2048 blocks), of the parts that a CTA walks, and
of the selection kernels (2048, 8192 blocks; beyond 16384 scores are written), with and without room for the statistics, for packed
batches and chunks, and for rows whose logits are infinite or not numbers."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lens,hq,hkv,tail", [([256 * 64], 2, 1, 1), ([257 * 64 - 1], 4, 4, 257), ([1025 * 64], 3, 1, 40), ([2048 * 64 - 5], 2, 2, 200),
                                             ([2049 * 64], 3, 3, 2049), ([8193 * 64], 1, 1, 130), ([16385 * 64 - 3], 1, 1, 70),
                                             ([300 * 64, 64, 0, 900 * 64 - 7, 130], 2, 1, 3)])
@pytest.mark.parametrize("spoilt", [False, True])
def test_lists_equal_those_of_the_two_calls(lens, hq, hkv, tail, spoilt):
    import torch
    from paper_2410_13276_b200 import binding as B
    from paper_2410_13276_b200.prefill import Prefill
    gen = torch.Generator(device="cuda").manual_seed(sum(lens))
    cu = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
    rand = lambda *s: torch.randn(*s, generator=gen, device="cuda")
    # 2.0: probabilities over several octaves
    q, k = (2.0 * rand(int(cu[-1]), hq, 128)).bfloat16(), rand(int(cu[-1]), hkv, 128).bfloat16()
    wq, wk = rand(hq, 128, 128) / 2, rand(hkv, 128, 128) / 2
    if spoilt:
        k[int(cu[-1]) // 3, 0, 5] = float("inf")
        q[int(cu[-1]) // 2, hq - 1, 7] = float("nan")
    blocks = [(n + 63) // 64 for n in lens]
    part = [min(n, n - 64 * max(nb - tail, 0)) for n, nb in zip(lens, blocks)]   # the last `tail` blocks of each sequence as a chunk
    cu_q = np.concatenate([[0], np.cumsum(part)]).astype(np.int32)
    tail_q = torch.cat([q[int(cu[b + 1]) - part[b]:int(cu[b + 1])] for b in range(len(lens))])
    for chunk in (False, True):
        if not chunk and max(blocks) > 9000:
            continue
        p = Prefill(cu, hq, hkv, want_lse=False, cu_seqlens_q=cu_q if chunk else None)
        p.q, p.k, p.wq, p.wk = tail_q if chunk else q, k, wq, wk
        p.gate()
        stats = 8 * p.rows * (max(blocks) // 256 + 2)
        for params in (B.make_mask_params(B.SEER_TOPK_RATIO, keep_num=1, keep_den=10, flags=3), B.make_mask_params(B.SEER_TOPK_COUNT, k=33, flags=1, dense_tail=2)):
            p.mask(params)
            assert p.status() == 0
            rp, n = p.row_ptr.clone(), int(p.nnz.item())
            col = p.col_idx[:n].clone()
            for band in (128 << 20, (64 * max(blocks) + 4) * 4 + stats + 256, 0):
                if band == 0 and max(blocks) > 2500:
                    continue                               # (a band per 64 rows and head)
                p.row_ptr.fill_(-7)
                p.col_idx.fill_(-7)
                p.gate_mask(params, band_bytes=band)
                assert p.status() == 0
                assert torch.equal(p.row_ptr, rp) and torch.equal(p.col_idx[:n], col) and int(p.nnz.item()) == n, (chunk, band)


# rows of several warps whose statistics are finite (from 2049 blocks four warps a row, from 8193 eight), the last block of a row a candidate like the others
@pytest.mark.parametrize("flags", [0, 2])
@pytest.mark.parametrize("n,tail", [(2049 * 64, 2049), (2563 * 64 - 9, 700), (8193 * 64, 130), (10241 * 64 - 1, 40)])
def test_rows_without_a_forced_diagonal(n, tail, flags):
    import torch
    from paper_2410_13276_b200 import binding as B
    from paper_2410_13276_b200.prefill import Prefill
    gen = torch.Generator(device="cuda").manual_seed(n + flags)
    rand = lambda *s: torch.randn(*s, generator=gen, device="cuda")
    nq = n - 64 * ((n + 63) // 64 - tail)
    p = Prefill([0, n], 2, 1, want_lse=False, cu_seqlens_q=[0, nq])
    p.q, p.k, p.wq, p.wk = (2.0 * rand(nq, 2, 128)).bfloat16(), rand(n, 1, 128).bfloat16(), rand(2, 128, 128) / 2, rand(1, 128, 128) / 2
    p.gate()
    for params in (B.make_mask_params(B.SEER_TOPK_RATIO, keep_num=1, keep_den=10, flags=flags), B.make_mask_params(B.SEER_TOPK_COUNT, k=33, flags=flags),
                   B.make_mask_params(B.SEER_TOPK_COUNT, k=n // 64 - tail // 2, flags=flags)):
        p.mask(params)
        assert p.status() == 0
        rp, nnz = p.row_ptr.clone(), int(p.nnz.item())
        col = p.col_idx[:nnz].clone()
        p.row_ptr.fill_(-7)
        p.col_idx.fill_(-7)
        p.gate_mask(params)
        assert p.status() == 0
        assert torch.equal(p.row_ptr, rp) and torch.equal(p.col_idx[:nnz], col) and int(p.nnz.item()) == nnz
