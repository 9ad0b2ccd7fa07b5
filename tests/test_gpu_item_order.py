"""The attention visits the sequences of chunks, and of batches of three work items a stream and more, from the longest to the shortest, and others in
the batch's order: results of batches in any order of lengths, with empty sequences and sequences without queries among them, equal those of
each sequence by itself, bit for bit, on both sides of that line (888 items), and so do the block maxima."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lens,qlens", [([64, 1500, 1, 900, 0, 1500, 333], None), ([0, 0, 65, 700, 64, 700], None), ([700, 2000, 300, 2000, 128], [60, 80, 0, 16, 128]),
                                        ([5000] + [70] * 40, [8] + [6] * 40), ([64 * 40, 0, 64 * 100 - 9, 64 * 7], None), ([64 * 41, 0, 64 * 100 - 9, 64 * 7], None)])
def test_batch_equals_its_sequences(lens, qlens):
    import torch
    from paper_2410_13276_b200 import binding as B
    from paper_2410_13276_b200.prefill import Prefill
    gen = torch.Generator(device="cuda").manual_seed(len(lens))
    hq, hkv = 6, 3
    rand = lambda n, h: torch.randn(n, h, 128, generator=gen, device="cuda").bfloat16()
    k, v = rand(sum(lens), hkv), rand(sum(lens), hkv)
    ql = lens if qlens is None else qlens
    q = rand(sum(ql), hq)
    cu, cu_q = (np.concatenate([[0], np.cumsum(x)]).astype(np.int32) for x in (lens, ql))

    def attend(cu, cu_q, q, k, v):
        p = Prefill(cu, hq, hkv, cu_seqlens_q=cu_q if qlens is not None else None)
        p.q, p.k, p.v = q, k, v
        p.scores.uniform_(generator=torch.Generator(device="cuda").manual_seed(1))
        p.mask(B.make_mask_params(B.SEER_TOPK_COUNT, k=1 << 20, flags=3))
        p.attn()
        assert p.status() == 0
        return p.o, p.lse, (p.row_ptr.cpu(), p.block_max().clone(), p.status())

    o, lse, (rp, bmax, status) = attend(cu, cu_q, q, k, v)
    for b in range(len(lens)):
        if ql[b] == 0:
            continue
        s, e, qs, qe = cu[b], cu[b + 1], cu_q[b], cu_q[b + 1]
        o1, lse1, (rp1, bmax1, status1) = attend(np.array([0, e - s], np.int32), np.array([0, qe - qs], np.int32), q[qs:qe].contiguous(), k[s:e].contiguous(), v[s:e].contiguous())
        assert torch.equal(o1.view(torch.int16), o[qs:qe].view(torch.int16)) and torch.equal(lse1, lse[:, qs:qe])
        at = hq * int(sum((n + 63) // 64 for n in lens[:b]))
        assert status == status1 == 0
        assert torch.equal(bmax[int(rp[at]):int(rp[at + len(rp1) - 1])], bmax1[:int(rp1[-1])])
