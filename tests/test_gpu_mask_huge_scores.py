"""TopK lists of caller's scores that mix both signs with values around 2^127, the largest and lowest floats and infinities, as
blocks are forced or forbidden by hand: the distance of such a row's keys takes all 32 bits.  Rows by one, four and eight warps
and by the general kernel, short rows of a batch with a long one; k around the number of the huge scores.  Lists as the oracle's;
what lies behind the capacity stays untouched."""
import numpy as np
import pytest

from oracle import seer_oracle as O

pytestmark = pytest.mark.gpu

HUGE = [float("inf"), 2.0 ** 127, 1.9 * 2.0 ** 127, 0.99 * 2.0 ** 127, float(np.finfo(np.float32).max)]
GUARD = 4096


@pytest.mark.parametrize("smallest", [-1.5, -5.0, -float("inf"), float(np.finfo(np.float32).min)])
@pytest.mark.parametrize("nb", [300, 2048, 2049, 8192, 8193, 16385])
def test_scores_of_both_signs_and_huge_ones(nb, smallest):
    import torch
    from paper_2410_13276_b200 import binding as B
    from paper_2410_13276_b200.prefill import Prefill
    lens = [nb * 64 - 3, 300 * 64]
    p = Prefill(np.concatenate([[0], np.cumsum(lens)]).astype(np.int32), 1, 1, want_lse=False, col_capacity=1)
    gen = torch.Generator(device="cuda").manual_seed(nb)
    rand = lambda *s: torch.rand(*s, generator=gen, device="cuda")
    mats, at = [], 0
    for n in (nb, 300):
        s = p.scores[at:at + n * n].view(n, n)
        at += n * n
        s.normal_(generator=gen)
        if np.isfinite(smallest):
            s.clamp_(min=max(smallest, -5.0))
        last = torch.arange(n, device="cuda")[:, None]
        causal = lambda m: torch.minimum((rand(n, m) * (last + 1)).long(), last)
        s.scatter_(1, causal(3), smallest)
        # four huge scores a row (fewer where two fall on one column), anywhere among the causal blocks
        s.scatter_(1, causal(4), torch.tensor(HUGE, device="cuda")[torch.randint(0, len(HUGE), (n, 4), generator=gen, device="cuda")])
        s[7::16] = torch.where(rand(*s[7::16].shape) < 0.5, HUGE[-1], -HUGE[-1])             # nothing but the ends of the range
        s[11::16] = torch.where(rand(*s[11::16].shape) < 0.2, HUGE[0], -HUGE[0])
        mats.append(s)
    rows = [(0, i) for i in sorted({0, 1, 7, 11, 127, 128, 231, 235, 511, 520, nb // 2, nb // 2 + 1} | {nb - 1 - d for d in range(18)}) if i < nb]
    rows += [(1, i) for i in (0, 5, 129, 231, 235, 290, 298, 299)]
    host = {(b, i): mats[b][i, :i + 1].cpu().numpy() for b, i in rows}
    for kw in [dict(mode=O.MODE_TOPK_COUNT, k=k, flags=f) for k, f in ((1, 0), (2, 0), (3, 0), (4, 0), (5, 0), (4, 3), (6, 3), (40, 0))] + \
              [dict(mode=O.MODE_TOPK_RATIO, keep_num=9, keep_den=10, flags=0)]:
        cap = sum(O.keep_count(i + 1, kw["mode"], kw.get("keep_num", 1), kw.get("keep_den", 1), kw.get("k", 0)) for n in (nb, 300) for i in range(n))
        p.col_capacity, p.col_idx = cap, torch.full((cap + GUARD,), -9, dtype=torch.int32, device="cuda")
        p.mask(B.make_mask_params(kw["mode"], keep_num=kw.get("keep_num", 1), keep_den=kw.get("keep_den", 1), k=kw.get("k", 0), flags=kw["flags"]))
        assert p.status() == 0
        assert bool((p.col_idx[cap:] == -9).all()) and bool((p.col_idx[:cap] >= 0).all()) and int(p.nnz.item()) == cap
        rp = p.row_ptr.cpu().numpy()
        for b, i in rows:
            r = b * nb + i
            got = p.col_idx[int(rp[r]):int(rp[r + 1])].cpu().tolist()
            assert got == O.select_row(host[b, i], i, **kw), (nb, b, i, kw)
