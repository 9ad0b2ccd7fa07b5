"""Kernels that start while their predecessor still runs: passes over changing inputs that share every intermediate buffer, enqueued
without a pause, return what passes return that are waited for kernel by kernel."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

PASSES, SETS = 60, 4
CASES = [
    # tokens per sequence, query tokens, heads, block, mask, one call for gate and mask
    ([500], None, (4, 1), 64, dict(mode=0, keep_num=1, keep_den=2, flags=1), False),      # every kernel fits on the GPU beside the next
    ([2048], None, (4, 1), 64, dict(mode=2, threshold=0.03, flags=3), False),
    ([700, 65, 3000, 1], None, (8, 2), 64, dict(mode=0, keep_num=1, keep_den=4, flags=3), False),
    ([9000], None, (32, 8), 64, dict(mode=0, keep_num=1, keep_den=4, flags=3), False),
    ([3000, 500], None, (4, 2), 128, dict(mode=1, k=5, flags=3), False),
    ([4099, 700], [2051, 60], (8, 4), 64, dict(mode=1, k=9, flags=3), True),
    ([45000], None, (1, 1), 64, dict(mode=0, keep_num=1, keep_den=20, flags=3), True),    # statistics first, several bands
]


@pytest.mark.parametrize("case", range(len(CASES)))
def test_passes_without_a_pause(case):
    import torch
    from paper_2410_13276_b200 import binding as B
    from paper_2410_13276_b200.prefill import Prefill
    lens, qlens, (hq, hkv), block, kw, fused = CASES[case]
    cu = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
    cu_q = None if qlens is None else np.concatenate([[0], np.cumsum(qlens)]).astype(np.int32)
    p = Prefill(cu, hq, hkv, block=block, cu_seqlens_q=cu_q)
    gen = torch.Generator(device="cuda").manual_seed(case)
    rand = lambda *s: torch.randn(*s, generator=gen, device="cuda")
    inputs = [[rand(p.Tq, hq, 128).bfloat16() * 2, rand(p.T, hkv, 128).bfloat16(), rand(p.T, hkv, 128).bfloat16(),
               rand(hq, 128, 128) / 11.3, rand(hkv, 128, 128) / 11.3] for _ in range(SETS)]
    params = B.make_mask_params(kw["mode"], keep_num=kw.get("keep_num", 1), keep_den=kw.get("keep_den", 1), k=kw.get("k", 0),
                                threshold=kw.get("threshold", 0.0), flags=kw["flags"])
    outs = [torch.full_like(p.o, -1.0) for _ in range(PASSES)]

    def step(i, pause=lambda: None):
        p.q, p.k, p.v, p.wq, p.wk = inputs[i % SETS]
        p.o = outs[i]
        if fused:
            p.gate_mask(params, band_bytes=2 << 20)
        else:
            p.gate(); pause()
            p.mask(params)
        pause()
        p.attn(); pause()

    want = []
    for i in range(SETS):
        step(i, torch.cuda.synchronize)
        want.append(outs[i].clone())
        assert not torch.equal(want[i], want[0]) or i == 0
    for i in range(PASSES):
        outs[i].fill_(-1.0)
    for i in range(PASSES):
        step(i)
    torch.cuda.synchronize()
    assert p.status() == 0
    assert all(torch.equal(outs[i], want[i % SETS]) for i in range(PASSES))
