"""seer_prefill_host where its last slice is taken in parts of the query heads (more than 8 MB of q each): two heads of four, one
of three, three of six, and a slice that stays whole; bit for bit what the three calls return on device tensors."""
import numpy as np
import pytest

from paper_2410_13276_b200 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lens,hq,hkv", [([20000], 8, 2), ([33000, 700], 3, 1), ([11000, 65], 6, 1), ([20000], 2, 2)])
def test_last_slice_in_parts(lens, hq, hkv):
    import torch
    from paper_2410_13276_b200 import binding as B
    from paper_2410_13276_b200.prefill import Prefill
    w = W.make_small(seed=130, seqlens=lens, hq=hq, hkv=hkv)
    p = Prefill(w.cu_seqlens, hq, hkv)
    p.set_inputs(w.q, w.k, w.v, w.wq, w.wk)
    params = B.make_mask_params(B.SEER_TOPK_RATIO, keep_num=1, keep_den=10, flags=3)
    p.run(params)
    assert p.status() == 0
    pinned = [torch.from_numpy(x.view(np.int16)).pin_memory() for x in (w.q, w.k, w.v)] + [torch.from_numpy(x).pin_memory() for x in (w.wq, w.wk)]
    o = torch.full(p.o.shape, -1, dtype=torch.bfloat16).pin_memory()
    lse = torch.full(p.lse.shape, float("nan")).pin_memory()
    arena = torch.empty(B.seer_prefill_host_arena_bytes(p.shape), dtype=torch.uint8, device="cuda")
    for _ in range(2):
        B.seer_prefill_host(p.ctx, p.shape, *pinned, params, o, lse, arena)
        torch.cuda.synchronize()
        assert B.seer_poll_device_status(p.ctx) == 0
        assert torch.equal(o, p.o.cpu()) and torch.equal(lse, p.lse.cpu())
        o.fill_(-1.0)


def test_arena_without_the_statistics():
    import torch
    from paper_2410_13276_b200 import binding as B
    from paper_2410_13276_b200.prefill import Prefill
    nb = 640                                                     # long enough for scores by two launches where there is room
    w = W.make_small(seed=131, seqlens=[nb * 64 - 3], hq=2, hkv=2)
    p = Prefill(w.cu_seqlens, 2, 2)
    p.set_inputs(w.q, w.k, w.v, w.wq, w.wk)
    params = B.make_mask_params(B.SEER_TOPK_RATIO, keep_num=1, keep_den=10, flags=3)
    p.run(params)
    pinned = [torch.from_numpy(x.view(np.int16)).pin_memory() for x in (w.q, w.k, w.v)] + [torch.from_numpy(x).pin_memory() for x in (w.wq, w.wk)]
    full = B.seer_prefill_host_arena_bytes(p.shape)
    statistics = (8 * nb * ((nb + 255) // 256 + 1) + 255) // 256 * 256   # (maximum, sum) per row of one head and segment of 256 columns
    launched = []
    for size in (full, full - 256, full - statistics):
        o = torch.full(p.o.shape, -1, dtype=torch.bfloat16).pin_memory()
        n0 = B.seer_launch_count(p.ctx)
        B.seer_prefill_host(p.ctx, p.shape, *pinned, params, o, None, torch.empty(size, dtype=torch.uint8, device="cuda"))
        torch.cuda.synchronize()
        launched.append(B.seer_launch_count(p.ctx) - n0)
        assert B.seer_poll_device_status(p.ctx) == 0 and torch.equal(o, p.o.cpu())
    assert launched[1] == launched[2] == launched[0] - 2             # a launch less for either KV head
    with pytest.raises(B.SeerError) as e:
        B.seer_prefill_host(p.ctx, p.shape, *pinned, params, o, None, torch.empty(full - statistics - 1, dtype=torch.uint8, device="cuda"))
    assert e.value.status == 3
