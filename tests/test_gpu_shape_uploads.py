"""Shapes that a context has not seen are uploaded from a staging ring of two of the largest batches: calls of more shapes than the ring or the slots
hold, issued one behind the other on a stream that is still busy, give what each gives by itself."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batches", [[4096, 4095, 4094, 4093, 4092], [4096, 1, 3000, 7, 2000, 64, 4000, 1500, 2, 3900, 5, 4096], list(range(1, 40)), [2048, 2049] * 6])
def test_calls_of_many_shapes_in_flight(batches):
    import torch
    from paper_2410_13276_b200 import binding as B
    params = B.make_mask_params(B.SEER_TOPK_RATIO, keep_num=1, keep_den=3, flags=1)
    rng = np.random.default_rng(len(batches))
    busy = torch.randn(4096, 4096, device="cuda")
    ctx, alone = B.Context(0), B.Context(0)
    calls = []
    for n, batch in enumerate(batches):
        cu = np.concatenate([[0], np.cumsum(rng.integers(0, 400, batch))]).astype(np.int32)
        shape = B.make_shape(cu, 2, 1)
        rows = B.seer_mask_rows(shape)
        scores = torch.rand(max(B.seer_scores_elems(shape), 1), device="cuda")
        out = [(torch.full((rows + 1,), -7, dtype=torch.int32, device="cuda"), torch.full((max(B.seer_causal_blocks(shape), 1),), -7, dtype=torch.int32, device="cuda"))
               for _ in range(2)]
        B.seer_block_mask(alone, shape, scores, params, *out[0])
        assert B.seer_poll_device_status(alone) == 0      # (waits: one call in flight at a time)
        calls.append((shape, scores, out))
    torch.cuda.synchronize()
    for turn in range(2):
        for _ in range(10):
            busy = busy @ busy * 1e-3                     # a few ms of work that the uploads queue behind
        for shape, scores, out in calls:
            out[1][0].fill_(-7)
            B.seer_block_mask(ctx, shape, scores, params, *out[1])
        assert B.seer_poll_device_status(ctx) == 0
        for shape, scores, ((rp, col), (rp1, col1)) in calls:
            assert torch.equal(rp, rp1) and torch.equal(col, col1)
