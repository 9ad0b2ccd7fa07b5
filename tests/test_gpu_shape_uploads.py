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


def test_the_two_shapes_of_an_expansion_have_a_slot_each():
    """seer_expand_block_lists reads the offsets of the 128-token and of the 64-token blocks.  With every other slot in flight on a busy stream the
    second shape must not take the slot of the first."""
    import torch
    from paper_2410_13276_b200 import binding as B
    ctx = B.Context(0)
    params = B.make_mask_params(B.SEER_TOPK_COUNT, k=2, flags=1)
    cu = np.array([0, 700, 1000], np.int32)
    shape = B.make_shape(cu, 2, 1, block=128)
    rows, rows64 = B.seer_mask_rows(shape), 2 * (11 + 5)
    scores = torch.rand(B.seer_scores_elems(shape), device="cuda")
    lists = lambda n, m: (torch.full((n + 1,), -7, dtype=torch.int32, device="cuda"), torch.full((m,), -7, dtype=torch.int32, device="cuda"))
    rp, col = lists(rows, B.seer_causal_blocks(shape))
    B.seer_block_mask(ctx, shape, scores, params, rp, col)
    assert B.seer_poll_device_status(ctx) == 0
    ref, out = lists(rows64, 4 * col.numel()), lists(rows64, 4 * col.numel())
    alone = B.Context(0)
    B.seer_expand_block_lists(alone, shape, rp, col, *ref)
    assert B.seer_poll_device_status(alone) == 0
    busy, side = torch.randn(4096, 4096, device="cuda"), torch.cuda.Stream()
    others = []
    for n in range(7):                                    # eight slots in all
        s = B.make_shape([0, 640 + 64 * n], 1, 1)
        others.append((s, torch.rand(B.seer_scores_elems(s), device="cuda"), *lists(B.seer_mask_rows(s), B.seer_causal_blocks(s))))
    torch.cuda.synchronize()
    with torch.cuda.stream(side):
        for _ in range(30):
            busy = busy @ busy * 1e-3
        for s, x, r, c in others:
            B.seer_block_mask(ctx, s, x, params, r, c)
    B.seer_expand_block_lists(ctx, shape, rp, col, *out)
    torch.cuda.synchronize()
    assert B.seer_poll_device_status(ctx) == 0
    assert torch.equal(out[0], ref[0]) and torch.equal(out[1], ref[1])
