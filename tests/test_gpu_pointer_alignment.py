"""Tensors that begin where their type allows but not on the width of the kernels' widest accesses, as slices of larger buffers
do: bit for bit what the calls return for tensors on their own."""
import numpy as np
import pytest

from oracle import seer_oracle as O
from paper_2410_13276_b200 import workloads as W

pytestmark = pytest.mark.gpu


def shifted(t, elements):
    """A copy of t that begins `elements` elements behind a 256-byte boundary."""
    import torch
    room = torch.empty(t.numel() + elements + 256, dtype=t.dtype, device=t.device)
    assert room.data_ptr() % 256 == 0
    out = room[elements:elements + t.numel()].view(t.shape)
    out.copy_(t)
    return out


@pytest.mark.parametrize("chunk", [False, True])
def test_attention_output_on_16_bytes(chunk):
    import torch
    from paper_2410_13276_b200 import binding as B
    from paper_2410_13276_b200.prefill import Prefill
    lens, starts = [64 * 9 - 5, 70, 64 * 5], [128, 64, 0]
    w = W.make_small(seed=210, seqlens=lens, hq=4, hkv=2)
    q, cu_q = w.q, None
    if chunk:
        part = [w.q[w.cu_seqlens[b] + s:w.cu_seqlens[b + 1]] for b, s in enumerate(starts)]
        q, cu_q = np.concatenate(part), np.concatenate([[0], np.cumsum([len(x) for x in part])]).astype(np.int32)
    p = Prefill(w.cu_seqlens, 4, 2, cu_seqlens_q=cu_q)
    p.set_inputs(q, w.k, w.v, w.wq, w.wk)
    r = np.random.default_rng(3)
    rows = [sorted(r.choice(i + 1, min(n, i + 1), replace=False).tolist()) for x in lens for h in range(4) for i, n in
            enumerate(r.integers(0, 6, (x + 63) // 64))]          # no, one, odd and even numbers of blocks
    p.set_lists(np.concatenate([[0], np.cumsum([len(x) for x in rows])]), np.array([j for x in rows for j in x]))
    p.o.fill_(-1.0)
    p.attn()
    want = p.o
    p.o = shifted(torch.full_like(want, -1.0), 8)                  # 16 bytes on
    assert p.o.data_ptr() % 32 == 16
    p.attn()
    assert p.status() == 0 and torch.equal(p.o, want)
    trace = torch.zeros(7 * 8192, dtype=torch.int64, device="cuda")   # the instrumented kernel
    B.seer_set_trace_buffer(p.ctx, trace)
    p.o.fill_(-1.0)
    p.attn()
    assert p.status() == 0 and torch.equal(p.o, want)


# 12 + 4 heads: pooled two blocks a CTA, and sixteen
@pytest.mark.parametrize("lens", [[300, 65], [300 * 64 - 5, 310 * 64 + 1]])
@pytest.mark.parametrize("elements", [1, 2])
def test_gate_matrices_on_4_and_8_bytes(lens, elements):
    import torch
    from paper_2410_13276_b200 import binding as B
    from paper_2410_13276_b200.prefill import Prefill
    w = W.make_small(seed=211, seqlens=lens, hq=12, hkv=4)
    p = Prefill(w.cu_seqlens, 12, 4, want_lse=False)
    p.set_inputs(w.q, w.k, w.v, w.wq, w.wk)
    wq3, wk3 = (torch.cat([x, 0.1 * x, -0.1 * x], 1).contiguous() for x in (p.wq, p.wk))
    options = B.seer_gate_options(B.SEER_POOL_AVG | B.SEER_POOL_MAX | B.SEER_POOL_MIN, B.SEER_POOL_AVG | B.SEER_POOL_MAX | B.SEER_POOL_MIN, 10000.0)
    got = {}
    for name, move in (("aligned", lambda t, k: t), ("both", lambda t, k: shifted(t, elements)), ("Wk", lambda t, k: shifted(t, elements * k))):
        p.scores.fill_(-1.0)                                       # (above the diagonal nothing is written)
        B.seer_gate_scores(p.ctx, p.shape, p.q, p.k, move(p.wq, 0), move(p.wk, 1), p.scores, p.ws)
        plain = p.scores.clone()
        p.gate_ex(options, move(wq3, 0), move(wk3, 1))
        got[name] = (plain, p.scores.clone())
        if lens[0] == 300:
            p.scores.fill_(-1.0)
            B.seer_gate_scores_static(p.shape, p.q, p.k, move(p.wq, 0), move(p.wk, 1), p.scores)
            got[name] += (p.scores.clone(),)
    assert p.status() == 0
    for name in ("both", "Wk"):
        assert all(torch.equal(a, b) for a, b in zip(got[name], got["aligned"]))


@pytest.mark.parametrize("lens", [[64 * 5], [300, 65, 64 * 7 - 1], [640 * 64]])
def test_scores_on_4_bytes(lens):
    import torch
    from paper_2410_13276_b200 import binding as B
    from paper_2410_13276_b200.prefill import Prefill
    w = W.make_small(seed=212, seqlens=lens, hq=2, hkv=1)
    p = Prefill(w.cu_seqlens, 2, 1, want_lse=False)
    p.set_inputs(w.q, w.k, w.v, w.wq, w.wk)
    params = B.make_mask_params(B.SEER_TOPK_RATIO, keep_num=1, keep_den=3, flags=3)
    got = []
    for elements in (0, 1, 2, 3):
        p.scores = shifted(torch.full_like(p.scores, -1.0), elements)
        p.row_ptr.fill_(-1)
        p.gate()
        p.mask(params)
        got.append((p.scores, p.row_ptr.clone(), p.col_idx[:int(p.nnz.item())].clone()))
    assert p.status() == 0
    assert all(torch.equal(a, b) for x in got[1:] for a, b in zip(x, got[0]))


@pytest.mark.parametrize("elements", [1, 4])
def test_bf16_tensors_off_16_bytes_are_refused(elements):
    import torch
    from paper_2410_13276_b200 import binding as B
    from paper_2410_13276_b200.prefill import Prefill
    w = W.make_small(seed=213, seqlens=[300, 65], hq=2, hkv=1)
    p = Prefill(w.cu_seqlens, 2, 1)
    p.set_inputs(w.q, w.k, w.v, w.wq, w.wk)
    params = B.make_mask_params(B.SEER_TOPK_RATIO, keep_num=1, keep_den=3, flags=3)
    options = B.seer_gate_options(B.SEER_POOL_AVG, B.SEER_POOL_AVG, 10000.0)
    p.run(params)
    want, good = p.o.clone(), {x: getattr(p, x) for x in "qkvo"}
    calls = [("qk", p.gate), ("qk", p.gate_project), ("qk", lambda: p.gate_ex(options, p.wq, p.wk)), ("qk", lambda: p.gate_mask(params)),
             ("qk", lambda: B.seer_gate_scores_static(p.shape, p.q, p.k, p.wq, p.wk, p.scores)), ("qkvo", p.attn), ("qk", p.block_max)]
    for impl in (1, 0):
        B.seer_set_attn_impl(p.ctx, impl)
        for names, call in calls:
            for x in names:
                launched = B.seer_launch_count(p.ctx)
                setattr(p, x, shifted(good[x], elements))
                with pytest.raises(B.SeerError) as e:
                    call()
                setattr(p, x, good[x])
                assert e.value.status == 7 and B.seer_launch_count(p.ctx) == launched
    p.o.fill_(-1.0)
    p.run(params)
    assert p.status() == 0 and torch.equal(p.o, want)
    # a pointer that nothing reads may be anything: queries of a chunk without any, inputs of an empty batch
    for lens, cu_q in (([300], np.array([0, 0], np.int32)), ([0], None)):
        e = Prefill(np.array([0, lens[0]], np.int32), 2, 1, ctx=p.ctx, cu_seqlens_q=cu_q)
        e.q, e.k, e.wq, e.wk = shifted(good["q"], elements), good["k"] if lens[0] else shifted(good["k"], elements), p.wq, p.wk
        e.row_ptr.fill_(-1)
        e.gate_mask(params)
        assert e.status() == 0 and not e.row_ptr.any()
