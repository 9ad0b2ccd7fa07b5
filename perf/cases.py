"""The workloads whose speed matters: block-sparse prefill of one attention layer, through the package's public calls.

Every case is one layer of a prompt: gate scores -> block lists -> block-sparse attention, with the options a serving or
training stack uses them with.  The kinds:

  prefill   Prefill.run: the three calls on device-resident tensors (whole prompts, one or many per batch)
  chunk     chunked prefill: the last tokens of each sequence against a longer KV cache, gate and mask in one call
  block128  gate blocks of 128 tokens: gate, mask, expansion to 64-token lists, attention
  variant   the gate with composed pooling and block-level RoPE, a dense tail for the question; the scores are kept
  lists     gate and mask in one call without the quadratic score matrix (the lists of a very long prompt)
  distill   full causal attention and its max-pooled map: what the gate is trained against
  host      the whole path from page-locked host buffers to a host buffer

Inputs are drawn on the GPU.  `structured` tensors carry what attention maps of long prompts show: a sink key, stripes of
key blocks that many queries look at, and a slowly varying latent that ties nearby tokens together, over noise; gate
matrices are tied per group so that the gate sees it.  The others are normal noise with rotary embedding.
"""
import math

import numpy as np
import torch

from paper_2410_13276_b200 import binding as B
from paper_2410_13276_b200.prefill import Prefill

D = 128
SCORE_FLOPS = 2 * D            # one pooled query against one pooled key
BLOCK_FLOPS = 4 * 64 * 64 * D  # one listed 64 x 64 block of the attention
MAX_COST = 14.0e12             # attention flops of the largest listed case (128k tokens, 32 heads, one block in ten)


def listed():
    return [
        # one short prompt on a slice of a layer (4 query heads, one KV head): launches and host work are what it costs
        dict(name="prompt_2k", kind="prefill", lens="2048", hq=4, hkv=1, mode="ratio", num=1, den=2, sink=False, structured=False),
        # a serving batch of short ragged prompts: many sequences, every block count odd, lists of a few blocks
        dict(name="short_batch", kind="prefill",
             lens="65,1500,384,901,77,640,1023,130,256,1187,511,733,64,99,1409,2000,301,850,1290,47,1111,575,960,420",
             hq=32, hkv=8, mode="ratio", num=1, den=4, sink=True, structured=True),
        # an ordinary long prompt, one threshold for all rows (the paper's setting), row lengths uneven
        dict(name="prompt_32k", kind="prefill", lens="32768", hq=32, hkv=8, mode="threshold", density=0.10, structured=True),
        # the benchmark layer: 128k tokens, a tenth of the blocks plus diagonal and sink
        dict(name="prompt_128k", kind="prefill", lens="131072", hq=32, hkv=8, mode="ratio", num=1, den=10, sink=True,
             structured=False),
        # packed prompts of very different ragged lengths, five query heads per KV head
        dict(name="varlen_120k", kind="prefill", lens="8191,16400,32737,65536", hq=40, hkv=8, mode="threshold", density=0.15,
             structured=True),
        # one prefill step of a long prompt fed in pieces: 8k new tokens against a 128k cache
        dict(name="chunk_8k", kind="chunk", lens="131072", qlens="8192", hq=32, hkv=8, mode="ratio", num=1, den=10, sink=True,
             structured=True),
        # the latency end of chunked prefill: a batch whose members each bring a few hundred tokens
        dict(name="chunk_small", kind="chunk", lens="16384,5003,29130,9216", qlens="512,139,10,256", hq=32, hkv=8, mode="ratio",
             num=1, den=8, sink=True, structured=True),
        # coarse gate blocks
        dict(name="block128_64k", kind="block128", lens="65536", hq=32, hkv=8, mode="ratio", num=1, den=10, sink=True,
             structured=True),
        # the gate's best reported form (average on Q; average, max and min on K; block RoPE), the question kept dense
        dict(name="variant_48k", kind="variant", lens="48999", hq=32, hkv=8, mode="ratio", num=1, den=10, sink=True, tail=4,
             structured=True),
        # lists of a prompt whose score matrix (8.6 GB) is not materialised
        dict(name="lists_256k", kind="lists", lens="262144", hq=32, hkv=8, mode="ratio", num=1, den=20, sink=True,
             structured=True),
        # one training-side pass: dense causal attention and its max-pooled map
        dict(name="distill_16k", kind="distill", lens="16384", hq=32, hkv=8, mode="all", structured=True),
        # inputs and result in host memory
        dict(name="host_32k", kind="host", lens="32768", hq=32, hkv=8, mode="ratio", num=1, den=10, sink=True, structured=True),
    ]


def _spread(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["prefill", "prefill", "prefill", "chunk", "block128", "variant", "lists", "distill", "host"])
    hq, hkv = rng.choice([(4, 1), (8, 2), (32, 8), (32, 8), (40, 8), (16, 16)])
    top = {"prefill": 131072, "chunk": 131072, "block128": 131072, "variant": 98304, "lists": 262144, "distill": 16384,
           "host": 49152}[kind]
    total = _spread(rng, 300, top)
    n = rng.choice([1, 1, 2, 3, 8, 24])
    cuts = sorted(rng.uniform(0, 1) for _ in range(n - 1))
    lens = [max(1, int(total * (b - a))) for a, b in zip([0.0] + cuts, cuts + [1.0])]
    case = dict(kind=kind, lens=",".join(map(str, lens)), hq=hq, hkv=hkv, structured=rng.random() < 0.7)
    if kind == "distill":
        case["mode"] = "all"
    elif kind == "prefill" and rng.random() < 0.4:
        case.update(mode="threshold", density=rng.choice([0.05, 0.08, 0.1, 0.15, 0.3]))
    else:
        case.update(mode="ratio", num=1, den=rng.choice([2, 4, 8, 10, 10, 20]), sink=rng.random() < 0.6)
    if kind == "chunk":
        block = 64
        case["qlens"] = ",".join(str(n_k - block * rng.randint(0, (n_k - 1) // block)) for n_k in lens)
    if kind == "variant":
        case["tail"] = rng.choice([0, 1, 4])
    return case if _kept(case) * BLOCK_FLOPS <= MAX_COST else draw(rng)


# ------------------------------------------------------------------------------------------------ shapes
def _ints(text):
    return [int(x) for x in text.split(",")]


def _block(case):
    return 128 if case["kind"] == "block128" else 64


def _rows(case):
    """Per sequence: (blocks, first query block, list length of every query row that exists)."""
    block = _block(case)
    lens = _ints(case["lens"])
    qlens = _ints(case["qlens"]) if "qlens" in case else lens
    out = []
    for n, nq in zip(lens, qlens):
        nb = (n + block - 1) // block
        first = (n - nq) // block
        size = np.arange(first + 1, nb + 1, dtype=np.int64)
        if case["mode"] == "ratio":
            keep = np.minimum(np.maximum(-(-size * case["num"] // case["den"]), 1), size)
            keep = np.maximum(keep, np.minimum(size, 1 + int(case["sink"])))
            tail = case.get("tail", 0)
            if tail:
                keep[-tail:] = size[-tail:]
        elif case["mode"] == "threshold":
            keep = size * case["density"]
        else:
            keep = size
        out.append((nb, first, keep))
    return out


def _kept(case):
    """64 x 64 blocks the attention visits, over all heads."""
    return case["hq"] * sum(float(k.sum()) for _, _, k in _rows(case)) * (_block(case) / 64) ** 2


def _cu(lens):
    return np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)


# ------------------------------------------------------------------------------------------------ inputs
def _normal(gen, *shape):
    return torch.randn(*shape, generator=gen, device="cuda", dtype=torch.float32)


def _rotate(x, lens):
    """Rotary embedding, positions local to each sequence (base 500000, half-split pairs)."""
    half = D // 2
    inv = 500000.0 ** (-torch.arange(half, device="cuda", dtype=torch.float64) * 2.0 / D)
    pos = torch.cat([torch.arange(n, device="cuda", dtype=torch.float64) for n in lens])
    for t0 in range(0, len(pos), 8192):
        ang = pos[t0:t0 + 8192, None] * inv[None, :]
        c, s = ang.cos().float()[:, None, :], ang.sin().float()[:, None, :]
        lo, hi = x[t0:t0 + 8192, :, :half].clone(), x[t0:t0 + 8192, :, half:].clone()
        x[t0:t0 + 8192, :, :half] = lo * c - hi * s
        x[t0:t0 + 8192, :, half:] = hi * c + lo * s


def _layer(case, seed):
    """q, k, v (bf16, whole sequences) and the gate matrices."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    lens, hq, hkv = _ints(case["lens"]), case["hq"], case["hkv"]
    group, total = hq // hkv, sum(lens)
    q, k, v = _normal(gen, total, hq, D), _normal(gen, total, hkv, D), _normal(gen, total, hkv, D)
    wk = _normal(gen, hkv, D, 128) / math.sqrt(128.0)
    wq = wk.repeat_interleave(group, 0).contiguous()
    if not case["structured"]:
        _rotate(q, lens)
        _rotate(k, lens)
        wq = _normal(gen, hq, D, 128) / math.sqrt(128.0)
    else:
        c = torch.nn.functional.normalize(_normal(gen, hkv, D), dim=-1)
        # strength of the stripes' direction and of the shared latent in the query heads: sharp, mixed and diffuse heads
        alpha = torch.tensor([8, 6, 5, 4, 3, 3, 2, 0], device="cuda", dtype=torch.float32)
        gamma = torch.tensor([0, .25, .5, .25, .5, .25, .5, 0], device="cuda", dtype=torch.float32)
        pick = torch.arange(hq, device="cuda") % 8
        t0 = 0
        for n in lens:
            nb = (n + 63) // 64
            knots = _normal(gen, n // 192 + 2, hkv, D)           # the latent turns over about three blocks
            pos = torch.arange(n, device="cuda", dtype=torch.float32) / 192.0
            i = pos.long()
            f = ((pos - i) * (math.pi / 2))[:, None, None]
            z = f.cos() * knots[i] + f.sin() * knots[i + 1]
            stripe = torch.rand(nb, hkv, generator=gen, device="cuda") < min(0.5, 16.0 / nb)
            stripe[0] = False
            on = stripe.repeat_interleave(64, 0)[:n].float()
            ks, qs = k[t0:t0 + n], q[t0:t0 + n]
            ks += z + 8.0 * on[:, :, None] * c
            ks[0] = 8.0 * math.sqrt(D) * torch.nn.functional.normalize(0.08 * c + _normal(gen, hkv, D) / math.sqrt(D), dim=-1)
            qs += alpha[pick][:, None] * c.repeat_interleave(group, 0) + gamma[pick][:, None] * z.repeat_interleave(group, 1)
            t0 += n
    return q.bfloat16(), k.bfloat16(), v.bfloat16(), wq, wk


def _threshold(case, q, k, wq, wk):
    """The one threshold that keeps the stated share of the causal blocks (diagonal included), from every third head."""
    block, group = _block(case), case["hq"] // case["hkv"]
    picked, t0 = [], 0
    for n in _ints(case["lens"]):
        nb = (n + block - 1) // block
        seg = torch.arange(n, device="cuda") // block
        cnt = torch.bincount(seg, minlength=nb).float()[:, None]
        tri = torch.ones(nb, nb, device="cuda", dtype=torch.bool).tril()
        for h in range(0, case["hq"], 3):
            pq = torch.zeros(nb, D, device="cuda").index_add_(0, seg, q[t0:t0 + n, h].float()) / cnt
            pk = torch.zeros(nb, D, device="cuda").index_add_(0, seg, k[t0:t0 + n, h // group].float()) / cnt
            s = (pq @ wq[h]) @ (pk @ wk[h // group]).T / math.sqrt(128.0)
            p = s.masked_fill(~tri, -math.inf).softmax(-1)
            p.diagonal().fill_(2.0)
            picked.append(p[tri])
        t0 += n
    x = torch.cat(picked)
    return float(x.kthvalue(max(1, int(round(x.numel() * (1.0 - case["density"]))))).values)


def prepare(case, seed):
    kind, lens, hq, hkv = case["kind"], _ints(case["lens"]), case["hq"], case["hkv"]
    q, k, v, wq, wk = _layer(case, seed)
    flags = B.SEER_FORCE_DIAG | (B.SEER_FORCE_SINK if case.get("sink") else 0)
    if case["mode"] == "ratio":
        params = B.make_mask_params(B.SEER_TOPK_RATIO, keep_num=case["num"], keep_den=case["den"], flags=flags,
                                    dense_tail=case.get("tail", 0))
    elif case["mode"] == "threshold":
        params = B.make_mask_params(B.SEER_THRESHOLD, threshold=_threshold(case, q, k, wq, wk), flags=flags)
    else:
        params = B.make_mask_params(B.SEER_TOPK_COUNT, k=1 << 20, flags=flags)
    if kind == "host":
        shape = B.make_shape(_cu(lens), hq, hkv)
        pinned = [t.cpu().pin_memory() for t in (q, k, v, wq, wk)]
        return dict(case=case, params=params, shape=shape, ctx=B.Context(0), inputs=pinned,
                    o=torch.empty(q.shape, dtype=torch.bfloat16).pin_memory(),
                    arena=torch.empty(B.seer_prefill_host_arena_bytes(shape), dtype=torch.uint8, device="cuda"))
    cu_q = None
    if kind == "chunk":
        qlens = _ints(case["qlens"])
        cu_q, ends = _cu(qlens), np.cumsum(lens)
        q = torch.cat([q[e - n:e] for e, n in zip(ends, qlens)]).contiguous()
    # top-k list lengths are known beforehand, so the lists get exactly the room they need
    cap = None if case["mode"] == "threshold" else case["hq"] * sum(int(kept.sum()) for _, _, kept in _rows(case))
    cls = _Lists if kind == "lists" else Prefill
    p = cls(_cu(lens), hq, hkv, block=_block(case), cu_seqlens_q=cu_q, col_capacity=cap)
    p.q, p.k, p.v, p.wq, p.wk = q, k, v, wq, wk
    p.scores.zero_()                                     # the entries above the diagonal are never written
    if kind == "block128":
        p.col_idx64.zero_()                              # sized for four entries per 128-token block, a diagonal block has three
    state = dict(case=case, params=params, p=p)
    if kind == "variant":
        gen = torch.Generator(device="cuda")
        gen.manual_seed(seed + 1)
        # the projections of max and min start small beside the average's
        wk3 = torch.cat([wk, 0.1 * _normal(gen, hkv, 2 * D, 128) / math.sqrt(128.0)], 1).contiguous()
        state.update(options=B.seer_gate_options(B.SEER_POOL_AVG, B.SEER_POOL_AVG | B.SEER_POOL_MAX | B.SEER_POOL_MIN, 500000.0),
                     wk3=wk3)
    return state


class _Lists(Prefill):
    """A Prefill that never holds the quadratic score matrix nor the attention's output."""

    def __init__(self, cu_seqlens, num_q_heads, num_kv_heads, *, block, cu_seqlens_q, col_capacity):
        self.device, self.ctx = torch.device("cuda", 0), B.Context(0)
        self.block, self.hq, self.hkv = block, num_q_heads, num_kv_heads
        self.shape = B.make_shape(cu_seqlens, num_q_heads, num_kv_heads, block=block)
        self.row_ptr = torch.zeros(B.seer_mask_rows(self.shape) + 1, dtype=torch.int32, device="cuda")
        self.col_idx = torch.empty(col_capacity, dtype=torch.int32, device="cuda")
        self.col_capacity = col_capacity
        self.nnz = torch.zeros(1, dtype=torch.int64, device="cuda")
        self.scores = self.nnz


# ------------------------------------------------------------------------------------------------ one pass
def run(state):
    kind, params = state["case"]["kind"], state["params"]
    if kind == "host":
        B.seer_prefill_host(state["ctx"], state["shape"], *state["inputs"], params, state["o"], None, state["arena"])
        torch.cuda.current_stream().synchronize()        # the result is read on the host
        return state["o"]
    p = state["p"]
    if kind == "lists":
        p.gate_mask(params)
        return p.row_ptr, p.col_idx
    if kind == "chunk":
        p.gate_mask(params)
        p.attn()
    elif kind == "variant":
        p.gate_ex(state["options"], p.wq, state["wk3"])
        p.mask(params)
        p.attn()
        return p.scores, p.row_ptr, p.col_idx, p.o, p.lse
    elif kind == "distill":
        p.mask(params)                                   # every causal block, whatever the scores
        p.attn()
        return p.o, p.lse, p.block_max()
    else:
        p.run(params)
    if state["case"]["mode"] == "threshold":             # (a score at the threshold may move every later list)
        return p.o, p.lse
    if kind == "block128":
        return p.row_ptr64, p.col_idx64, p.o, p.lse
    return p.row_ptr, p.col_idx, p.o, p.lse


def work(case):
    """Inputs read once, outputs written once; the products of the pooled vectors and of the listed blocks (a diagonal
    block is half masked)."""
    kind, hq, hkv, block = case["kind"], case["hq"], case["hkv"], _block(case)
    lens = _ints(case["lens"])
    total = sum(lens)
    total_q = sum(_ints(case["qlens"])) if "qlens" in case else total
    rows = _rows(case)
    qblocks = sum(len(kept) for _, _, kept in rows)
    pairs = hq * sum(float(np.arange(first + 1, nb + 1).sum()) for nb, first, _ in rows)
    kept = _kept(case)
    parts_k = 3 if kind == "variant" else 1
    flops, nbytes = 0.0, 0.0
    if kind != "distill":                                # gate
        nbytes += 2.0 * D * (total_q * hq + total * hkv) + 4.0 * D * 128 * (hq + hkv * parts_k)
        flops += D * (total_q * hq + total * hkv * parts_k) + 2.0 * D * 128 * (qblocks * hq + sum(nb for nb, _, _ in rows) * hkv * parts_k)
        flops += SCORE_FLOPS * pairs
    if kind == "lists":
        return {"bytes": nbytes + 4.0 * (kept + hq * qblocks), "flops": flops}
    nbytes += 2.0 * D * (total_q * hq + total * hkv) + 4.0 * total_q * hq      # v and o, lse
    if kind == "distill":
        nbytes += 2.0 * D * (total * hq + total * hkv) + 4.0 * kept
        flops += 2.0 * D * 64 * 64 * (kept - 0.5 * hq * qblocks)              # the map needs its own normalised product
    if kind == "variant":
        nbytes += 4.0 * pairs
    elif case["mode"] == "ratio" and kind != "host":
        nbytes += 4.0 * (kept + hq * qblocks)
    flops += BLOCK_FLOPS * (kept - 0.5 * hq * qblocks * (block // 64))
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    """bf16 results: the package's two attention kernels (other order of the sums, other references of the exponentials)
    differ by up to 3.0e-3 in the 2-norm.  Lists: no entry of 160 000 differed from those of scores computed in 64 bits,
    but blocks whose scores are closer than the rounding of the sums may change places."""
    return {"rel": 1.2e-2, "differ": 1e-3}
