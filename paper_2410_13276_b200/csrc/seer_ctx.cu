// Context, shape validation, per-batch metadata upload and the three ABI entry points.
#include <algorithm>
#include <cstring>

#include "seer_internal.cuh"

namespace seer {

static size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

// Byte offsets of the arrays inside a metadata slot: as long as the batch, so that a new shape's upload is.
struct SlotLayout {
  size_t place, score, cu, blk, qoff, qdelta, qblk, pair, bytes;
  explicit constexpr SlotLayout(int batch)
      : place(0), score(place + sizeof(int4) * batch), cu(score + sizeof(int64_t) * (batch + 1)), blk(cu + sizeof(int32_t) * (batch + 1)),
        qoff(blk + sizeof(int32_t) * (batch + 1)), qdelta(qoff + sizeof(int32_t) * batch), qblk(qdelta + sizeof(int32_t) * batch),
        pair(qblk + sizeof(int32_t) * (batch + 1)), bytes(pair + sizeof(int32_t) * (batch + 1)) {}
};
constexpr size_t kSlotBytes = (SlotLayout(kMaxBatch).bytes + 255) / 256 * 256;

// Uploads are staged one behind the other in a page-locked ring of two slots of the largest batch: page-locking is what creating a
// context is bound by (by the megabyte), and a batch of 64 needs 3 KB of it.
constexpr size_t kStageBytes = 2 * kSlotBytes;

// Room for `bytes` in the ring, for the upload of slot `slot`; waits for uploads still in flight that lie there.
static char* stage_room(seer_ctx* ctx, int slot, size_t bytes) {
  size_t at = ctx->stage_pos;
  if (at + bytes > kStageBytes) at = 0;
  for (int i = 0; i < kMetaSlots; ++i) {
    const MetaSlot& o = ctx->slots[i];
    if (i != slot && o.stage_lo < at + bytes && at < o.stage_hi && cudaEventSynchronize(o.ready) != cudaSuccess) return nullptr;
  }
  ctx->slots[slot].stage_lo = at;
  ctx->slots[slot].stage_hi = at + bytes;
  ctx->stage_pos = align_up(at + bytes, 256);
  return (char*)ctx->stage + at;
}

seer_status shape_totals(const seer_shape* s, ShapeTotals* t) {
  if (!s || !s->cu_seqlens_host || s->batch < 1) return SEER_ERR_INVALID_ARG;
  if (s->num_q_heads < 1 || s->num_kv_heads < 1) return SEER_ERR_INVALID_ARG;
  if (s->batch > kMaxBatch) return SEER_ERR_UNSUPPORTED;
  if (s->head_dim != kHeadDim || (s->block != kBlock && s->block != 2 * kBlock) || s->gate_dim != kGateDim)
    return SEER_ERR_UNSUPPORTED;
  if (s->num_q_heads % s->num_kv_heads != 0) return SEER_ERR_UNSUPPORTED;
  const int32_t* cu = s->cu_seqlens_host;
  if (cu[0] != 0) return SEER_ERR_INVALID_ARG;
  if (const int32_t* cq = s->cu_seqlens_q_host) {
    // the queries are the last positions of each sequence and start on a block boundary
    if (cq[0] != 0) return SEER_ERR_INVALID_ARG;
    for (int b = 0; b < s->batch; ++b) {
      if (cu[b + 1] < cu[b]) return SEER_ERR_INVALID_ARG;
      const int64_t sq = (int64_t)cq[b + 1] - cq[b], sk = (int64_t)cu[b + 1] - cu[b];
      if (sq < 0 || sq > sk) return SEER_ERR_INVALID_ARG;
      if (sq > 0 && (sk - sq) % s->block != 0) return SEER_ERR_UNSUPPORTED;
    }
  }
  int64_t blocks = 0, sq = 0, causal = 0;
  int32_t max_nb = 0;
  for (int b = 0; b < s->batch; ++b) {
    if (cu[b + 1] < cu[b]) return SEER_ERR_INVALID_ARG;
    int64_t nb = ((int64_t)cu[b + 1] - cu[b] + s->block - 1) / s->block;
    blocks += nb;
    sq += nb * nb;
    causal += nb * (nb + 1) / 2;
    if (nb > max_nb) max_nb = (int32_t)nb;
  }
  t->total_tokens = cu[s->batch];
  t->total_q_tokens = s->cu_seqlens_q_host ? s->cu_seqlens_q_host[s->batch] : cu[s->batch];
  t->total_blocks = blocks;
  t->rows = blocks * s->num_q_heads;
  t->score_elems = sq * s->num_q_heads;
  t->causal_blocks = causal * s->num_q_heads;
  t->max_nb = max_nb;
  // int32 row ids / CSR offsets and 32-bit grids
  if (t->rows >= (int64_t)1 << 31 || t->causal_blocks >= (int64_t)1 << 31) return SEER_ERR_UNSUPPORTED;
  if ((int64_t)t->total_tokens * s->num_q_heads * kHeadDim >= (int64_t)1 << 40) return SEER_ERR_UNSUPPORTED;
  return SEER_OK;
}

size_t gate_workspace_bytes(const ShapeTotals& t, const seer_shape* s) {
  // projected pooled Q [Hq, blocks] and K [Hkv, blocks], three bf16 planes (hi, mid, lo of the fp32 value) each
  size_t gq = align_up((size_t)s->num_q_heads * t.total_blocks * kGatePairBytes, 256);
  size_t gk = align_up((size_t)s->num_kv_heads * t.total_blocks * kGatePairBytes, 256);
  return gq + gk;
}

size_t gate_stats_bytes(const ShapeTotals& t, const seer_shape* s) {
  return align_up((size_t)s->num_q_heads * t.total_blocks * gate_stat_segs(t.max_nb) * sizeof(float2), 256);
}

seer_status prepare(seer_ctx* ctx, const seer_shape* shape, cudaStream_t stream, SeqMeta* m, int* slot_out, int keep) {
  if (!ctx) return SEER_ERR_INVALID_ARG;
  ShapeTotals t;
  seer_status st = shape_totals(shape, &t);
  if (st != SEER_OK) return st;
  if (cudaSetDevice(ctx->device) != cudaSuccess) return SEER_ERR_CUDA;

  const SlotLayout at(shape->batch);
  const int n = shape->batch + 1;
  std::vector<int32_t> key(shape->cu_seqlens_host, shape->cu_seqlens_host + n);
  key.push_back(shape->num_q_heads);
  key.push_back(shape->block);
  if (shape->cu_seqlens_q_host) key.insert(key.end(), shape->cu_seqlens_q_host, shape->cu_seqlens_q_host + n);
  int slot = -1;
  for (int i = 0; i < kMetaSlots; ++i)
    if (ctx->slots[i].key == key) { slot = i; break; }
  if (slot < 0) {
    // the least recently used slot whose last reader and last upload have finished; only if every slot is still
    // in flight (more than kMetaSlots shapes cycling faster than the GPU works through them) does the call wait
    // for the oldest one
    slot = -1;
    int oldest = keep == 0 ? 1 : 0;
    for (int i = 0; i < kMetaSlots; ++i) {
      if (i == keep) continue;
      if (ctx->slots[i].stamp < ctx->slots[oldest].stamp) oldest = i;
      if (cudaEventQuery(ctx->slots[i].last_use) == cudaSuccess && cudaEventQuery(ctx->slots[i].ready) == cudaSuccess &&
          (slot < 0 || ctx->slots[i].stamp < ctx->slots[slot].stamp))
        slot = i;
    }
    (void)cudaGetLastError();                        // cudaErrorNotReady from the queries is not an error
    if (slot < 0) {
      slot = oldest;
      if (cudaEventSynchronize(ctx->slots[slot].last_use) != cudaSuccess) return SEER_ERR_CUDA;
      if (cudaEventSynchronize(ctx->slots[slot].ready) != cudaSuccess) return SEER_ERR_CUDA;
    }
    MetaSlot& s = ctx->slots[slot];
    char* h = stage_room(ctx, slot, at.bytes);
    if (h == nullptr) return SEER_ERR_CUDA;
    int32_t* cu = (int32_t*)(h + at.cu);
    int32_t* blk = (int32_t*)(h + at.blk);
    int64_t* sc = (int64_t*)(h + at.score);
    int32_t* qo = (int32_t*)(h + at.qoff);
    int32_t* qd = (int32_t*)(h + at.qdelta);
    int32_t* qb = (int32_t*)(h + at.qblk);
    int4* place = (int4*)(h + at.place);
    int32_t* order = qb + 1;                           // (its places are read before they become block counts)
    int32_t* pairs = (int32_t*)(h + at.pair);
    blk[0] = 0; sc[0] = 0; qb[0] = 0; pairs[0] = 0;
    for (int b = 0; b < shape->batch; ++b) {
      cu[b] = shape->cu_seqlens_host[b];
      int32_t nb = (shape->cu_seqlens_host[b + 1] - shape->cu_seqlens_host[b] + shape->block - 1) / shape->block;
      blk[b + 1] = blk[b] + nb;
      sc[b + 1] = sc[b] + (int64_t)shape->num_q_heads * nb * nb;
      qo[b] = 0; qd[b] = 0;
      if (const int32_t* cq = shape->cu_seqlens_q_host) {
        const int32_t sq = cq[b + 1] - cq[b], sk = shape->cu_seqlens_host[b + 1] - shape->cu_seqlens_host[b];
        qo[b] = sq > 0 ? (sk - sq) / shape->block : nb;          // no queries: past the last block
        qd[b] = cq[b] - (shape->cu_seqlens_host[b] + (sk - sq));  // first query token <-> key token cu[b] + sk - sq
      }
      order[b] = b;
    }
    // The attention works from the longest sequence to the shortest, so that the longest lists are not begun last (917 tokens
    // against 60k in a batch of four, 512 items for 296 streams: 58 us in batch order, 49 so).  Whole prompts of fewer than three items
    // a stream stay in the batch's order: a sequence's lists are of every length then, and a stream's second item, which it draws when
    // it begins its first, goes to the streams that begin first, those of the longest lists (prompts of 815 and 1965 tokens, 8
    // heads, 352 items: 30 us, 34 longest first; 8 prompts of 90 to 6295, 16 heads, 2960 items: 165 and 157).
    if (shape->cu_seqlens_q_host || (int64_t)blk[shape->batch] * shape->num_q_heads >= 6 * (int64_t)ctx->num_sms)
      std::stable_sort(order, order + shape->batch, [blk](int32_t x, int32_t y) { return blk[x + 1] - blk[x] > blk[y + 1] - blk[y]; });
    cu[shape->batch] = shape->cu_seqlens_host[shape->batch];
    for (int p = 0; p < shape->batch; ++p) {
      const int b = order[p];
      place[p] = make_int4(cu[b], cu[b + 1] - cu[b], blk[b], qd[b]);
      qb[p + 1] = qb[p] + blk[b + 1] - blk[b] - qo[b];
      pairs[p + 1] = pairs[p] + (qo[b] < blk[b + 1] - blk[b] ? (blk[b + 1] - blk[b] + 1) / 2 - qo[b] / 2 : 0);
    }
    if (cudaMemcpyAsync(s.dev, h, at.bytes, cudaMemcpyHostToDevice, stream) != cudaSuccess) return SEER_ERR_CUDA;
    if (cudaEventRecord(s.ready, stream) != cudaSuccess) return SEER_ERR_CUDA;
    s.key = key;
  } else {
    // another stream may have uploaded it
    if (cudaStreamWaitEvent(stream, ctx->slots[slot].ready, 0) != cudaSuccess) return SEER_ERR_CUDA;
  }
  MetaSlot& s = ctx->slots[slot];
  s.stamp = ++ctx->clock;
  const char* d = (const char*)s.dev;
  m->cu_seqlens = (const int32_t*)(d + at.cu);
  m->blk_off = (const int32_t*)(d + at.blk);
  m->score_off = (const int64_t*)(d + at.score);
  m->batch = shape->batch;
  m->num_q_heads = shape->num_q_heads;
  m->num_kv_heads = shape->num_kv_heads;
  m->group = shape->num_q_heads / shape->num_kv_heads;
  m->total_tokens = (int32_t)t.total_tokens;
  m->total_blocks = (int32_t)t.total_blocks;
  m->max_nb = t.max_nb;
  m->rows = t.rows;
  m->score_elems = t.score_elems;
  m->softmax_scale = shape->softmax_scale > 0.f ? shape->softmax_scale : 0.08838834764831845f;  // 1/sqrt(128)
  m->block = shape->block;
  m->qoff = (const int32_t*)(d + at.qoff);
  m->qdelta = (const int32_t*)(d + at.qdelta);
  m->qblk_off = (const int32_t*)(d + at.qblk);
  m->place = (const int4*)(d + at.place);
  m->total_q_tokens = (int32_t)t.total_q_tokens;
  m->chunked = shape->cu_seqlens_q_host ? 1 : 0;
  double tiles = 0;
  int64_t q_blocks = 0, pair_blocks = 0;
  for (int b = 0; b < shape->batch; ++b) {
    const double nb = (shape->cu_seqlens_host[b + 1] - shape->cu_seqlens_host[b] + shape->block - 1) / shape->block;
    double before = 0;                                 // blocks before the chunk
    if (const int32_t* cq = shape->cu_seqlens_q_host)
      before = ((shape->cu_seqlens_host[b + 1] - shape->cu_seqlens_host[b]) - (cq[b + 1] - cq[b])) / shape->block;
    tiles += (nb * nb - before * before) / 2 / (128.0 * kScoreTile);
    const int32_t* cq = shape->cu_seqlens_q_host;
    if (!cq || cq[b + 1] > cq[b]) {                       // (a chunk starts on a block)
      q_blocks += (int64_t)(nb - before);
      if (nb > before) pair_blocks += ((int64_t)nb + 1) / 2 - (int64_t)before / 2;
    }
    if (shape->batch == 1) m->first_q_block = (int32_t)before;
  }
  if (shape->batch != 1) m->first_q_block = 0;
  m->q_rows = q_blocks * shape->num_q_heads;
  m->pair_off = (const int32_t*)(d + at.pair);
  m->pair_units = pair_blocks * shape->num_q_heads;
  m->score_tiles = (int64_t)(tiles * shape->num_q_heads);
  m->wait_limit_us = ctx->wait_limit_us;
  m->lose_v_copy = ctx->lose_v_copy;
  *slot_out = slot;
  return SEER_OK;
}

void finish_call(seer_ctx* ctx, int slot, cudaStream_t stream) {
  cudaEventRecord(ctx->slots[slot].last_use, stream);
}

static bool ws_ok(const void* ws, size_t have, size_t need) {
  if (need == 0) return true;
  return ws && ((uintptr_t)ws & 255) == 0 && have >= need;
}

bool on_16(const void* a, const void* b, const void* c, const void* d) {
  return (((uintptr_t)a | (uintptr_t)b | (uintptr_t)c | (uintptr_t)d) & 15) == 0;
}

// ---- bands of the one-call gate + mask
namespace {
constexpr size_t kBandSlackElems = 4;   // the band's base is rounded down to a multiple of four elements

size_t min_band_bytes(const ShapeTotals& t) { return ((size_t)kScoreTile * (size_t)t.max_nb + kBandSlackElems) * sizeof(float); }

// The bands of a scratch of `cap` elements, in CSR row order: fn(band, first row, last row + 1) until it returns false.
template <class Fn>
void walk_bands(const seer_shape* shape, int64_t cap, Fn&& fn) {
  const int32_t* cu = shape->cu_seqlens_host;
  const int Hq = shape->num_q_heads;
  auto blocks_of = [&](int b) { return ((int64_t)cu[b + 1] - cu[b] + shape->block - 1) / shape->block; };
  int64_t blk_off = 0, score_off = 0;                  // of sequence b
  for (int b = 0; b < shape->batch;) {
    const int64_t nb = blocks_of(b);
    if ((int64_t)Hq * nb * nb <= cap) {
      // whole sequences, as many as fit
      int b1 = b;
      int64_t blocks = 0, elems = 0;
      while (b1 < shape->batch) {
        const int64_t n1 = blocks_of(b1);
        if (elems + (int64_t)Hq * n1 * n1 > cap) break;
        elems += (int64_t)Hq * n1 * n1; blocks += n1;
        ++b1;
      }
      if (!fn({(int32_t)blk_off, (int32_t)(blk_off + blocks), 0, Hq, score_off, 0, 0}, Hq * blk_off, Hq * (blk_off + blocks))) return;
      blk_off += blocks; score_off += elems;
      b = b1;
      continue;
    }
    // query blocks of the sequence that have scores: all of them, or those of its chunk
    int64_t i_lo = 0;
    if (shape->cu_seqlens_q_host) {
      const int64_t sq = (int64_t)shape->cu_seqlens_q_host[b + 1] - shape->cu_seqlens_q_host[b], sk = (int64_t)cu[b + 1] - cu[b];
      i_lo = sq > 0 ? (sk - sq) / shape->block : nb;
    }
    const int64_t per_head = packed_rows((int)nb) - packed_rows((int)i_lo);
    if (per_head <= cap) {
      // whole heads of this sequence, packed: causal columns alone, no rows before the chunk
      const int hb = per_head > 0 ? (int)(cap / per_head < Hq ? cap / per_head : Hq) : Hq;
      for (int h0 = 0; h0 < Hq; h0 += hb) {
        const int h1 = h0 + hb < Hq ? h0 + hb : Hq;
        if (!fn({(int32_t)(blk_off + i_lo), (int32_t)(blk_off + nb), h0, h1 - h0, 0, per_head > 0 ? per_head : 1, (int32_t)i_lo},
                Hq * blk_off + (int64_t)h0 * nb, Hq * blk_off + (int64_t)h1 * nb)) return;
      }
    } else {
      // runs of 64-row tiles of one head
      const int64_t ntile = (nb + kScoreTile - 1) / kScoreTile, tb = cap / ((int64_t)kScoreTile * nb);   // tb >= 1: the workspace check above
      for (int h = 0; h < Hq; ++h)
        for (int64_t t0 = 0; t0 < ntile; t0 += tb) {
          const int64_t t1 = t0 + tb < ntile ? t0 + tb : ntile;
          const int64_t i0 = t0 * kScoreTile, i1 = t1 * kScoreTile < nb ? t1 * kScoreTile : nb;
          if (!fn({(int32_t)(blk_off + i0), (int32_t)(blk_off + i1), h, 1, score_off + ((int64_t)h * nb + i0) * nb, 0, 0},
                  Hq * blk_off + (int64_t)h * nb + i0, Hq * blk_off + (int64_t)h * nb + i1)) return;
        }
    }
    blk_off += nb; score_off += (int64_t)Hq * nb * nb;
    ++b;
  }
}

int64_t count_bands(const seer_shape* shape, int64_t cap, int64_t limit) {
  int64_t n = 0;
  walk_bands(shape, cap, [&](const ScoreBand&, int64_t row_lo, int64_t row_hi) { n += row_hi > row_lo ? 1 : 0; return n < limit; });
  return n;
}
}  // namespace

}  // namespace seer

using namespace seer;

extern "C" {

const char* seer_status_string(seer_status s) {
  switch (s) {
    case SEER_OK: return "ok";
    case SEER_ERR_INVALID_ARG: return "invalid argument";
    case SEER_ERR_UNSUPPORTED: return "unsupported shape";
    case SEER_ERR_WORKSPACE: return "workspace too small or misaligned";
    case SEER_ERR_CAPACITY: return "col_idx capacity exceeded";
    case SEER_ERR_INVALID_INDEX: return "block index out of range";
    case SEER_ERR_TIMEOUT: return "bounded device wait expired";
    case SEER_ERR_CUDA: return "CUDA call failed";
  }
  return "unknown status";
}

seer_status seer_create(seer_ctx** out, int device) {
  if (!out) return SEER_ERR_INVALID_ARG;
  *out = nullptr;
  int count = 0;
  if (cudaGetDeviceCount(&count) != cudaSuccess || device < 0 || device >= count) return SEER_ERR_CUDA;
  if (cudaSetDevice(device) != cudaSuccess) return SEER_ERR_CUDA;
  int major = 0, sms = 0;                            // (all of a device's properties take 2.5 ms)
  if (cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, device) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device) != cudaSuccess) return SEER_ERR_CUDA;
  if (major != 10) return SEER_ERR_CUDA;  // kernels are built for sm_100a only
  seer_ctx* ctx = new seer_ctx();
  ctx->device = device;
  ctx->num_sms = sms;
  bool ok = cudaMalloc(&ctx->d_status, sizeof(int)) == cudaSuccess &&
            cudaMemset(ctx->d_status, 0, sizeof(int)) == cudaSuccess && cudaMallocHost(&ctx->stage, kStageBytes) == cudaSuccess;
  for (int i = 0; ok && i < kMetaSlots; ++i) {
    MetaSlot& s = ctx->slots[i];
    ok = cudaMalloc(&s.dev, kSlotBytes) == cudaSuccess &&
         cudaEventCreateWithFlags(&s.ready, cudaEventDisableTiming) == cudaSuccess &&
         cudaEventCreateWithFlags(&s.last_use, cudaEventDisableTiming) == cudaSuccess;
  }
  if (ok) ok = cudaStreamCreateWithFlags(&ctx->h2d_stream, cudaStreamNonBlocking) == cudaSuccess &&
              cudaStreamCreateWithFlags(&ctx->d2h_stream, cudaStreamNonBlocking) == cudaSuccess &&
              cudaEventCreateWithFlags(&ctx->ev_start, cudaEventDisableTiming) == cudaSuccess;
  for (int i = 0; ok && i < 2; ++i)
    ok = cudaEventCreateWithFlags(&ctx->ev_h2d[i], cudaEventDisableTiming) == cudaSuccess &&
         cudaEventCreateWithFlags(&ctx->ev_comp[i], cudaEventDisableTiming) == cudaSuccess &&
         cudaEventCreateWithFlags(&ctx->ev_d2h[i], cudaEventDisableTiming) == cudaSuccess;
  if (ok) ok = init_gate(ctx) == SEER_OK && init_mask(ctx) == SEER_OK && init_attn_mma(ctx) == SEER_OK &&
              init_attn_tc(ctx) == SEER_OK;
  if (!ok) { seer_destroy(ctx); return SEER_ERR_CUDA; }
  *out = ctx;
  return SEER_OK;
}

void seer_destroy(seer_ctx* ctx) {
  if (!ctx) return;
  cudaSetDevice(ctx->device);
  cudaDeviceSynchronize();
  for (int i = 0; i < kMetaSlots; ++i) {
    MetaSlot& s = ctx->slots[i];
    if (s.dev) cudaFree(s.dev);
    if (s.ready) cudaEventDestroy(s.ready);
    if (s.last_use) cudaEventDestroy(s.last_use);
  }
  if (ctx->d_status) cudaFree(ctx->d_status);
  if (ctx->stage) cudaFreeHost(ctx->stage);
  if (ctx->h2d_stream) cudaStreamDestroy(ctx->h2d_stream);
  if (ctx->d2h_stream) cudaStreamDestroy(ctx->d2h_stream);
  if (ctx->ev_start) cudaEventDestroy(ctx->ev_start);
  for (int i = 0; i < 2; ++i) {
    if (ctx->ev_h2d[i]) cudaEventDestroy(ctx->ev_h2d[i]);
    if (ctx->ev_comp[i]) cudaEventDestroy(ctx->ev_comp[i]);
    if (ctx->ev_d2h[i]) cudaEventDestroy(ctx->ev_d2h[i]);
  }
  delete ctx;
}

size_t seer_workspace_bytes(const seer_shape* shape) {
  ShapeTotals t;
  if (shape_totals(shape, &t) != SEER_OK) return 0;
  return gate_workspace_bytes(t, shape);
}

size_t seer_scores_elems(const seer_shape* shape) {
  ShapeTotals t;
  if (shape_totals(shape, &t) != SEER_OK) return 0;
  return (size_t)t.score_elems;
}

int64_t seer_mask_rows(const seer_shape* shape) {
  ShapeTotals t;
  if (shape_totals(shape, &t) != SEER_OK) return -1;
  return t.rows;
}

int64_t seer_causal_blocks(const seer_shape* shape) {
  ShapeTotals t;
  if (shape_totals(shape, &t) != SEER_OK) return -1;
  return t.causal_blocks;
}

seer_status seer_gate_scores(seer_ctx* ctx, const seer_shape* shape, const void* q, const void* k, const float* Wq,
                             const float* Wk, float* scores, void* ws, size_t ws_bytes, void* stream_) {
  cudaStream_t stream = (cudaStream_t)stream_;
  if (!ctx || !shape) return SEER_ERR_INVALID_ARG;
  ShapeTotals t;
  seer_status st = shape_totals(shape, &t);
  if (st != SEER_OK) return st;
  if (t.total_blocks == 0 || t.total_q_tokens == 0) return SEER_OK;   // no score row to write
  if (!q || !k || !Wq || !Wk || !scores) return SEER_ERR_INVALID_ARG;
  if (!ws_ok(ws, ws_bytes, gate_workspace_bytes(t, shape))) return SEER_ERR_WORKSPACE;
  if (!on_16(q, k)) return SEER_ERR_CUDA;
  SeqMeta m; int slot;
  st = prepare(ctx, shape, stream, &m, &slot);
  if (st != SEER_OK) return st;
  int n = launch_gate(ctx, m, q, k, Wq, Wk, scores, ws, ws_bytes, stream);
  finish_call(ctx, slot, stream);
  if (n < 0) return SEER_ERR_CUDA;
  ctx->launches += n;
  return SEER_OK;
}

seer_status seer_gate_project(seer_ctx* ctx, const seer_shape* shape, const void* q, const void* k, const float* Wq,
                              const float* Wk, void* ws, size_t ws_bytes, void* stream_) {
  cudaStream_t stream = (cudaStream_t)stream_;
  if (!ctx || !shape) return SEER_ERR_INVALID_ARG;
  ShapeTotals t;
  seer_status st = shape_totals(shape, &t);
  if (st != SEER_OK) return st;
  if (t.total_blocks == 0 || t.total_q_tokens == 0) return SEER_OK;
  if (!q || !k || !Wq || !Wk) return SEER_ERR_INVALID_ARG;
  if (!ws_ok(ws, ws_bytes, gate_workspace_bytes(t, shape))) return SEER_ERR_WORKSPACE;
  if (!on_16(q, k)) return SEER_ERR_CUDA;
  SeqMeta m; int slot;
  st = prepare(ctx, shape, stream, &m, &slot);
  if (st != SEER_OK) return st;
  int n = launch_gate(ctx, m, q, k, Wq, Wk, nullptr, ws, ws_bytes, stream);   // no score buffer: pooling and projection only
  finish_call(ctx, slot, stream);
  if (n < 0) return SEER_ERR_CUDA;
  ctx->launches += n;
  return SEER_OK;
}

seer_status seer_gate_scores_ex(seer_ctx* ctx, const seer_shape* shape, const seer_gate_options* opt, const void* q,
                                const void* k, const float* Wq, const float* Wk, float* scores, void* ws, size_t ws_bytes,
                                void* stream_) {
  cudaStream_t stream = (cudaStream_t)stream_;
  if (!ctx || !shape || !opt) return SEER_ERR_INVALID_ARG;
  const uint32_t all = SEER_POOL_AVG | SEER_POOL_MAX | SEER_POOL_MIN;
  if (opt->pool_q == 0 || opt->pool_k == 0 || (opt->pool_q & ~all) || (opt->pool_k & ~all)) return SEER_ERR_INVALID_ARG;
  if (!(opt->rope_theta >= 0.f) || opt->rope_theta > 3.0e38f) return SEER_ERR_INVALID_ARG;   // also rejects NaN
  ShapeTotals t;
  seer_status st = shape_totals(shape, &t);
  if (st != SEER_OK) return st;
  if (t.total_blocks == 0 || t.total_q_tokens == 0) return SEER_OK;   // no score row to write
  if (!q || !k || !Wq || !Wk || !scores) return SEER_ERR_INVALID_ARG;
  if (!ws_ok(ws, ws_bytes, gate_workspace_bytes(t, shape))) return SEER_ERR_WORKSPACE;
  if (!on_16(q, k)) return SEER_ERR_CUDA;
  SeqMeta m; int slot;
  st = prepare(ctx, shape, stream, &m, &slot);
  if (st != SEER_OK) return st;
  int n = launch_gate_ex(ctx, m, *opt, q, k, Wq, Wk, scores, ws, ws_bytes, stream);
  finish_call(ctx, slot, stream);
  if (n < 0) return SEER_ERR_CUDA;
  ctx->launches += n;
  return SEER_OK;
}

seer_status seer_block_mask(seer_ctx* ctx, const seer_shape* shape, const float* scores, const seer_mask_params* p,
                            int32_t* row_ptr, int32_t* col_idx, int64_t col_capacity, int64_t* nnz_out, void* ws,
                            size_t ws_bytes, void* stream_) {
  (void)ws; (void)ws_bytes;
  cudaStream_t stream = (cudaStream_t)stream_;
  if (!ctx || !shape || !p) return SEER_ERR_INVALID_ARG;
  ShapeTotals t;
  seer_status st = shape_totals(shape, &t);
  if (st != SEER_OK) return st;
  if (!row_ptr || col_capacity < 0 || (col_capacity > 0 && !col_idx)) return SEER_ERR_INVALID_ARG;
  if (p->mode != SEER_TOPK_RATIO && p->mode != SEER_TOPK_COUNT && p->mode != SEER_THRESHOLD) return SEER_ERR_INVALID_ARG;
  if (p->mode == SEER_TOPK_RATIO && (p->keep_num < 0 || p->keep_den < 1)) return SEER_ERR_INVALID_ARG;
  if (p->flags & ~(uint32_t)(SEER_FORCE_DIAG | SEER_FORCE_SINK)) return SEER_ERR_INVALID_ARG;
  if (p->dense_tail_blocks < 0) return SEER_ERR_INVALID_ARG;
  if (t.total_blocks > 0 && !scores) return SEER_ERR_INVALID_ARG;
  SeqMeta m; int slot;
  st = prepare(ctx, shape, stream, &m, &slot);
  if (st != SEER_OK) return st;
  int n = launch_mask(ctx, m, scores, *p, row_ptr, col_idx, col_capacity, nnz_out, stream);
  finish_call(ctx, slot, stream);
  if (n < 0) return SEER_ERR_CUDA;
  ctx->launches += n;
  return SEER_OK;
}

seer_status seer_sparse_attn(seer_ctx* ctx, const seer_shape* shape, const void* q, const void* k, const void* v,
                             const int32_t* row_ptr, const int32_t* col_idx, void* o, float* lse, void* ws,
                             size_t ws_bytes, void* stream_) {
  cudaStream_t stream = (cudaStream_t)stream_;
  if (!ctx || !shape) return SEER_ERR_INVALID_ARG;
  ShapeTotals t;
  seer_status st = shape_totals(shape, &t);
  if (st != SEER_OK) return st;
  if (shape->block != kBlock) return SEER_ERR_UNSUPPORTED;   // 128-token lists go through seer_expand_block_lists first
  // the first word of the workspace is the counter the tcgen05 kernel's streams draw their work items from; without
  // a workspace the items are dealt statically
  int* work_counter = ws_ok(ws, ws_bytes, 256) ? (int*)ws : nullptr;
  if (t.total_blocks == 0 || t.total_q_tokens == 0) return SEER_OK;   // no output row
  if (!q || !k || !v || !row_ptr || !col_idx || !o) return SEER_ERR_INVALID_ARG;
  if (!on_16(q, k, v, o)) return SEER_ERR_CUDA;
  SeqMeta m; int slot;
  st = prepare(ctx, shape, stream, &m, &slot);
  if (st != SEER_OK) return st;
  // impl 2: by shape, where the lists (at most the causal blocks) are short.  Not for speed any more: on batches of 1 to 4000
  // sequences of 40 to 960 tokens the tcgen05 kernel takes 0.3 to 1.0 of the mma.sync kernel's time (64 sequences of 900 tokens, 32
  // heads, all blocks: 990 against 2572 us; 8 of 64 tokens: 13.3 against 13.4).
  const bool legacy = ctx->attn_impl == 1 || (ctx->attn_impl == 2 && t.causal_blocks <= 8 * t.rows);
  int n = legacy ? launch_attn_mma(ctx, m, q, k, v, row_ptr, col_idx, o, lse, stream)
                 : launch_attn_tc(ctx, m, q, k, v, row_ptr, col_idx, o, lse, work_counter, stream);
  finish_call(ctx, slot, stream);
  if (n < 0) return SEER_ERR_CUDA;
  ctx->launches += n;
  return SEER_OK;
}

seer_status seer_attn_block_max(seer_ctx* ctx, const seer_shape* shape, const void* q, const void* k,
                                const int32_t* row_ptr, const int32_t* col_idx, const float* lse, float* block_max,
                                void* stream_) {
  cudaStream_t stream = (cudaStream_t)stream_;
  if (!ctx || !shape) return SEER_ERR_INVALID_ARG;
  ShapeTotals t;
  seer_status st = shape_totals(shape, &t);
  if (st != SEER_OK) return st;
  if (shape->block != kBlock) return SEER_ERR_UNSUPPORTED;
  if (t.total_blocks == 0 || t.total_q_tokens == 0) return SEER_OK;
  if (!q || !k || !row_ptr || !col_idx || !lse || !block_max) return SEER_ERR_INVALID_ARG;
  if (!on_16(q, k)) return SEER_ERR_CUDA;
  SeqMeta m; int slot;
  st = prepare(ctx, shape, stream, &m, &slot);
  if (st != SEER_OK) return st;
  // the same choice of kernel as seer_sparse_attn: the tcgen05 pipeline without V, or the mma.sync kernel
  const bool legacy = ctx->attn_impl == 1 || (ctx->attn_impl == 2 && t.causal_blocks <= 8 * t.rows);
  int n = legacy ? launch_block_max(ctx, m, q, k, row_ptr, col_idx, lse, block_max, stream)
                 : launch_block_max_tc(ctx, m, q, k, row_ptr, col_idx, lse, block_max, stream);
  finish_call(ctx, slot, stream);
  if (n < 0) return SEER_ERR_CUDA;
  ctx->launches += n;
  return SEER_OK;
}

// ---- gate and mask in one call, the scores held one band at a time
size_t seer_gate_mask_workspace_bytes(const seer_shape* shape, size_t band_bytes) {
  ShapeTotals t;
  if (shape_totals(shape, &t) != SEER_OK) return 0;
  const size_t need = min_band_bytes(t);
  return gate_workspace_bytes(t, shape) + align_up(band_bytes > need ? band_bytes : need, 256);
}

seer_status seer_gate_block_mask(seer_ctx* ctx, const seer_shape* shape, const seer_gate_options* opt, const void* q,
                                 const void* k, const float* Wq, const float* Wk, const seer_mask_params* p,
                                 int32_t* row_ptr, int32_t* col_idx, int64_t col_capacity, int64_t* nnz_out, void* ws,
                                 size_t ws_bytes, void* stream_) {
  cudaStream_t stream = (cudaStream_t)stream_;
  if (!ctx || !shape || !p) return SEER_ERR_INVALID_ARG;
  if (opt) {
    const uint32_t all = SEER_POOL_AVG | SEER_POOL_MAX | SEER_POOL_MIN;
    if (opt->pool_q == 0 || opt->pool_k == 0 || (opt->pool_q & ~all) || (opt->pool_k & ~all)) return SEER_ERR_INVALID_ARG;
    if (!(opt->rope_theta >= 0.f) || opt->rope_theta > 3.0e38f) return SEER_ERR_INVALID_ARG;
  }
  ShapeTotals t;
  seer_status st = shape_totals(shape, &t);
  if (st != SEER_OK) return st;
  if (!row_ptr || col_capacity < 0 || (col_capacity > 0 && !col_idx)) return SEER_ERR_INVALID_ARG;
  if (p->mode != SEER_TOPK_RATIO && p->mode != SEER_TOPK_COUNT && p->mode != SEER_THRESHOLD) return SEER_ERR_INVALID_ARG;
  if (p->mode == SEER_TOPK_RATIO && (p->keep_num < 0 || p->keep_den < 1)) return SEER_ERR_INVALID_ARG;
  if (p->flags & ~(uint32_t)(SEER_FORCE_DIAG | SEER_FORCE_SINK)) return SEER_ERR_INVALID_ARG;
  if (p->dense_tail_blocks < 0) return SEER_ERR_INVALID_ARG;
  if (t.total_blocks > 0 && ((!q && t.total_q_tokens > 0) || !k || !Wq || !Wk)) return SEER_ERR_INVALID_ARG;
  const size_t planes_bytes = gate_workspace_bytes(t, shape), stats_bytes = gate_stats_bytes(t, shape);
  if (t.total_blocks > 0 && !ws_ok(ws, ws_bytes, planes_bytes + min_band_bytes(t))) return SEER_ERR_WORKSPACE;
  if (t.total_blocks > 0 && !on_16(t.total_q_tokens > 0 ? q : nullptr, k)) return SEER_ERR_CUDA;
  SeqMeta m; int slot;
  st = prepare(ctx, shape, stream, &m, &slot);
  if (st != SEER_OK) return st;
  if (t.total_blocks == 0) {
    int n0 = launch_mask(ctx, m, nullptr, *p, row_ptr, col_idx, col_capacity, nnz_out, stream);
    finish_call(ctx, slot, stream);
    return n0 < 0 ? SEER_ERR_CUDA : SEER_OK;
  }
  // Several bands, or a problem of few long rows: the statistics of all rows by one launch that fills the GPU, if what follows the
  // projected vectors has room for them (1 / 28 of the scores of a 2048-block sequence, 1 / 51 at 4096) and for the smallest band.  For
  // short sequences they are as large as the scores: statistics that would make several bands of one, or more than twice as many, are not
  // worth their room.  (700 tokens, 32 heads, a scratch of exactly the scores: 18 us in one band, 133 in eleven.)
  const auto band_elems = [&](size_t at) { return (int64_t)((ws_bytes - at) / sizeof(float)) - (int64_t)kBandSlackElems; };
  const bool room = ws_bytes >= planes_bytes + stats_bytes + min_band_bytes(t);
  bool with_stats = false, logits = false;
  if (room) {
    const int64_t plain = band_elems(planes_bytes), rest = band_elems(planes_bytes + stats_bytes);
    const bool split = gate_split(m, ctx->num_sms);
    int64_t bands = 1, limit = 1;
    if (t.score_elems > rest) {
      const int64_t without = count_bands(shape, plain, INT64_MAX);
      limit = without > 1 ? 2 * without : 1;
      bands = count_bands(shape, rest, limit + 1);
      if (split && bands > limit) bands = count_bands(shape, rest, INT64_MAX);
    }
    with_stats = split || (t.score_elems > plain && bands <= limit);
    // Where the selection can form the scores itself the bands hold logits: every logit is computed once, its row's statistics beside it.
    logits = mask_takes_logits(m, *p) && (bands == 1 || (with_stats && gate_logits_pay(m, bands, ctx->num_sms)));
    with_stats = with_stats || logits;
  }
  const size_t gate_bytes = planes_bytes + (with_stats ? stats_bytes : 0);
  float* band_buf = (float*)((char*)ws + gate_bytes);
  const int64_t cap = band_elems(gate_bytes);          // elements per band
  int64_t launched = 0;
  bool bad = false, first = true;
  {
    int n = opt ? launch_gate_ex(ctx, m, *opt, q, k, Wq, Wk, nullptr, ws, ws_bytes, stream)
                : launch_gate(ctx, m, q, k, Wq, Wk, nullptr, ws, ws_bytes, stream);
    if (n < 0) bad = true; else launched += n;
    if (!bad && with_stats && !logits) {
      n = launch_gate_stats_all(ctx, m, ws, stream);
      if (n < 0) bad = true; else launched += n;
    }
  }
  // One band after the other, in CSR row order: scores of the band -> counts -> row_ptr (continued) -> lists.
  auto run_band = [&](ScoreBand band, int64_t row_lo, int64_t row_hi) {
    if (bad || row_hi <= row_lo) return;
    band.score_base &= ~(int64_t)3;
    int n = band.blk_hi <= band.blk_lo ? 0
            : logits ? launch_gate_logits_band(ctx, m, band, ws, band_buf, stream) : launch_gate_scores_band(ctx, m, band, ws, band_buf, with_stats, stream);
    if (n >= 0) {
      launched += n;
      n = launch_mask_band(ctx, m, band_buf, with_stats ? gate_stats(m, ws) : nullptr, logits, band, row_lo, row_hi, first, *p, row_ptr, col_idx, col_capacity, nnz_out, stream);
    }
    if (n < 0) { bad = true; return; }
    launched += n;
    first = false;
  };
  walk_bands(shape, cap, [&](const ScoreBand& band, int64_t row_lo, int64_t row_hi) { run_band(band, row_lo, row_hi); return !bad; });
  finish_call(ctx, slot, stream);
  if (bad) return SEER_ERR_CUDA;
  ctx->launches += launched;
  return SEER_OK;
}

seer_status seer_expand_block_lists(seer_ctx* ctx, const seer_shape* shape, const int32_t* row_ptr, const int32_t* col_idx,
                                    int32_t* row_ptr64, int32_t* col_idx64, int64_t col_capacity64, int64_t* nnz_out,
                                    void* stream_) {
  cudaStream_t stream = (cudaStream_t)stream_;
  if (!ctx || !shape) return SEER_ERR_INVALID_ARG;
  if (shape->block != 2 * kBlock) return SEER_ERR_UNSUPPORTED;
  seer_shape fine = *shape;
  fine.block = kBlock;
  ShapeTotals t128, t64;
  seer_status st = shape_totals(shape, &t128);
  if (st == SEER_OK) st = shape_totals(&fine, &t64);
  if (st != SEER_OK) return st;
  if (!row_ptr64 || col_capacity64 < 0 || (col_capacity64 > 0 && !col_idx64)) return SEER_ERR_INVALID_ARG;
  if (t128.total_blocks > 0 && !row_ptr) return SEER_ERR_INVALID_ARG;
  SeqMeta m128, m64; int slot128, slot64;
  st = prepare(ctx, shape, stream, &m128, &slot128);
  if (st != SEER_OK) return st;
  st = prepare(ctx, &fine, stream, &m64, &slot64, slot128);
  if (st != SEER_OK) { finish_call(ctx, slot128, stream); return st; }
  int n = launch_expand_lists(ctx, m128, m64, row_ptr, col_idx, row_ptr64, col_idx64, col_capacity64, nnz_out, stream);
  finish_call(ctx, slot128, stream);
  finish_call(ctx, slot64, stream);
  if (n < 0) return SEER_ERR_CUDA;
  ctx->launches += n;
  return SEER_OK;
}

seer_status seer_debug_lost_wait(seer_ctx* ctx, uint32_t wait_limit_us, int32_t lose_v_copy_of_tile) {
  if (!ctx || wait_limit_us == 0u) return SEER_ERR_INVALID_ARG;
  ctx->wait_limit_us = wait_limit_us;
  ctx->lose_v_copy = lose_v_copy_of_tile;
  return SEER_OK;
}

seer_status seer_set_attn_impl(seer_ctx* ctx, int impl) {
  if (!ctx || impl < 0 || impl > 2) return SEER_ERR_INVALID_ARG;
  ctx->attn_impl = impl;
  return SEER_OK;
}

seer_status seer_poll_device_status(seer_ctx* ctx, void* stream_) {
  if (!ctx) return SEER_ERR_INVALID_ARG;
  cudaStream_t stream = (cudaStream_t)stream_;
  if (cudaSetDevice(ctx->device) != cudaSuccess) return SEER_ERR_CUDA;
  int h = 0;
  if (cudaMemcpyAsync(&h, ctx->d_status, sizeof(int), cudaMemcpyDeviceToHost, stream) != cudaSuccess) return SEER_ERR_CUDA;
  if (cudaStreamSynchronize(stream) != cudaSuccess) return SEER_ERR_CUDA;
  if (h != 0) {
    if (cudaMemsetAsync(ctx->d_status, 0, sizeof(int), stream) != cudaSuccess) return SEER_ERR_CUDA;
    if (cudaStreamSynchronize(stream) != cudaSuccess) return SEER_ERR_CUDA;
  }
  return (seer_status)h;
}

int64_t seer_launch_count(const seer_ctx* ctx) { return ctx ? ctx->launches : -1; }

seer_status seer_set_trace_buffer(seer_ctx* ctx, void* device_buffer) {
  if (!ctx) return SEER_ERR_INVALID_ARG;
  ctx->trace = device_buffer;
  return SEER_OK;
}

namespace {
// seer_prefill_host works on one KV head (and the query heads of its group) at a time: a slice is a problem of its own
// with num_q_heads = G, num_kv_heads = 1.  The arena holds two sets of slice inputs and outputs (copy of slice s + 1 and
// read-back of slice s - 1 overlap the kernels of slice s) and one set of intermediates.
struct ArenaLayout {
  size_t q[2], k[2], v[2], o[2], lse[2], wq[2], wk[2], scores, row_ptr, col_idx, nnz, ws, need, total;
};
ArenaLayout arena_layout(const seer_shape* slice, const ShapeTotals& t) {   // shape and totals of ONE slice
  ArenaLayout a;
  size_t p = 0;
  auto take = [&](size_t bytes) { size_t at = p; p = align_up(p + bytes, 256); return at; };
  const size_t T = (size_t)t.total_tokens;
  for (int b = 0; b < 2; ++b) {
    a.q[b] = take(T * slice->num_q_heads * kHeadDim * 2);
    a.k[b] = take(T * kHeadDim * 2);
    a.v[b] = take(T * kHeadDim * 2);
    a.o[b] = take(T * slice->num_q_heads * kHeadDim * 2);
    a.lse[b] = take(T * slice->num_q_heads * 4);
    a.wq[b] = take((size_t)slice->num_q_heads * kHeadDim * kGateDim * 4);
    a.wk[b] = take((size_t)kHeadDim * kGateDim * 4);
  }
  a.scores = take((size_t)t.score_elems * 4);
  a.row_ptr = take(((size_t)t.rows + 1) * 4);
  a.col_idx = take((size_t)t.causal_blocks * 4);
  a.nnz = take(8);
  a.ws = take(gate_workspace_bytes(t, slice));
  a.need = p;
  take(gate_stats_bytes(t, slice));                        // behind the projected vectors: used where there is room
  a.total = p;
  return a;
}
}  // namespace

static bool slice_of(const seer_shape* shape, seer_shape* slice, ShapeTotals* t) {
  *slice = *shape;
  if (shape->num_kv_heads <= 0 || shape->num_q_heads % shape->num_kv_heads != 0) return false;
  slice->num_q_heads = shape->num_q_heads / shape->num_kv_heads;
  slice->num_kv_heads = 1;
  return shape_totals(slice, t) == SEER_OK;
}

size_t seer_prefill_host_arena_bytes(const seer_shape* shape) {
  ShapeTotals full, t;
  seer_shape slice;
  if (!shape || shape_totals(shape, &full) != SEER_OK || !slice_of(shape, &slice, &t)) return 0;
  return arena_layout(&slice, t).total;
}

seer_status seer_prefill_host(seer_ctx* ctx, const seer_shape* shape, const void* q_host, const void* k_host,
                              const void* v_host, const float* Wq_host, const float* Wk_host,
                              const seer_mask_params* params, void* o_host, float* lse_host, void* arena,
                              size_t arena_bytes, void* stream_) {
  cudaStream_t stream = (cudaStream_t)stream_;
  if (!ctx || !shape || !params) return SEER_ERR_INVALID_ARG;
  ShapeTotals full, t;
  seer_status st = shape_totals(shape, &full);
  if (st != SEER_OK) return st;
  if (shape->block != kBlock || shape->cu_seqlens_q_host) return SEER_ERR_UNSUPPORTED;
  if (full.total_blocks == 0) return SEER_OK;
  if (!q_host || !k_host || !v_host || !Wq_host || !Wk_host || !o_host) return SEER_ERR_INVALID_ARG;
  seer_shape slice;
  if (!slice_of(shape, &slice, &t)) return SEER_ERR_INVALID_ARG;
  const ArenaLayout a = arena_layout(&slice, t);
  if (!ws_ok(arena, arena_bytes, a.need)) return SEER_ERR_WORKSPACE;
  const size_t ws_bytes = (arena_bytes < a.total ? arena_bytes : a.total) - a.ws;
  if (cudaSetDevice(ctx->device) != cudaSuccess) return SEER_ERR_CUDA;
  char* d = (char*)arena;
  const size_t T = (size_t)t.total_tokens;
  const int Hq = shape->num_q_heads, Hkv = shape->num_kv_heads, G = slice.num_q_heads;
  const size_t head_bytes = (size_t)kHeadDim * 2;                       // one head of one token
  const size_t wq_bytes = (size_t)G * kHeadDim * kGateDim * 4, wk_bytes = (size_t)kHeadDim * kGateDim * 4;
  cudaStream_t h2d = ctx->h2d_stream, d2h = ctx->d2h_stream;
#define SEER_TRY(call) do { if ((call) != cudaSuccess) return SEER_ERR_CUDA; } while (0)
  // the copy streams start after whatever precedes this call on the caller's stream
  SEER_TRY(cudaEventRecord(ctx->ev_start, stream));
  SEER_TRY(cudaStreamWaitEvent(h2d, ctx->ev_start, 0));
  SEER_TRY(cudaStreamWaitEvent(d2h, ctx->ev_start, 0));
  // The copies in are what the call is bound by (55 GB/s), so what follows the last of them counts in full: the kernels of the last
  // slice and its read-back.  The last slice is therefore taken in parts of its query heads, each of more than 8 MB (150 us
  // of copying, as long as the kernels of that many heads take): the parts' kernels and read-backs overlap the copies of the later
  // parts (32 / 8 heads, a tenth kept, 128k tokens: 36.1 ms with the slice whole, 34.8 so; parts of 4 MB: no faster).
  int tail_heads = (int)(((size_t)8 << 20) / (T * head_bytes)) + 1;
  while (tail_heads < G && G % tail_heads != 0) ++tail_heads;
  if (tail_heads > G) tail_heads = G;
  for (int g = 0; g < Hkv; ++g) {
    const int b = g & 1;
    // ---- host -> device: the slice's heads are strided in the host tensors ([T, H, 128]) and packed on the device
    if (g >= 2) SEER_TRY(cudaStreamWaitEvent(h2d, ctx->ev_comp[b], 0));   // slice g - 2 has finished with these buffers
    SEER_TRY(cudaMemcpy2DAsync(d + a.k[b], head_bytes, (const char*)k_host + (size_t)g * head_bytes, (size_t)Hkv * head_bytes,
                               head_bytes, T, cudaMemcpyHostToDevice, h2d));
    SEER_TRY(cudaMemcpy2DAsync(d + a.v[b], head_bytes, (const char*)v_host + (size_t)g * head_bytes, (size_t)Hkv * head_bytes,
                               head_bytes, T, cudaMemcpyHostToDevice, h2d));
    SEER_TRY(cudaMemcpyAsync(d + a.wq[b], (const char*)Wq_host + (size_t)g * wq_bytes, wq_bytes, cudaMemcpyHostToDevice, h2d));
    SEER_TRY(cudaMemcpyAsync(d + a.wk[b], (const char*)Wk_host + (size_t)g * wk_bytes, wk_bytes, cudaMemcpyHostToDevice, h2d));
    if (g >= 2) SEER_TRY(cudaStreamWaitEvent(stream, ctx->ev_d2h[b], 0));  // o / lse of slice g - 2 have been read back
    seer_shape part = slice;
    part.num_q_heads = g == Hkv - 1 ? tail_heads : G;
    const size_t P = (size_t)part.num_q_heads;
    for (size_t h0 = 0; h0 < (size_t)G; h0 += P) {         // heads h0 .. h0 + P - 1 of the slice
      const size_t head = (size_t)g * G + h0;
      char *dq = d + a.q[b] + h0 * T * head_bytes, *dout = d + a.o[b] + h0 * T * head_bytes;
      float* dlse = lse_host ? (float*)(d + a.lse[b]) + h0 * T : nullptr;
      SEER_TRY(cudaMemcpy2DAsync(dq, P * head_bytes, (const char*)q_host + head * head_bytes, (size_t)Hq * head_bytes, P * head_bytes, T,
                                 cudaMemcpyHostToDevice, h2d));
      SEER_TRY(cudaEventRecord(ctx->ev_h2d[b], h2d));
      // ---- the three calls, on the caller's stream
      SEER_TRY(cudaStreamWaitEvent(stream, ctx->ev_h2d[b], 0));
      st = seer_gate_scores(ctx, &part, dq, d + a.k[b], (const float*)(d + a.wq[b]) + h0 * kHeadDim * kGateDim, (const float*)(d + a.wk[b]),
                            (float*)(d + a.scores), d + a.ws, ws_bytes, stream);
      if (st != SEER_OK) return st;
      st = seer_block_mask(ctx, &part, (const float*)(d + a.scores), params, (int32_t*)(d + a.row_ptr),
                           (int32_t*)(d + a.col_idx), t.causal_blocks, (int64_t*)(d + a.nnz), nullptr, 0, stream);
      if (st != SEER_OK) return st;
      st = seer_sparse_attn(ctx, &part, dq, d + a.k[b], d + a.v[b], (const int32_t*)(d + a.row_ptr), (const int32_t*)(d + a.col_idx),
                            dout, dlse, d + a.ws, ws_bytes, stream);   // (the gate's workspace is free again: the attention's work counter)
      if (st != SEER_OK) return st;
      SEER_TRY(cudaEventRecord(ctx->ev_comp[b], stream));
      // ---- device -> host
      SEER_TRY(cudaStreamWaitEvent(d2h, ctx->ev_comp[b], 0));
      SEER_TRY(cudaMemcpy2DAsync((char*)o_host + head * head_bytes, (size_t)Hq * head_bytes, dout, P * head_bytes, P * head_bytes, T,
                                 cudaMemcpyDeviceToHost, d2h));
      if (lse_host) SEER_TRY(cudaMemcpyAsync(lse_host + head * T, dlse, P * T * 4, cudaMemcpyDeviceToHost, d2h));
      SEER_TRY(cudaEventRecord(ctx->ev_d2h[b], d2h));
    }
  }
  // the caller's stream is complete when the last read-backs are
  SEER_TRY(cudaStreamWaitEvent(stream, ctx->ev_d2h[(Hkv - 1) & 1], 0));
  if (Hkv >= 2) SEER_TRY(cudaStreamWaitEvent(stream, ctx->ev_d2h[Hkv & 1], 0));
#undef SEER_TRY
  return SEER_OK;
}

}  // extern "C"
