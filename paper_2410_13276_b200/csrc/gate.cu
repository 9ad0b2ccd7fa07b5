// AttnGate (Sec. 3.1, Eq. 1) in two kernels:
//   pool_project_kernel : streams Q and K once (HBM-bound), average-pools each 64-token block per head and
//                         multiplies the pooled vectors by the head's gate matrix (fp32 on the CUDA cores) -> gq, gk
//   gate_scores_kernel  : logits = gq gk^T / sqrt(dg) over the causal blocks, row softmax -> scores (gate_scores.cu)
// The logits need fp32-grade products (plain bf16 or tf32 tensor-core inputs would not hold the 1e-3 relative bound on
// softmax outputs when logits reach tens), so gq and gk are stored as three bf16 planes each, x = hi + mid + lo with
// every part the bf16 rounding of what is left, and the second kernel takes the product on the tensor cores as six
// bf16 terms.
#include <cuda_bf16.h>
#include <math_constants.h>

#include <cstddef>
#include <mutex>

#include "seer_internal.cuh"

namespace seer {

// ----------------------------------------------------------------------------------------------- kernel 1
constexpr int kPoolThreads = 256;
constexpr int kPoolChunkEx = 16;            // blocks per CTA of the variants' kernel
constexpr unsigned kBigChunkFrom = 600;   // CTAs of 16 blocks from which the large chunk is taken

// Element o of the projected vector of block gb (numbered over the batch) as x = hi + mid + lo, each part the bf16
// (round-to-nearest-even) of the remainder, into the tile layout of the head's planes.
__device__ __forceinline__ void store_split3(char* __restrict__ head, int total_blocks, int gb, int o, float x) {
  const __nv_bfloat16 hi = __float2bfloat16_rn(x);
  const float r1 = x - __bfloat162float(hi);
  const __nv_bfloat16 mid = __float2bfloat16_rn(r1);
  const float r2 = r1 - __bfloat162float(mid);
  const __nv_bfloat16 lo = __float2bfloat16_rn(r2);
  const GateTile t(gb >> 6, total_blocks);
  const int plane = t.rows * 256;
  char* dst = head + t.base + (size_t)((o >> 6) * t.rows * 128 + (gb & 63) * 128 + ((((o >> 3) & 7) ^ (gb & 7)) << 4) + (o & 7) * 2);
  *reinterpret_cast<uint16_t*>(dst) = __bfloat16_as_ushort(hi);
  *reinterpret_cast<uint16_t*>(dst + plane) = __bfloat16_as_ushort(mid);
  *reinterpret_cast<uint16_t*>(dst + 2 * plane) = __bfloat16_as_ushort(lo);
}

// Four consecutive elements, the first a multiple of four.
__device__ __forceinline__ void store_split3x4(char* __restrict__ head, int total_blocks, int gb, int o, const float4& x) {
  const float v[4] = {x.x, x.y, x.z, x.w};
  uint32_t pl[3][2];
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const __nv_bfloat162 hi = __floats2bfloat162_rn(v[2 * i], v[2 * i + 1]);
    const float2 h = __bfloat1622float2(hi);
    const float a1 = v[2 * i] - h.x, b1 = v[2 * i + 1] - h.y;
    const __nv_bfloat162 mid = __floats2bfloat162_rn(a1, b1);
    const float2 g = __bfloat1622float2(mid);
    const __nv_bfloat162 lo = __floats2bfloat162_rn(a1 - g.x, b1 - g.y);
    pl[0][i] = *reinterpret_cast<const uint32_t*>(&hi);
    pl[1][i] = *reinterpret_cast<const uint32_t*>(&mid);
    pl[2][i] = *reinterpret_cast<const uint32_t*>(&lo);
  }
  const GateTile t(gb >> 6, total_blocks);
  const int plane = t.rows * 256;
  char* dst = head + t.base + (size_t)((o >> 6) * t.rows * 128 + (gb & 63) * 128 + ((((o >> 3) & 7) ^ (gb & 7)) << 4) + (o & 7) * 2);
#pragma unroll
  for (int q = 0; q < 3; ++q) *reinterpret_cast<uint2*>(dst + q * plane) = make_uint2(pl[q][0], pl[q][1]);
}

// Four consecutive columns of a gate matrix: one load where the matrices begin on 16 bytes, otherwise four.
template <bool kVecW>
__device__ __forceinline__ float4 ld_w4(const float* __restrict__ p) {
  if (kVecW) return __ldg(reinterpret_cast<const float4*>(p));
  return make_float4(__ldg(p), __ldg(p + 1), __ldg(p + 2), __ldg(p + 3));
}
static bool vec_w(const float* Wq, const float* Wk) { return (((uintptr_t)Wq | (uintptr_t)Wk) & 15) == 0; }   // (a head's matrix is 64 KB)

__device__ __forceinline__ uint4 ld_stream_16(const void* p) {
  uint4 r;
  asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];"
               : "=r"(r.x), "=r"(r.y), "=r"(r.z), "=r"(r.w) : "l"(p));
  return r;
}

__device__ __forceinline__ void acc_bf16x8(float (&a)[8], const uint4& u) {
  a[0] += __uint_as_float(u.x << 16); a[1] += __uint_as_float(u.x & 0xffff0000u);
  a[2] += __uint_as_float(u.y << 16); a[3] += __uint_as_float(u.y & 0xffff0000u);
  a[4] += __uint_as_float(u.z << 16); a[5] += __uint_as_float(u.z & 0xffff0000u);
  a[6] += __uint_as_float(u.w << 16); a[7] += __uint_as_float(u.w & 0xffff0000u);
}

// What a CTA pools: a chunk of blocks of one head, the head varying fastest so that CTAs running together read neighbouring
// 256-byte segments of the same token rows.  Chunked prefill: most chunks of Q lie before its queries, and CTAs with nothing to
// do between those of K keep the memory system idle.  So K comes first there, and of Q the chunks of a single sequence that
// lie before its queries have no CTA, other such CTAs leave at once (8k tokens against 128k: 135 us, 78 so).
struct PoolWork {
  int chunk, h, H;
  bool is_q, idle;
  __device__ __forceinline__ PoolWork(const SeqMeta& m, int blocks) {
    idle = false;
    if (!m.chunked) {
      const int heads = m.num_q_heads + m.num_kv_heads, hh = (int)blockIdx.x % heads;
      chunk = (int)blockIdx.x / heads;
      is_q = hh < m.num_q_heads;
      H = is_q ? m.num_q_heads : m.num_kv_heads;
      h = is_q ? hh : hh - m.num_q_heads;
      return;
    }
    const int kv = (m.total_blocks + blocks - 1) / blocks * m.num_kv_heads;
    is_q = (int)blockIdx.x >= kv;
    const int at = is_q ? (int)blockIdx.x - kv : (int)blockIdx.x;
    H = is_q ? m.num_q_heads : m.num_kv_heads;
    chunk = at / H;
    h = at - chunk * H;
    if (is_q) {
      chunk += m.first_q_block / blocks;
      const int lane = threadIdx.x & 31, g = chunk * blocks + lane;
      bool live = false;
      if (lane < blocks && g < m.total_blocks) {
        const int b = find_sequence(m.blk_off, m.batch, g);
        live = g - m.blk_off[b] >= m.qoff[b];
      }
      idle = !__any_sync(0xffffffffu, live);               // (the same in every warp)
    }
  }
  static unsigned grid(const SeqMeta& m, int blocks) {
    const int chunks = (m.total_blocks + blocks - 1) / blocks;
    return (unsigned)chunks * (unsigned)m.num_kv_heads + (unsigned)(chunks - m.first_q_block / blocks) * (unsigned)m.num_q_heads;
  }
};

// One CTA pools and projects kChunk consecutive blocks of the packed batch (whatever sequences they belong to: a chunk per
// sequence would leave most of a CTA idle on batches of short ones) for one head.
//
// What bounds it: the bytes of Q and K in a large batch; in a small one the latency of a CTA's loads, one after the other,
// because there are too few CTAs.  So a chunk is 16 blocks where that still makes more than a wave of CTAs (the head's 64 KB
// matrix, read once per CTA from L2, is then a fifth of its traffic) and 2 blocks otherwise, with four warps per block.
// The sums are formed in the same order for every chunk size (16 rows at a time; the two halves of the matrix's rows apart),
// so the result does not depend on it.
template <int kChunk, bool kVecW = true>
__global__ void __launch_bounds__(kPoolThreads, kChunk == 16 ? 3 : 1)
pool_project_kernel(SeqMeta m, const uint16_t* __restrict__ q, const uint16_t* __restrict__ k,
                    const float* __restrict__ Wq, const float* __restrict__ Wk, char* __restrict__ gq,
                    char* __restrict__ gk) {
  constexpr int kWarps = kPoolThreads / 32;
  constexpr int kSplit = kChunk < kWarps ? kWarps / kChunk : 1;      // warps per block
  constexpr int kMaxSteps = 8;                                       // groups of 16 rows in a block of 128 tokens
  __shared__ __align__(16) float pooled[kChunk == 16 ? 1 : kChunk][kHeadDim];
  __shared__ __align__(16) float by_col[kChunk == 16 ? kHeadDim * 16 + kHeadDim / 2 : 4];   // [column][block], 16 bytes more per eight columns
  __shared__ __align__(16) float part[kSplit > 1 ? kChunk * kMaxSteps * 2 * kHeadDim : kChunk * kHeadDim];

  const PoolWork work(m, kChunk);
  grid_wait();
  if (work.idle) return;
  const int chunk = work.chunk, H = work.H, h = work.h;
  const bool is_q = work.is_q;
  const uint16_t* __restrict__ x = is_q ? q : k;
  const float* __restrict__ W = (is_q ? Wq : Wk) + (size_t)h * kHeadDim * kGateDim;
  char* __restrict__ out = (is_q ? gq : gk) + (size_t)h * m.total_blocks * kGatePairBytes;

  const int g0 = chunk * kChunk;                                // first block of the chunk, numbered over the batch
  const int nblk = min(kChunk, m.total_blocks - g0);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int half = lane >> 4, cchunk = lane & 15;
  const size_t row_stride = (size_t)H * kHeadDim;  // elements between consecutive tokens
  const int steps = m.block / 16;
  bool any = false;

  for (int bi = warp / kSplit; bi < nblk; bi += kWarps / kSplit) {
    const int b = find_sequence(m.blk_off, m.batch, g0 + bi);
    const int i = g0 + bi - m.blk_off[b];
    const int s0 = m.cu_seqlens[b], s1 = m.cu_seqlens[b + 1];
    // chunked prefill: q holds the last positions only; query blocks before the chunk are skipped (projected as zeros)
    const int q_first = (m.chunked && is_q) ? m.qoff[b] : 0;
    const int q_shift = (m.chunked && is_q) ? m.qdelta[b] : 0;
    const int t0 = s0 + i * m.block;
    const int cnt = (i < q_first) ? 0 : min(m.block, s1 - t0);
    any |= cnt > 0;
    const uint16_t* base = x + ((ptrdiff_t)t0 + q_shift) * (ptrdiff_t)row_stride + (size_t)h * kHeadDim + cchunk * 8;
    float a[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll 1
    for (int st = warp % kSplit; st < steps; st += kSplit) {
      uint4 u[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const int row = 16 * st + 2 * j + half;
        u[j] = row < cnt ? ld_stream_16(base + (size_t)row * row_stride) : make_uint4(0, 0, 0, 0);
      }
      float t[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int j = 0; j < 8; ++j) acc_bf16x8(t, u[j]);
      if (kSplit > 1) {
        float4* dst = reinterpret_cast<float4*>(&part[((bi * kMaxSteps + st) * 2 + half) * kHeadDim + cchunk * 8]);
        dst[0] = make_float4(t[0], t[1], t[2], t[3]);
        dst[1] = make_float4(t[4], t[5], t[6], t[7]);
      } else {
#pragma unroll
        for (int j = 0; j < 8; ++j) a[j] = __fadd_rn(a[j], t[j]);
      }
    }
    if (kSplit == 1) {
      const float inv = cnt > 0 ? 1.0f / (float)cnt : 0.f;
#pragma unroll
      for (int j = 0; j < 8; ++j) a[j] = __fmul_rn(__fadd_rn(a[j], __shfl_xor_sync(0xffffffffu, a[j], 16)), inv);
#pragma unroll
      for (int e = 0; e < 4; ++e) by_col[(cchunk * 8 + half * 4 + e) * 16 + cchunk * 4 + bi] = half ? a[4 + e] : a[e];
    } else if (lane == 0 && warp % kSplit == 0) pooled[bi][0] = cnt > 0 ? 1.0f / (float)cnt : 0.f;   // (until the sums are combined)
  }
  if (!__syncthreads_or(any ? 1 : 0)) return;                   // every block of the chunk lies before its queries
  if (kSplit > 1) {
    float v[(kChunk * kHeadDim + kPoolThreads - 1) / kPoolThreads];
    int e = 0;
#pragma unroll
    for (int idx = threadIdx.x; idx < kChunk * kHeadDim; idx += kPoolThreads, ++e) {
      const int bi = idx / kHeadDim, c = idx % kHeadDim;
      float s0 = 0.f, s1 = 0.f;
      for (int st = 0; st < steps; ++st) {
        s0 = __fadd_rn(s0, part[((bi * kMaxSteps + st) * 2) * kHeadDim + c]);
        s1 = __fadd_rn(s1, part[((bi * kMaxSteps + st) * 2 + 1) * kHeadDim + c]);
      }
      v[e] = __fmul_rn(__fadd_rn(s0, s1), pooled[bi][0]);
    }
    __syncthreads();
    e = 0;
#pragma unroll
    for (int idx = threadIdx.x; idx < kChunk * kHeadDim; idx += kPoolThreads, ++e) pooled[idx / kHeadDim][idx % kHeadDim] = v[e];
    __syncthreads();
  }

  if constexpr (kChunk == 16) {
    // projection: a thread takes four output columns, four blocks and one half of the matrix's rows, two columns to an instruction.
    // What bounds it is the 128 bytes a clock that loads return to the registers: a step is 16 bytes of W, 16 of four blocks'
    // column and 16 products (a column and sixteen blocks to a thread: 68 bytes for as many, and 296 us where this takes 266 at 128k
    // tokens, 32 / 8 heads; the bytes take 205).
    const int bg = warp & 3, ch = warp >> 2, o = 4 * lane;
    float2 acc[4][2];
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[j][0] = acc[j][1] = make_float2(0.f, 0.f);
    const float* __restrict__ Wh = W + (size_t)ch * 64 * kGateDim + o;
#pragma unroll 2
    for (int c = 0; c < 64; c += 8) {
      float4 w[8];
#pragma unroll
      for (int e = 0; e < 8; ++e) w[e] = ld_w4<kVecW>(Wh + (size_t)(c + e) * kGateDim);
      const float4* col = reinterpret_cast<const float4*>(by_col + (ch * 64 + c) * 16 + (ch * 64 + c) / 2) + bg;
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        const float4 pv = col[e * 4];
        const float2 w0 = make_float2(w[e].x, w[e].y), w1 = make_float2(w[e].z, w[e].w);
        acc[0][0] = __ffma2_rn(make_float2(pv.x, pv.x), w0, acc[0][0]); acc[0][1] = __ffma2_rn(make_float2(pv.x, pv.x), w1, acc[0][1]);
        acc[1][0] = __ffma2_rn(make_float2(pv.y, pv.y), w0, acc[1][0]); acc[1][1] = __ffma2_rn(make_float2(pv.y, pv.y), w1, acc[1][1]);
        acc[2][0] = __ffma2_rn(make_float2(pv.z, pv.z), w0, acc[2][0]); acc[2][1] = __ffma2_rn(make_float2(pv.z, pv.z), w1, acc[2][1]);
        acc[3][0] = __ffma2_rn(make_float2(pv.w, pv.w), w0, acc[3][0]); acc[3][1] = __ffma2_rn(make_float2(pv.w, pv.w), w1, acc[3][1]);
      }
    }
    // the halves are added by the thread that stores: the first half's threads two blocks, the second half's the other two
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if ((j >= 2) != (ch == 1))
        *reinterpret_cast<float4*>(&part[(bg * 4 + j) * kGateDim + o]) = make_float4(acc[j][0].x, acc[j][0].y, acc[j][1].x, acc[j][1].y);
    __syncthreads();
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if ((j >= 2) == (ch == 1) && bg * 4 + j < nblk) {
        const float4 t = *reinterpret_cast<const float4*>(&part[(bg * 4 + j) * kGateDim + o]);
        store_split3x4(out, m.total_blocks, g0 + bg * 4 + j, o, make_float4(__fadd_rn(acc[j][0].x, t.x), __fadd_rn(acc[j][0].y, t.y),
                                                                            __fadd_rn(acc[j][1].x, t.z), __fadd_rn(acc[j][1].y, t.w)));
      }
    return;
  }

  // projection: a thread takes output column o, one half of the matrix's rows and all blocks of the chunk
  const int o = threadIdx.x & (kGateDim - 1);
  const int ch = threadIdx.x >> 7;
  float acc[kChunk];
#pragma unroll
  for (int j = 0; j < kChunk; ++j) acc[j] = 0.f;
  const float* __restrict__ Wh = W + (size_t)ch * 64 * kGateDim + o;
#pragma unroll 2
  for (int c = 0; c < 64; c += 8) {
    float w[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) w[e] = __ldg(Wh + (size_t)(c + e) * kGateDim);
#pragma unroll
    for (int j = 0; j < kChunk; ++j) {
      const float4 p0 = *reinterpret_cast<const float4*>(&pooled[j][ch * 64 + c]), p1 = *reinterpret_cast<const float4*>(&pooled[j][ch * 64 + c + 4]);
      acc[j] = fmaf(p0.x, w[0], acc[j]); acc[j] = fmaf(p0.y, w[1], acc[j]); acc[j] = fmaf(p0.z, w[2], acc[j]); acc[j] = fmaf(p0.w, w[3], acc[j]);
      acc[j] = fmaf(p1.x, w[4], acc[j]); acc[j] = fmaf(p1.y, w[5], acc[j]); acc[j] = fmaf(p1.z, w[6], acc[j]); acc[j] = fmaf(p1.w, w[7], acc[j]);
    }
  }
  // the halves are added by the thread that stores: the first half of the threads the first half of the blocks
#pragma unroll
  for (int j = 0; j < kChunk; ++j) if ((j >= kChunk / 2) != (ch == 1)) part[j * kGateDim + o] = acc[j];
  __syncthreads();
#pragma unroll
  for (int j = 0; j < kChunk; ++j)
    if ((j >= kChunk / 2) == (ch == 1) && j < nblk) store_split3(out, m.total_blocks, g0 + j, o, __fadd_rn(acc[j], part[j * kGateDim + o]));
}


// ----------------------------------------------------------------------------------------------- kernel 1, variants
// Sec. 3.1, "Pooling Method Selection" and "Block-level RoPE in AttnGate": the same single pass over Q and K, but
//   * a tensor may be pooled by any subset of {average, max, min}; the pooled vectors are concatenated in that order
//     in the hidden dimension, so the head's gate matrix is [n * d, dg] (n = methods chosen for that tensor);
//   * with rope_theta > 0 the projected vector of block i is rotated as position i with base rope_theta / B
//     (pairs (c, c + dg/2), frequency base^(-2c/dg)); the angle and its sine / cosine are taken in double precision
//     (an fp32 angle near position 2000 would already cost more than the 1e-3 bound on large logits).
// max and min ride along the average's loads: the kernel stays one HBM pass.
__device__ __forceinline__ void max_bf16x8(float (&a)[8], const uint4& u) {
  a[0] = fmaxf(a[0], __uint_as_float(u.x << 16)); a[1] = fmaxf(a[1], __uint_as_float(u.x & 0xffff0000u));
  a[2] = fmaxf(a[2], __uint_as_float(u.y << 16)); a[3] = fmaxf(a[3], __uint_as_float(u.y & 0xffff0000u));
  a[4] = fmaxf(a[4], __uint_as_float(u.z << 16)); a[5] = fmaxf(a[5], __uint_as_float(u.z & 0xffff0000u));
  a[6] = fmaxf(a[6], __uint_as_float(u.w << 16)); a[7] = fmaxf(a[7], __uint_as_float(u.w & 0xffff0000u));
}
__device__ __forceinline__ void min_bf16x8(float (&a)[8], const uint4& u) {
  a[0] = fminf(a[0], __uint_as_float(u.x << 16)); a[1] = fminf(a[1], __uint_as_float(u.x & 0xffff0000u));
  a[2] = fminf(a[2], __uint_as_float(u.y << 16)); a[3] = fminf(a[3], __uint_as_float(u.y & 0xffff0000u));
  a[4] = fminf(a[4], __uint_as_float(u.z << 16)); a[5] = fminf(a[5], __uint_as_float(u.z & 0xffff0000u));
  a[6] = fminf(a[6], __uint_as_float(u.w << 16)); a[7] = fminf(a[7], __uint_as_float(u.w & 0xffff0000u));
}


// The pooling of the gate's variants: average, maximum and minimum of a block side by side, one product with the wider matrix, and
// the block rotation.  Bound by issue and shared memory beside the bytes: only the pools asked for are formed, an angle's cosine and
// sine are taken once per block and pair, by the warps that do not project, and three CTAs share an SM (49k tokens, average of Q, all
// three of K, rotation, with the scores: 178 us; 223 without any of this and a column of eight blocks to a thread; the bytes take 77).
template <bool kVecW>
__global__ void __launch_bounds__(kPoolThreads, 3)
pool_project_ex_kernel(SeqMeta m, const uint16_t* __restrict__ q, const uint16_t* __restrict__ k,
                       const float* __restrict__ Wq, const float* __restrict__ Wk, char* __restrict__ gq,
                       char* __restrict__ gk, uint32_t pool_q, uint32_t pool_k, float rope_theta) {
  constexpr int kChunk = kPoolChunkEx;
  __shared__ __align__(16) float by_col[3 * kHeadDim * kChunk + 3 * kHeadDim / 2];   // [column][block], 16 bytes more per eight columns
  __shared__ __align__(16) double2 turn[kChunk][kGateDim / 2];   // cosine and sine of each block's angle, by pair
  __shared__ int block_pos[kChunk];                        // position of each block in its sequence (block RoPE)
  __shared__ double angle[kGateDim / 2];                   // of one block's step, by pair

  const PoolWork work(m, kChunk);
  if (rope_theta > 0.f && threadIdx.x < kGateDim / 2)
    angle[threadIdx.x] = pow((double)rope_theta / (double)m.block, -2.0 * (double)threadIdx.x / (double)kGateDim);
  grid_wait();
  if (work.idle) return;
  const int chunk = work.chunk, H = work.H, h = work.h;
  const bool is_q = work.is_q;
  const uint32_t methods = is_q ? pool_q : pool_k;
  const bool extremes = (methods & ~SEER_POOL_AVG) != 0u;
  const int nparts = __popc(methods);
  const int width = nparts * kHeadDim;                       // rows of the head's gate matrix
  const uint16_t* __restrict__ x = is_q ? q : k;
  const float* __restrict__ W = (is_q ? Wq : Wk) + (size_t)h * width * kGateDim;
  char* __restrict__ out = (is_q ? gq : gk) + (size_t)h * m.total_blocks * kGatePairBytes;
  // offsets of the parts inside the concatenated vector (order: average, max, min)
  const int off_avg = 0;
  const int off_max = (methods & SEER_POOL_AVG) ? kHeadDim : 0;
  const int off_min = off_max + ((methods & SEER_POOL_MAX) ? kHeadDim : 0);

  const int g0 = chunk * kChunk;                            // first block of the chunk, numbered over the batch
  const int nblk = min(kChunk, m.total_blocks - g0);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int half = lane >> 4, cchunk = lane & 15;
  const size_t row_stride = (size_t)H * kHeadDim;
  bool any = false;

  for (int bi = warp; bi < nblk; bi += kPoolThreads / 32) {
    const int b = find_sequence(m.blk_off, m.batch, g0 + bi);
    const int i = g0 + bi - m.blk_off[b];
    const int s0 = m.cu_seqlens[b], s1 = m.cu_seqlens[b + 1];
    // chunked prefill: q holds the last positions only; query blocks before the chunk are skipped (projected as zeros)
    const int q_first = (m.chunked && is_q) ? m.qoff[b] : 0;
    const int q_shift = (m.chunked && is_q) ? m.qdelta[b] : 0;
    const int t0 = s0 + i * m.block;
    const int cnt = (i < q_first) ? 0 : min(m.block, s1 - t0);
    any |= cnt > 0;
    if (lane == 0) block_pos[bi] = i;
    const uint16_t* base = x + ((ptrdiff_t)t0 + q_shift) * (ptrdiff_t)row_stride + (size_t)h * kHeadDim + cchunk * 8;
    float a[8], hi[8], lo[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) { a[j] = 0.f; hi[j] = -CUDART_INF_F; lo[j] = CUDART_INF_F; }
#pragma unroll 1
    for (int it = 0; it < m.block / 2; it += 8) {
      uint4 u[8];
      bool live[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const int row = 2 * (it + j) + half;
        live[j] = row < cnt;
        u[j] = live[j] ? ld_stream_16(base + (size_t)row * row_stride) : make_uint4(0, 0, 0, 0);
      }
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        acc_bf16x8(a, u[j]);
        if (extremes && live[j]) { max_bf16x8(hi, u[j]); min_bf16x8(lo, u[j]); }   // rows past the end of the sequence take no part
      }
    }
    const float inv = cnt > 0 ? 1.0f / (float)cnt : 0.f;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      a[j] = (a[j] + __shfl_xor_sync(0xffffffffu, a[j], 16)) * inv;
      hi[j] = fmaxf(hi[j], __shfl_xor_sync(0xffffffffu, hi[j], 16));
      lo[j] = fminf(lo[j], __shfl_xor_sync(0xffffffffu, lo[j], 16));
      if (cnt == 0) { hi[j] = 0.f; lo[j] = 0.f; }      // a skipped block: zeros, not the identities of max and min
    }
    auto put = [&](int off, const float (&v)[8]) {
#pragma unroll
      for (int e = 0; e < 4; ++e) by_col[(off + cchunk * 8 + half * 4 + e) * kChunk + (off / 8 + cchunk) * 4 + bi] = half ? v[4 + e] : v[e];
    };
    if (methods & SEER_POOL_AVG) put(off_avg, a);
    if (methods & SEER_POOL_MAX) put(off_max, hi);
    if (methods & SEER_POOL_MIN) put(off_min, lo);
  }
  if (!__syncthreads_or(any ? 1 : 0)) return;                   // every block of the chunk lies before its queries

  // projection, by four warps: a thread takes four output columns and four blocks, as in pool_project_kernel; the other four warps take
  // the cosines and sines meanwhile
  const int o = 4 * lane, bg = warp & 3;
  float2 acc[4][2];
  if (warp < 4) {
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[j][0] = acc[j][1] = make_float2(0.f, 0.f);
    const float* __restrict__ Wh = W + o;
#pragma unroll 2
    for (int c = 0; c < width; c += 8) {
      float4 w[8];
#pragma unroll
      for (int e = 0; e < 8; ++e) w[e] = ld_w4<kVecW>(Wh + (size_t)(c + e) * kGateDim);
      const float4* col = reinterpret_cast<const float4*>(by_col + c * kChunk + c / 2) + bg;
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        const float4 pv = col[e * (kChunk / 4)];
        const float2 w0 = make_float2(w[e].x, w[e].y), w1 = make_float2(w[e].z, w[e].w);
        acc[0][0] = __ffma2_rn(make_float2(pv.x, pv.x), w0, acc[0][0]); acc[0][1] = __ffma2_rn(make_float2(pv.x, pv.x), w1, acc[0][1]);
        acc[1][0] = __ffma2_rn(make_float2(pv.y, pv.y), w0, acc[1][0]); acc[1][1] = __ffma2_rn(make_float2(pv.y, pv.y), w1, acc[1][1]);
        acc[2][0] = __ffma2_rn(make_float2(pv.z, pv.z), w0, acc[2][0]); acc[2][1] = __ffma2_rn(make_float2(pv.z, pv.z), w1, acc[2][1]);
        acc[3][0] = __ffma2_rn(make_float2(pv.w, pv.w), w0, acc[3][0]); acc[3][1] = __ffma2_rn(make_float2(pv.w, pv.w), w1, acc[3][1]);
      }
    }
  } else if (rope_theta > 0.f) {
    const int f = threadIdx.x & (kGateDim / 2 - 1);
    const double freq = angle[f];
    for (int bi = (threadIdx.x - 128) / (kGateDim / 2); bi < nblk; bi += 128 / (kGateDim / 2)) {
      double sn, cs;
      sincos((double)block_pos[bi] * freq, &sn, &cs);
      turn[bi][f] = make_double2(cs, sn);
    }
  }
  if (rope_theta > 0.f) __syncthreads();
  if (warp >= 4) return;
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int bi = bg * 4 + j;
    float v[4] = {acc[j][0].x, acc[j][0].y, acc[j][1].x, acc[j][1].y};
    if (rope_theta > 0.f) {
      // rotate (o, o + dg/2) pairs: the partner's value is that of lane ^ 16
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const float partner = __shfl_xor_sync(0xffffffffu, v[u], 16);
        const double2 t = turn[bi][(o + u) & (kGateDim / 2 - 1)];
        // first half: x1 cos - x2 sin; second half: x2 cos + x1 sin
        v[u] = lane < 16 ? (float)((double)v[u] * t.x - (double)partner * t.y) : (float)((double)v[u] * t.x + (double)partner * t.y);
      }
    }
    if (bi < nblk) store_split3x4(out, m.total_blocks, g0 + bi, o, make_float4(v[0], v[1], v[2], v[3]));
  }
}

// ----------------------------------------------------------------------------------------------- kernel 2
// gate_scores_kernel (tcgen05) lives in gate_scores.cu.
int launch_gate_stats(const SeqMeta& m, const uint16_t* gq, const uint16_t* gk, float2* stats, int* status, cudaStream_t stream);
int launch_gate_scores(const SeqMeta& m, const ScoreBand& band, const uint16_t* gq, const uint16_t* gk, float* scores,
                       float2* stats, int* status, int num_sms, cudaStream_t stream);
int launch_gate_logits(const SeqMeta& m, const ScoreBand& band, const uint16_t* gq, const uint16_t* gk, float* logits, float2* stats,
                       int* status, int num_sms, cudaStream_t stream);
bool init_gate_scores();

namespace {
// The workspace: planes of gq, of gk and, where it has room, the statistics.
struct GateWs {
  char *gq, *gk;
  float2* stats;
  GateWs(const SeqMeta& m, void* ws, size_t ws_bytes) {
    auto up = [](size_t x) { return (x + 255) / 256 * 256; };
    gq = (char*)ws;
    gk = gq + up((size_t)m.num_q_heads * m.total_blocks * kGatePairBytes);
    stats = (float2*)(gk + up((size_t)m.num_kv_heads * m.total_blocks * kGatePairBytes));
    if ((size_t)((char*)stats - gq) + (size_t)m.num_q_heads * m.total_blocks * gate_stat_segs(m.max_nb) * sizeof(float2) > ws_bytes) stats = nullptr;
  }
};

int launch_scores_whole(seer_ctx* ctx, const SeqMeta& m, const GateWs& w, float* scores, cudaStream_t stream) {
  int* status = ctx ? ctx->d_status : nullptr;
  // (the allocation-free variant has no context)
  float2* stats = ctx && gate_split(m, ctx->num_sms) ? w.stats : nullptr;
  const int n1 = stats ? launch_gate_stats(m, (const uint16_t*)w.gq, (const uint16_t*)w.gk, stats, status, stream) : 0;
  if (n1 < 0) return n1;
  const ScoreBand all = {m.first_q_block, m.total_blocks, 0, m.num_q_heads, 0, 0, 0};
  const int n2 = launch_gate_scores(m, all, (const uint16_t*)w.gq, (const uint16_t*)w.gk, scores, stats, status, ctx ? ctx->num_sms : 0, stream);
  return n2 < 0 ? n2 : n1 + n2;
}
}  // namespace

int launch_gate(seer_ctx* ctx, const SeqMeta& m, const void* q, const void* k, const float* Wq, const float* Wk,
                float* scores, void* ws, size_t ws_bytes, cudaStream_t stream) {
  const GateWs w(m, ws, ws_bytes);
  const unsigned big = PoolWork::grid(m, 16);
  const cudaError_t e0 = big > kBigChunkFrom
      ? launch_next(vec_w(Wq, Wk) ? pool_project_kernel<16> : pool_project_kernel<16, false>, big, kPoolThreads, 0, stream, m, (const uint16_t*)q, (const uint16_t*)k, Wq, Wk, w.gq, w.gk)
      : launch_next(pool_project_kernel<2>, PoolWork::grid(m, 2), kPoolThreads, 0, stream, m, (const uint16_t*)q, (const uint16_t*)k, Wq, Wk, w.gq, w.gk);
  if (e0 != cudaSuccess) return -(int)e0;
  if (scores == nullptr) return 1;                     // projection only: the scores follow band by band
  const int n2 = launch_scores_whole(ctx, m, w, scores, stream);
  return n2 < 0 ? n2 : 1 + n2;
}

int launch_gate_ex(seer_ctx* ctx, const SeqMeta& m, const seer_gate_options& opt, const void* q, const void* k,
                   const float* Wq, const float* Wk, float* scores, void* ws, size_t ws_bytes, cudaStream_t stream) {
  // averages alone and no rotation: the plain gate
  if (opt.pool_q == SEER_POOL_AVG && opt.pool_k == SEER_POOL_AVG && opt.rope_theta == 0.f) return launch_gate(ctx, m, q, k, Wq, Wk, scores, ws, ws_bytes, stream);
  const GateWs w(m, ws, ws_bytes);
  const unsigned grid1 = PoolWork::grid(m, kPoolChunkEx);
  const cudaError_t e0 = launch_next(vec_w(Wq, Wk) ? pool_project_ex_kernel<true> : pool_project_ex_kernel<false>, grid1, kPoolThreads, 0, stream, m, (const uint16_t*)q, (const uint16_t*)k, Wq, Wk,
                                     w.gq, w.gk, opt.pool_q, opt.pool_k, opt.rope_theta);
  if (e0 != cudaSuccess) return -(int)e0;
  if (scores == nullptr) return 1;
  const int n2 = launch_scores_whole(ctx, m, w, scores, stream);
  return n2 < 0 ? n2 : 1 + n2;
}

int launch_gate_stats_all(seer_ctx* ctx, const SeqMeta& m, void* ws, cudaStream_t stream) {
  const GateWs w(m, ws, SIZE_MAX);
  return launch_gate_stats(m, (const uint16_t*)w.gq, (const uint16_t*)w.gk, w.stats, ctx->d_status, stream);
}

int launch_gate_scores_band(seer_ctx* ctx, const SeqMeta& m, const ScoreBand& band, void* ws, float* scores, bool with_stats,
                            cudaStream_t stream) {
  const GateWs w(m, ws, SIZE_MAX);
  return launch_gate_scores(m, band, (const uint16_t*)w.gq, (const uint16_t*)w.gk, scores, with_stats ? w.stats : nullptr, ctx->d_status,
                            ctx->num_sms, stream);
}

int launch_gate_logits_band(seer_ctx* ctx, const SeqMeta& m, const ScoreBand& band, void* ws, float* logits, cudaStream_t stream) {
  const GateWs w(m, ws, SIZE_MAX);
  return launch_gate_logits(m, band, (const uint16_t*)w.gq, (const uint16_t*)w.gk, logits, w.stats, ctx->d_status, ctx->num_sms, stream);
}

const float2* gate_stats(const SeqMeta& m, void* ws) { return GateWs(m, ws, SIZE_MAX).stats; }

// ----------------------------------------------------------------------------------------------- allocation-free variant
// Scratch for seer_gate_scores_static lives in the library image: every GPU that loads the library carries these
// bytes until the process exits.  Host code must never hand the symbol itself to a kernel; its device address is
// looked up once per device with cudaGetSymbolAddress.
constexpr int kStaticMaxBatch = SEER_STATIC_MAX_BATCH;
constexpr size_t kStaticMetaBytes = 16 * 1024;                              // cu_seqlens and the two offset arrays (block, score)
constexpr size_t kStaticScratchBytes = (size_t)SEER_STATIC_SCRATCH_BYTES;   // projected pooled Q and K, three bf16 planes each (768 B per (head, block))
static __device__ __align__(256) unsigned char g_static_scratch[kStaticMetaBytes + kStaticScratchBytes];

constexpr int kStaticMaxDevices = 64;
static std::mutex g_static_mutex;
static void* g_static_addr[kStaticMaxDevices];     // device address of g_static_scratch, per device ordinal
static bool g_static_ready[kStaticMaxDevices];

// Once per device, with that device current: resolve the array's device address and lift the score kernels'
// shared-memory limit.  Neither call allocates.
static seer_status static_setup(int dev, unsigned char** out) {
  std::lock_guard<std::mutex> lock(g_static_mutex);
  if (!g_static_ready[dev]) {
    void* ptr = nullptr;
    if (cudaGetSymbolAddress(&ptr, g_static_scratch) != cudaSuccess || ptr == nullptr) return SEER_ERR_CUDA;
    if (!init_gate_scores()) return SEER_ERR_CUDA;
    g_static_addr[dev] = ptr;
    g_static_ready[dev] = true;
  }
  *out = (unsigned char*)g_static_addr[dev];
  return SEER_OK;
}

seer_status gate_scores_static(const seer_shape* shape, const void* q, const void* k, const float* Wq, const float* Wk,
                               float* scores, cudaStream_t stream) {
  ShapeTotals t;
  seer_status st = shape_totals(shape, &t);
  if (st != SEER_OK) return st;
  if (shape->cu_seqlens_q_host) return SEER_ERR_UNSUPPORTED;   // no chunked prefill through the built-in scratch
  if (t.total_blocks == 0) return SEER_OK;
  if (!q || !k || !Wq || !Wk || !scores) return SEER_ERR_INVALID_ARG;
  // sizes beyond the built-in scratch are refused, never truncated
  if (shape->batch > kStaticMaxBatch || gate_workspace_bytes(t, shape) > kStaticScratchBytes) return SEER_ERR_WORKSPACE;
  if (!on_16(q, k)) return SEER_ERR_CUDA;
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kStaticMaxDevices) return SEER_ERR_CUDA;
  unsigned char* base = nullptr;
  st = static_setup(dev, &base);
  if (st != SEER_OK) return st;

  // per-batch offsets, built in a host staging area that lives as long as the library (one per device, so that the
  // copy below never refers to a stack frame that has gone) and copied into the head of the array
  struct HostMeta {
    int32_t cu[kStaticMaxBatch + 4], blk[kStaticMaxBatch + 4];
    int64_t score[kStaticMaxBatch + 2];
  };
  static_assert(sizeof(HostMeta) <= kStaticMetaBytes, "metadata region too small");
  static HostMeta g_host_meta[kStaticMaxDevices];
  std::lock_guard<std::mutex> lock(g_static_mutex);   // (static_setup has released it)
  HostMeta& hm = g_host_meta[dev];
  hm.blk[0] = 0;
  hm.score[0] = 0;
  for (int b = 0; b < shape->batch; ++b) {
    hm.cu[b] = shape->cu_seqlens_host[b];
    const int32_t nb = (shape->cu_seqlens_host[b + 1] - shape->cu_seqlens_host[b] + shape->block - 1) / shape->block;
    hm.blk[b + 1] = hm.blk[b] + nb;
    hm.score[b + 1] = hm.score[b] + (int64_t)shape->num_q_heads * nb * nb;
  }
  hm.cu[shape->batch] = shape->cu_seqlens_host[shape->batch];
  // pageable source: the runtime stages the bytes before returning, so the next call may refill the staging area
  if (cudaMemcpyAsync(base, &hm, sizeof(HostMeta), cudaMemcpyHostToDevice, stream) != cudaSuccess) return SEER_ERR_CUDA;

  SeqMeta m;
  m.cu_seqlens = (const int32_t*)(base + offsetof(HostMeta, cu));
  m.blk_off = (const int32_t*)(base + offsetof(HostMeta, blk));
  m.score_off = (const int64_t*)(base + offsetof(HostMeta, score));
  m.batch = shape->batch;
  m.num_q_heads = shape->num_q_heads;
  m.num_kv_heads = shape->num_kv_heads;
  m.group = shape->num_q_heads / shape->num_kv_heads;
  m.total_tokens = (int32_t)t.total_tokens;
  m.total_blocks = (int32_t)t.total_blocks;
  m.max_nb = t.max_nb;
  m.rows = t.rows;
  m.score_elems = t.score_elems;
  m.softmax_scale = 0.f;   // unused by the gate
  m.block = shape->block;
  m.qoff = nullptr; m.qdelta = nullptr; m.qblk_off = nullptr; m.place = nullptr; m.chunked = 0; m.q_rows = t.rows;
  m.total_q_tokens = (int32_t)t.total_tokens;
  m.wait_limit_us = 0u; m.lose_v_copy = -1;   // unused by the gate
  m.score_tiles = 0; m.first_q_block = 0;
  // The kernels of seer_gate_scores without room for the statistics (pooling, then scores by one launch); only the scratch pointer
  // differs.  Nothing in the scratch has to start at zero: the first kernel writes every projected vector the second one reads.
  const int n = launch_gate(nullptr, m, q, k, Wq, Wk, scores, base + kStaticMetaBytes, kStaticScratchBytes, stream);
  return n < 0 ? SEER_ERR_CUDA : SEER_OK;
}

seer_status init_gate(seer_ctx* ctx) {
  (void)ctx;
  return init_gate_scores() ? SEER_OK : SEER_ERR_CUDA;
}

}  // namespace seer

extern "C" seer_status seer_gate_scores_static(const seer_shape* shape, const void* q, const void* k, const float* Wq,
                                               const float* Wk, float* scores, void* stream) {
  if (!shape) return SEER_ERR_INVALID_ARG;
  return seer::gate_scores_static(shape, q, k, Wq, Wk, scores, (cudaStream_t)stream);
}
