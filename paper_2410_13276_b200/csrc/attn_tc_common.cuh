// Pieces shared by the tcgen05 kernels of the attention and of the gate's scores: PTX wrappers (mbarrier, TMA, tcgen05, named barriers),
// shared-memory matrix descriptors, the work-item decoder and the optional cycle accounting.
#pragma once

#include <cuda.h>
#include <math_constants.h>

#include "seer_internal.cuh"

namespace seer {
namespace tcc {


// ------------------------------------------------------------------------------------------------ PTX wrappers
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
               : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
  return ok != 0;
}


struct Shared {
  uint32_t base;         // 1024-aligned shared address
  uint32_t bar0;         // shared address of mbarrier 0
  uint32_t abort_addr;   // shared address of the abort flag
  uint32_t limit_us;     // a wait that lasts this long is declared lost (2 s unless a test shortens it)
  __device__ __forceinline__ uint32_t bar(int i) const { return bar0 + 8u * (uint32_t)i; }
  __device__ __forceinline__ uint32_t abort_flag() const { return abort_addr; }
};

__device__ __forceinline__ uint32_t ld_shared_u32(uint32_t a) {
  uint32_t v;
  asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ void st_shared_u32(uint32_t a, uint32_t v) {
  asm volatile("st.shared.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}

__device__ __forceinline__ void st_shared_v2(uint32_t a, uint32_t x, uint32_t y) {
  asm volatile("st.shared.v2.u32 [%0], {%1,%2};" ::"r"(a), "r"(x), "r"(y) : "memory");
}
__device__ __forceinline__ void st_shared_v4(uint32_t a, uint32_t x, uint32_t y, uint32_t z, uint32_t w) {
  asm volatile("st.shared.v4.u32 [%0], {%1,%2,%3,%4};" ::"r"(a), "r"(x), "r"(y), "r"(z), "r"(w) : "memory");
}
__device__ __forceinline__ uint4 ld_shared_v4(uint32_t a) {
  uint4 v;
  asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ float ld_shared_f32(uint32_t a) { return __uint_as_float(ld_shared_u32(a)); }
__device__ __forceinline__ float4 ld_shared_f4(uint32_t a) {
  const uint4 v = ld_shared_v4(a);
  return make_float4(__uint_as_float(v.x), __uint_as_float(v.y), __uint_as_float(v.z), __uint_as_float(v.w));
}

__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// Bounded wait.  Returns false after the limit (or when another role has already given up); the caller drains.
__device__ __forceinline__ bool mbar_wait(const Shared& sh, int bar, uint32_t parity, int* status) {
  const uint32_t addr = sh.bar(bar);
  {
    uint32_t done;
    asm volatile("{\n\t.reg .pred p;\n\tmbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(done) : "r"(addr), "r"(parity) : "memory");
    if (done) return true;
  }
  if (mbar_try(addr, parity)) return true;
  const unsigned long long t0 = global_ns();
  for (uint32_t it = 1;; ++it) {
    if (mbar_try(addr, parity)) return true;
    if ((it & 255u) == 0u) {
      if (ld_shared_u32(sh.abort_flag()) != 0u) return false;
      if (global_ns() - t0 > (unsigned long long)sh.limit_us * 1000ull) break;
    }
  }
  st_shared_u32(sh.abort_flag(), 1u);
  atomicCAS(status, 0, (int)SEER_ERR_TIMEOUT);
  return false;
}

// The same by a converged warp; the outcome is the warp's, from one vote where the phase is complete.
__device__ __forceinline__ bool mbar_wait_warp(const Shared& sh, int bar, uint32_t parity, int* status) {
  uint32_t done;
  asm volatile("{\n\t.reg .pred p, q;\n\tmbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\tvote.sync.all.pred q, p, 0xffffffff;\n\tselp.u32 %0, 1, 0, q;\n\t}"
               : "=r"(done) : "r"(sh.bar(bar)), "r"(parity) : "memory");
  if (done) return true;
  return __all_sync(0xffffffffu, mbar_wait(sh, bar, parity, status));
}

__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap* map, uint32_t bar, int c0, int c1, int c2) {
  asm volatile("cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], [%2];"
               ::"r"(dst), "l"(map), "r"(bar), "r"(c0), "r"(c1), "r"(c2) : "memory");
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// True in one lane of a converged warp.  A thread that issues tcgen05.mma must be picked by this instruction inside a
// warp-uniform branch: the operands of the MMA live in uniform registers, and behind an ordinary condition (lane == 0) the
// compiler cannot know that a single thread is active and wraps every MMA in a loop over the active threads.  Measured,
// one issuing thread, M 128 N 64 K 16 from shared memory: 57 clocks per MMA instead of 89 (the pipe's own limit is 48).
__device__ __forceinline__ bool elect_one() {
  uint32_t r;
  asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(r));
  return r != 0;
}

__device__ __forceinline__ void tc_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
// A from tensor memory (lane = row, two bf16 per column)
__device__ __forceinline__ void tc_mma_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc, uint32_t accumulate) {
  asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
               "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
               ::"r"(d_tmem), "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate) : "memory");
}
// A from shared memory
__device__ __forceinline__ void tc_mma_ss(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, uint32_t accumulate) {
  asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
               "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
               ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate) : "memory");
}
// Weight-stationary form, A from shared memory / from tensor memory (M = 64: see attn_tc.cu)
__device__ __forceinline__ void tc_mma_ws(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, uint32_t accumulate) {
  asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
               "tcgen05.mma.ws.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
               ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate) : "memory");
}
__device__ __forceinline__ void tc_mma_ws_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc, uint32_t accumulate) {
  asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
               "tcgen05.mma.ws.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
               ::"r"(d_tmem), "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate) : "memory");
}
__device__ __forceinline__ void tc_ld16(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
                 "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
               : "r"(taddr) : "memory");
}
__device__ __forceinline__ void tc_ld32(uint32_t taddr, uint32_t (&r)[32]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
                 "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
                 "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
                 "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
               : "r"(taddr) : "memory");
}
// Waits for the loads of this thread; the loaded registers are in/out operands so that no use of them moves above it.
__device__ __forceinline__ void tc_wait_ld32(uint32_t (&r)[32]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                 "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15]),
                 "+r"(r[16]), "+r"(r[17]), "+r"(r[18]), "+r"(r[19]), "+r"(r[20]), "+r"(r[21]), "+r"(r[22]), "+r"(r[23]),
                 "+r"(r[24]), "+r"(r[25]), "+r"(r[26]), "+r"(r[27]), "+r"(r[28]), "+r"(r[29]), "+r"(r[30]), "+r"(r[31])
               :: "memory");
}
__device__ __forceinline__ void tc_st16(uint32_t taddr, const uint32_t (&r)[16]) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};"
               ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),
                 "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]) : "memory");
}
__device__ __forceinline__ void tc_st32(uint32_t taddr, const uint32_t (&r)[32]) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32};"
               ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),
                 "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]),
                 "r"(r[16]), "r"(r[17]), "r"(r[18]), "r"(r[19]), "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]),
                 "r"(r[24]), "r"(r[25]), "r"(r[26]), "r"(r[27]), "r"(r[28]), "r"(r[29]), "r"(r[30]), "r"(r[31]) : "memory");
}
// Same wait, with the loaded registers as in/out operands so that no use of them can be scheduled above it.
__device__ __forceinline__ void tc_wait_ld(uint32_t (&r)[16]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                 "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15])
               :: "memory");
}
__device__ __forceinline__ void tc_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

__device__ __forceinline__ void named_bar_sync(int id, int threads) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
// CTA-subset OR reduction of a predicate over `threads` threads on barrier `id`
__device__ __forceinline__ bool named_bar_or(int id, int threads, bool pred) {
  uint32_t r;
  asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.u32 p, %3, 0;\n\tbar.red.or.pred q, %1, %2, p;\n\tselp.u32 %0, 1, 0, q;\n\t}"
               : "=r"(r) : "r"(id), "r"(threads), "r"((uint32_t)pred) : "memory");
  return r != 0;
}

// Shared-memory matrix descriptors (128-byte swizzle, descriptor version 1)
__device__ __forceinline__ uint64_t make_desc(uint32_t saddr, uint32_t lbo_bytes, uint32_t sbo_bytes) {
  return (uint64_t)((saddr & 0x3ffffu) >> 4) | ((uint64_t)(lbo_bytes >> 4) << 16) | ((uint64_t)(sbo_bytes >> 4) << 32) |
         (1ull << 46) | (2ull << 61);
}

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  uint32_t r;
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
  return r;
}
__device__ __forceinline__ float ex2f(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

struct Item {
  int h, g, i, nb, s0, slen, l0, nlist, ntiles, q_valid, dq;
  int64_t row;
};

// kChunk: chunked prefill.  q / o / lse hold the last positions of each sequence only: their token index is the k / v
// token index plus dq.  Query blocks before the chunk have nothing to do whatever their lists say, and no work item is counted for
// them: a stream takes about a microsecond to draw one, look it up and drop it (917 queries against 60k tokens: 29 888 items
// for 512 of work, 163 us and 67 so).
//
// kPlaced: the sequences in the order of SeqMeta::place; otherwise (never with kChunk) in the batch's: the block maxima of whole prompts, whose
// static deal gives a CTA the longest list of every round if they come longest first (1965 and 815 tokens, 8 heads: 14.6 us, 18.5 so).
template <bool kChunk, bool kPlaced>
__device__ __forceinline__ Item decode_item(const SeqMeta& m, const int32_t* row_ptr, int64_t w) {
  static_assert(kPlaced || !kChunk, "blk_off counts the blocks before a chunk too");
  Item it;
  const int32_t* off = kPlaced ? m.qblk_off : m.blk_off;
  const int p = find_sequence(off, m.batch, (int)(w / m.num_q_heads)), before = off[p];
  int blk0, nq;                                            // first block of the sequence, blocks with queries (its last ones)
  if (kPlaced) {
    const int4 s = m.place[p];
    it.s0 = s.x; it.slen = s.y; blk0 = s.z; it.dq = kChunk ? s.w : 0;
    it.nb = (it.slen + kBlock - 1) / kBlock;
    nq = kChunk ? off[p + 1] - before : it.nb;
  } else {
    it.s0 = m.cu_seqlens[p];
    it.slen = m.cu_seqlens[p + 1] - it.s0;
    blk0 = before; it.dq = 0;
    it.nb = off[p + 1] - before;
    nq = it.nb;
  }
  const int local = (int)(w - (int64_t)m.num_q_heads * before);
  it.g = local / (nq * m.group);
  const int rem = local - it.g * nq * m.group;
  it.i = it.nb - 1 - rem / m.group;
  it.h = it.g * m.group + rem % m.group;
  it.row = (int64_t)m.num_q_heads * blk0 + (int64_t)it.h * it.nb + it.i;
  it.q_valid = min(kBlock, it.slen - it.i * kBlock);
  it.l0 = row_ptr[it.row];
  it.nlist = row_ptr[it.row + 1] - it.l0;
  it.ntiles = (it.nlist + 1) >> 1;
  return it;
}

// Optional cycle accounting of CTA 0 (diagnostics): every role attributes the clocks between two consecutive marks to the
// tag of the later mark and adds them, and the mark, to trace[role * 8192 + tag * 2 ...] (reductions: nothing is waited for).
template <bool ON>
struct Tracer {
  unsigned long long* p;      // global destination (nullptr: off)
  long long last;
  bool on;
  // Only every 8th tile is timed, so that the bookkeeping does not distort what it measures.
  __device__ __forceinline__ void sample(uint32_t ordinal) {
    const bool was = on;
    on = p != nullptr && (ordinal & 7u) == 0u;
    if (on && !was) last = clock64();
  }
  __device__ __forceinline__ void init(unsigned long long* base, int role) {
    p = (base != nullptr && blockIdx.x == 0) ? base + (size_t)role * 8192 : nullptr;
    last = 0;
    on = false;
  }
  __device__ __forceinline__ void ev(uint32_t tag) {
    if (on) {
      const long long now = clock64();
      asm volatile("red.global.add.u64 [%0], %1;" ::"l"(p + 2 * tag), "l"((unsigned long long)(now - last)) : "memory");
      asm volatile("red.global.add.u64 [%0], %1;" ::"l"(p + 2 * tag + 1), "l"(1ull) : "memory");
      last = clock64();
    }
  }
};
template <>
struct Tracer<false> {   // the production instantiation carries no state and no code
  __device__ __forceinline__ void sample(uint32_t) {}
  __device__ __forceinline__ void init(unsigned long long*, int) {}
  __device__ __forceinline__ void ev(uint32_t) {}
};

// kind::f16 instruction descriptor: fp32 accumulate, bf16 x bf16
constexpr uint32_t make_idesc(bool a_mn_major, bool b_mn_major, uint32_t n = 64u, uint32_t m = 128u) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((a_mn_major ? 1u : 0u) << 15) | ((b_mn_major ? 1u : 0u) << 16) |
         ((n >> 3) << 17) | ((m >> 4) << 24);
}

// ------------------------------------------------------------------------------------------------ softmax of the attention
constexpr float kNoRef = -1e30f;   // reference of a row that has not seen a live block
// A tile whose row sum reaches this moves the row's reference: 2^60 above the first block's maximum, far from the 2^127 at
// which P or the sums would overflow, and far above what a prompt's sink or stripes rise (a move costs about two tiles).
constexpr float kRise = 1.152921504606847e18f;   // 2^60
// of every eight pairs of a pass this many take their exponentials on the FMA pipe (0, 1 and 3 measured within 2 % of it)
constexpr int kPolyPairsOf8 = 2;

__device__ __forceinline__ bool mbar_test(uint32_t addr, uint32_t parity) {
  uint32_t done;
  asm volatile("{\n\t.reg .pred p;\n\tmbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
               : "=r"(done) : "r"(addr), "r"(parity) : "memory");
  return done != 0;
}

// 2^x for two values at once on the FMA pipe (the special-function unit does 16 exponentials per clock and SM): x = n + f
// with n = round(x), 2^f by a cubic (relative error 7.5e-5, far below the bf16 rounding of P), 2^n by adding n to the
// exponent field.  x is clamped to [-125, 128] so that the exponent field stays in 1..255: below gives ~2^-125, above
// something no smaller than 2^127, which the caller's test of the sum sees; so does a NaN, which the clamp lets through.
__device__ __forceinline__ float clamp_nan(float x) {
  float y;
  asm("max.NaN.f32 %0, %1, 0fC2FA0000;" : "=f"(y) : "f"(x));   // -125
  asm("min.NaN.f32 %0, %1, 0f43000000;" : "=f"(x) : "f"(y));   // 128
  return x;
}
__device__ __forceinline__ float2 exp2_poly2(float2 x) {
  x.x = clamp_nan(x.x); x.y = clamp_nan(x.y);
  const float2 magic = make_float2(12582912.f, 12582912.f);        // 1.5 * 2^23: the sum's low mantissa bits are round(x)
  const float2 t = __fadd2_rn(x, magic);
  const float2 n = __fadd2_rn(t, make_float2(-12582912.f, -12582912.f));
  const float2 f = __fadd2_rn(x, make_float2(-n.x, -n.y));         // in [-0.5, 0.5]
  float2 r = __ffma2_rn(make_float2(0.05517168343067169f, 0.05517168343067169f), f, make_float2(0.2426111251115799f, 0.2426111251115799f));
  r = __ffma2_rn(r, f, make_float2(0.6932609677314758f, 0.6932609677314758f));
  r = __ffma2_rn(r, f, make_float2(0.9999280571937561f, 0.9999280571937561f));
  r.x = __int_as_float(__float_as_int(r.x) + (__float_as_int(t.x) << 23));
  r.y = __int_as_float(__float_as_int(r.y) + (__float_as_int(t.y) << 23));
  return r;
}

// One pass over this thread's row of a 64 x 64 block of scores: p = 2^(sl2 * s - R), packed to bf16 pairs in pk; returns the
// sum of the row.  kPolyPairsOf8 of every eight pairs take their exponentials on the FMA pipe, the others on the
// special-function unit.  MASKED: the causal mask of the diagonal block (keys after `row` are dropped).  half(ch): the row's 32 keys from 32 ch on.
template <bool MASKED, class Half>
__device__ __forceinline__ float row_pass_of(Half half, float sl2, float R, int row, uint32_t (&pk)[32]) {
  const float2 sl22 = make_float2(sl2, sl2), nr = make_float2(-R, -R);
  float2 acc[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) acc[i] = make_float2(0.f, 0.f);
#pragma unroll
  for (int ch = 0; ch < 2; ++ch) {
    const uint32_t (&sv)[32] = half(ch);
    // stage by stage over the 32 keys, each stage a run of independent instructions, in place
    float2 v[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = __ffma2_rn(make_float2(__uint_as_float(sv[2 * i]), __uint_as_float(sv[2 * i + 1])), sl22, nr);
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      if ((i & 7) < kPolyPairsOf8) v[i] = exp2_poly2(v[i]);
      else v[i] = make_float2(ex2f(v[i].x), ex2f(v[i].y));
    }
    if (MASKED) {
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        const int c = ch * 32 + 2 * i;
        if (c > row) v[i].x = 0.f;
        if (c + 1 > row) v[i].y = 0.f;
      }
    }
#pragma unroll
    for (int i = 0; i < 16; ++i) pk[ch * 16 + i] = pack_bf16(v[i].x, v[i].y);
#pragma unroll
    for (int i = 0; i < 16; ++i) acc[i & 3] = __fadd2_rn(acc[i & 3], v[i]);
  }
  const float2 a = __fadd2_rn(__fadd2_rn(acc[0], acc[1]), __fadd2_rn(acc[2], acc[3]));
  return a.x + a.y;
}
// The row from tensor memory, in two round trips: the second half is requested before the first is worked on
template <bool MASKED>
__device__ __forceinline__ float row_pass(uint32_t s_addr, float sl2, float R, int row, uint32_t (&pk)[32]) {
  uint32_t sv[2][32];
  tc_ld32(s_addr, sv[0]);
  return row_pass_of<MASKED>([&](int ch) -> const uint32_t (&)[32] {
    tc_wait_ld32(sv[ch]);
    if (ch == 0) tc_ld32(s_addr + 32, sv[1]);
    return sv[ch];
  }, sl2, R, row, pk);
}
// The largest raw score of this thread's row (MASKED: among the keys it sees, key <= last; -inf if there is none).
// Off the diagonal the 64 predicates are left out (with them a 128k prompt takes 2 % longer).
template <bool MASKED>
__device__ __forceinline__ float row_max(uint32_t s_addr, int last) {
  float mx[4] = {-CUDART_INF_F, -CUDART_INF_F, -CUDART_INF_F, -CUDART_INF_F};
  uint32_t sv[2][32];
  tc_ld32(s_addr, sv[0]);
  tc_ld32(s_addr + 32, sv[1]);
  tc_wait_ld32(sv[0]);
  tc_wait_ld32(sv[1]);
#pragma unroll
  for (int ch = 0; ch < 2; ++ch)
#pragma unroll
    for (int e = 0; e < 32; ++e)
      if (!MASKED || ch * 32 + e <= last) mx[e & 3] = fmaxf(mx[e & 3], __uint_as_float(sv[ch][e]));
  return fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3]));
}

// A tile where some row's reference has to move; by pairs also the diagonal block (last = row) and one that is not this row's (last < 0); from the scores
// to P in their place.  `fresh`: the row has no reference yet.  Returns the row's (reference, sum) and whether a wait was lost.  Conditions around
// tensor memory loads are the same for a whole warp: all its lanes take part in them.
// A function of its own, not inlined: the plain pass would pay for sharing its registers (attn_tc.cu).
static __device__ __noinline__ float4 other_tile(Shared sh, uint32_t s_addr, uint32_t o_addr, float sl2, float R, float l, int last, bool fresh, int t, int pv_bar, uint32_t pv_par, int* status) {
  uint32_t pk[32];
  if (last < 0) {                                           // contributes nothing
#pragma unroll
    for (int i = 0; i < 32; ++i) pk[i] = 0u;
  } else {
    float sum = 0.f;
    bool over = false;
    for (int taken = 0;; taken = 1) {
      uint32_t sv[2][32];
      tc_ld32(s_addr, sv[0]);
      tc_ld32(s_addr + 32, sv[1]);
      tc_wait_ld32(sv[0]);
      tc_wait_ld32(sv[1]);
      if (taken || fresh) {                                 // (the same for the whole warp)
        float mx4[4] = {-CUDART_INF_F, -CUDART_INF_F, -CUDART_INF_F, -CUDART_INF_F};
#pragma unroll
        for (int c = 0; c < 64; ++c)
          if (c <= last) mx4[c & 3] = fmaxf(mx4[c & 3], __uint_as_float(sv[c >> 5][c & 31]));
        const float raw = fmaxf(fmaxf(mx4[0], mx4[1]), fmaxf(mx4[2], mx4[3]));
        if (!taken) {
          if (fabsf(raw) < 3.0e38f) R = raw * sl2;
        } else {
          const float mx = raw * sl2;
          const float nr = over && fabsf(mx) < 3.0e38f ? fmaxf(R, mx) : R;
          const float alpha = nr == R ? 1.f : exp2f(R - nr);
          R = nr;
          l = alpha == 0.f ? 0.f : __fmul_rn(l, alpha);
          if (t > 0) {
#pragma unroll 1
            for (int ch = 0; ch < 8; ++ch) {
              uint32_t ov[16];
              tc_ld16(o_addr + ch * 16, ov);
              tc_wait_ld(ov);
#pragma unroll
              for (int e = 0; e < 16; ++e) ov[e] = alpha == 0.f ? 0u : __float_as_uint(__uint_as_float(ov[e]) * alpha);
              tc_st16(o_addr + ch * 16, ov);
            }
          }
        }
      }
      sum = row_pass_of<true>([&](int ch) -> const uint32_t (&)[32] { return sv[ch]; }, sl2, R, last, pk);
      if (taken) {
        if (!(sum < kRise)) sum = CUDART_NAN_F;             // an infinite score or a NaN: so is the row
        break;
      }
      over = !(sum < kRise);
      if (!__any_sync(0xffffffffu, over)) break;
      // ---- some row's reference has to move (or its scores are not finite): O at rest, rows rescaled, tile taken again
      if (t > 0) {
        const bool fail = !mbar_wait(sh, pv_bar, pv_par, status);
        if (__any_sync(0xffffffffu, fail)) return make_float4(R, l, 1.f, 0.f);
        tc_fence_after();
      }
    }
    l = __fadd_rn(l, sum);
  }
  tc_st32(s_addr, pk);                                      // P over the scores this thread has read
  tc_wait_st();
  tc_fence_before();
  return make_float4(R, l, 0.f, 0.f);
}

// 32 bytes, at once where the address allows it (the host asks for 16)
__device__ __forceinline__ void st_global_32(void* p, const uint32_t (&w)[8], bool aligned) {
  if (!aligned) {
    reinterpret_cast<uint4*>(p)[0] = make_uint4(w[0], w[1], w[2], w[3]);
    reinterpret_cast<uint4*>(p)[1] = make_uint4(w[4], w[5], w[6], w[7]);
    return;
  }
  asm volatile("st.global.v8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"l"(p), "r"(w[0]), "r"(w[1]), "r"(w[2]), "r"(w[3]), "r"(w[4]),
               "r"(w[5]), "r"(w[6]), "r"(w[7]) : "memory");
}

}  // namespace tcc

// Attention where pairs of query blocks list the same blocks (attn_pair.cu).  The check answers in `nwords` words, all of them written by every call: `epoch`
// in all of them where all pairs do.  attn_tc_kernel then returns at once, otherwise attn_pair_kernel.  (The words lie behind the counter in a workspace of 256 bytes or more.)
struct PairAnswer {
  int* words;
  int nwords, epoch;
  PairAnswer(const seer_ctx* ctx, const SeqMeta& m, int* at) : words(at), nwords((int)min((int64_t)kPairWords, m.pair_units)), epoch(1 + (int)(ctx->clock & 0x3fffffff)) {}
};
int launch_pair_check(seer_ctx* ctx, const SeqMeta& m, const int32_t* row_ptr, const int32_t* col_idx, int* counter, const PairAnswer& a, cudaStream_t stream);
int launch_attn_pair(seer_ctx* ctx, const SeqMeta& m, const CUtensorMap& mq, const CUtensorMap& mk, const CUtensorMap& mv, const CUtensorMap& mv32, const int32_t* row_ptr,
                     const int32_t* col_idx, void* o, float* lse, int* counter, const PairAnswer& a, cudaStream_t stream);

}  // namespace seer
