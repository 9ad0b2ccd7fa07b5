// Block-sparse causal attention (Sec. 3.3) where query blocks 2u and 2u + 1 of every head list the same blocks, up to the second one's own:
// gate blocks of 128 tokens, and dense lists.  A work item is the two blocks, 128 query rows that share every K and V tile.
//
// attn_tc_kernel has an item's 64 rows on both halves of tensor memory's lanes, the even list positions on one and the odd ones on the
// other, and 64 KB of K and V come from L2 for each pair of listed blocks: 885 clocks of the 960 that they take.  Here the lane
// half is the query block, and the even and the odd positions belong to two softmax groups with an S, P and O of their own:
//     S[128 q x 128 keys] = Q (smem) * [K_a; K_b]^T      M = N = 128: columns 0-63 are the even position's scores, 64-127 the odd one's
//     O_0 += P_a V_a, O_1 += P_b V_b                     M = N = 128, A = P in tensor memory
// so a tile's 64 KB serve four 64 x 64 blocks instead of two, and its 16 MMAs run at the full rate (1024 clocks for four blocks; the
// weight-stationary forms take 1376).  What every row is made of is the same, in the same order: the results equal attn_tc_kernel's bit for
// bit.  A launch by itself, on a cool board and under its power limit: 65 536 tokens, 32 heads, 128-token blocks, one in ten 3740 -> 3100 and 4180
// -> 3510 us; 16 384 tokens, every block 2190 -> 1850 and 2356 -> 2082.
//
// What bounds it: the power limit in launches of milliseconds; under it the groups, 1400 to 1500 clocks a tile (the pass 1100, with two warps
// a scheduler that begin it together), and an item's end, 1000 to 2500 clocks until the last P V and 2300 for merge and stores, which both
// groups reach together.  Tried: S in one buffer, given back as soon as it is in registers, so that the next tile's comes during the pass (3370 us
// where this takes 3150, the pass then keeps 64 more registers for rows whose reference moves); S and P V from two issuing threads (3400: their
// chains of waits add up); this body inside attn_tc_kernel instead of a launch of its own (5200, and the other kernel 2 % slower); one K or V
// barrier for each half of a tile (the issuer, one thread, is busy 1100 clocks a tile with its waits and commits).
//
// Roles (384 threads): warp 0 producer of Q and K, draws the items; warp 1 MMA issuer; warp 2 producer of V; warps 4-7 and 8-11 the groups.
#include "attn_pair.cuh"

namespace seer {
namespace tp {

using namespace tcc;

constexpr int kThreads = 384;                    // four helper warps, two softmax groups of four
constexpr int kHelperRegs = 64, kSoftmaxRegs = 216;   // 128 * 64 + 256 * 216 <= 384 * 168
constexpr uint32_t kVBlock = 2 * kHalfTile;      // V of one block: [d half]
constexpr uint32_t kKUnits = 3, kVUnits = 2;
constexpr uint32_t kOffV = kOffK + kKUnits * kUnit;
constexpr uint32_t kOffMl = kOffV + kVUnits * kUnit;              // (reference, sum) of 2 x 128 rows
constexpr uint32_t kOffBar = kOffMl + 2048;
constexpr int kBars = 32;
constexpr uint32_t kOffRing = kOffBar + kBars * 8;                // four item slots of 64 bytes
constexpr uint32_t kOffMisc = kOffRing + 4 * 64;                  // tmem base, abort flag
constexpr uint32_t kSmemBytes = kOffMisc + 64;
static_assert(kSmemBytes <= 232448, "shared memory budget of one CTA");

enum Bar { Q_FULL = 0 /* + buf */, Q_EMPTY = 2, K_FULL = 4 /* + unit */, K_EMPTY = 7, V_FULL = 10, V_EMPTY = 12, S_FULL = 14 /* + buf */,
           P_FULL = 16 /* + 2 * group + buf */, PV_DONE = 20 /* + buf */, O_FREE = 22, ITEM_FULL = 23 /* + slot */, ITEM_EMPTY = 27, kBarsUsed = 31 };
static_assert(K_EMPTY == K_FULL + (int)kKUnits && V_EMPTY == V_FULL + (int)kVUnits && S_FULL == V_EMPTY + (int)kVUnits && kBarsUsed <= kBars, "barrier map");

constexpr uint32_t kTmemCols = 512;
// Tensor memory columns: two S buffers of two key blocks (group g's scores, then its P in the first 32 of them), O of each group
__device__ __forceinline__ uint32_t col_s(uint32_t buf, int g) { return buf * 128u + (uint32_t)g * 64u; }
__device__ __forceinline__ uint32_t col_o(int g) { return 256u + (uint32_t)g * 128u; }

constexpr uint32_t kIdescPV = make_idesc(false, true, 128u, 128u);
constexpr uint32_t kIdescLone = make_idesc(false, true, 256u, 64u);

// Whether every pair of query blocks has one list (pair_ok), answered block by block: words[block] becomes `epoch` where the block found its pairs
// so, else 0.  Also zeroes the attention's work counter.  A warp goes through its pairs by itself and leaves where one of its block's differs: where lists
// differ it finds out with the first, after three trips to L2.
constexpr int kCheckWarps = 32;
template <bool kChunk>
__global__ void __launch_bounds__(kCheckWarps * 32) check_kernel(SeqMeta m, const int32_t* row_ptr, const int32_t* col_idx, int* counter, int* words, int epoch) {
  __shared__ int differs;
  if (threadIdx.x == 0) differs = 0;
  __syncthreads();
  grid_wait();
  if (blockIdx.x == 0 && threadIdx.x == 0) *counter = 0;
  const int lane = threadIdx.x & 31;
  for (int64_t w = (int64_t)(threadIdx.x >> 5) * gridDim.x + blockIdx.x; w < m.pair_units; w += (int64_t)gridDim.x * kCheckWarps) {
    if (__any_sync(0xffffffffu, *(volatile int*)&differs != 0)) break;
    if (!pair_ok<kChunk>(m, row_ptr, reinterpret_cast<const uint32_t*>(col_idx), w, lane) && lane == 0) *(volatile int*)&differs = 1;
  }
  __syncthreads();
  if (threadIdx.x == 0) *(volatile int*)(words + blockIdx.x) = differs == 0 ? epoch : 0;
}

template <bool kChunk, bool kO32>
__global__ void __launch_bounds__(kThreads, 1)
attn_pair_kernel(const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_k, const __grid_constant__ CUtensorMap map_v,
                 const __grid_constant__ CUtensorMap map_v32, SeqMeta m, const int32_t* row_ptr, const int32_t* col_idx, uint16_t* __restrict__ o, float* lse, int* __restrict__ status,
                 int* __restrict__ work_counter, const int* words, int nwords, int epoch) {
  extern __shared__ __align__(1024) unsigned char smem[];
  Shared sh;
  sh.base = smem_u32(smem);
  sh.bar0 = sh.base + kOffBar;
  sh.abort_addr = sh.base + kOffMisc + 8;
  sh.limit_us = m.wait_limit_us;
  if ((sh.base & 1023u) != 0u) {                           // the swizzled tiles need the alignment
    grid_wait();
    if (threadIdx.x == 0) atomicCAS(status, 0, (int)SEER_ERR_CUDA);
    return;
  }
  grid_wait();
  if (!lists_agree(words, nwords, epoch)) return;           // attn_tc_kernel has done it
  const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
  volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(smem + kOffMisc);
  if (threadIdx.x == 0) {
    for (int i = 0; i < kBarsUsed; ++i) {
      // O_FREE: both groups' warps; P_FULL: a group's; ITEM_EMPTY: both groups', the V producer and the issuer
      const uint32_t count = i == O_FREE ? 8u : i >= P_FULL && i < P_FULL + 4 ? 4u : i >= ITEM_EMPTY && i < ITEM_EMPTY + 4 ? 10u : 1u;
      mbar_init(sh.bar(i), count);
    }
    st_shared_u32(sh.abort_flag(), 0u);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(sh.base + kOffMisc), "r"(kTmemCols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  auto ring_addr = [&](uint32_t n) -> uint32_t { return sh.base + kOffRing + (n & 3u) * 64u; };
  struct Slot {
    int h, i0, l0, len, n[2], tok0, s0, valid[2], first[2];
    int plain[2];                                           // entries before the block's diagonal, where that is listed, or all
    __device__ __forceinline__ int tiles() const { return (len + 1) >> 1; }
    // the last entry belongs to the second block alone, and its group's O has rows of the first: they must not see its V (0 * inf)
    __device__ __forceinline__ bool lone() const { return valid[0] > 0 && n[0] < len && len > 2; }
  };
  auto read_slot = [&](uint32_t n) -> Slot {
    const uint4 a = ld_shared_v4(ring_addr(n)), b = ld_shared_v4(ring_addr(n) + 16u), c = ld_shared_v4(ring_addr(n) + 32u), d = ld_shared_v4(ring_addr(n) + 48u);
    Slot it;
    it.h = (int)a.x; it.i0 = (int)a.y; it.l0 = (int)a.z; it.len = (int)a.w;
    it.n[0] = (int)b.x; it.n[1] = (int)b.y; it.tok0 = (int)b.z; it.s0 = (int)b.w;
    it.valid[0] = (int)c.x; it.valid[1] = (int)c.y; it.first[0] = (int)c.z; it.first[1] = (int)c.w;
    it.plain[0] = (int)d.x; it.plain[1] = (int)d.y;
    return it;
  };
  auto entry = [&](const Slot& it, int p) -> int { return p < it.len ? (int)ld_global(reinterpret_cast<const uint32_t*>(col_idx) + it.l0 + p) : -1; };

  if (warp < 4) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kHelperRegs));
    // ========================================================================================== producer of Q and K (TMA), draws the items
    if (warp == 0) {
      if (elect_one()) {
        uint32_t nitem = 0, ku = 0, kph = 0;
        bool ok = true, more = false;
        PairItem nx{};
        auto locate = [&](int64_t w) {
          more = w < m.pair_units;
          nx = PairItem{};
          if (more) nx = decode_pair<kChunk>(m, row_ptr, w);
        };
        auto announce = [&](uint32_t n) -> bool {
          const int e0 = 0 < nx.len ? (int)ld_global(reinterpret_cast<const uint32_t*>(col_idx) + nx.l0) : -1;
          const int e1 = 1 < nx.len ? (int)ld_global(reinterpret_cast<const uint32_t*>(col_idx) + nx.l0 + 1) : -1;
          const int x0 = nx.n[0] > 0 ? (int)ld_global(reinterpret_cast<const uint32_t*>(col_idx) + nx.l0 + nx.n[0] - 1) : -1;
          const int x1 = nx.n[1] > 0 ? (int)ld_global(reinterpret_cast<const uint32_t*>(col_idx) + nx.l0 + nx.n[1] - 1) : -1;
          if (!mbar_wait(sh, ITEM_EMPTY + (int)(n & 3u), ((n >> 2) & 1u) ^ 1u, status)) return false;
          st_shared_v4(ring_addr(n) + 48u, (uint32_t)(nx.n[0] - (x0 == nx.i0)), (uint32_t)(nx.n[1] - (x1 == nx.i0 + 1)), 0u, 0u);
          st_shared_v4(ring_addr(n), (uint32_t)nx.h, (uint32_t)nx.i0, (uint32_t)nx.l0, more ? (uint32_t)nx.len : 0xffffffffu);
          st_shared_v4(ring_addr(n) + 16u, (uint32_t)nx.n[0], (uint32_t)nx.n[1], (uint32_t)nx.tok0, (uint32_t)nx.s0);
          st_shared_v4(ring_addr(n) + 32u, (uint32_t)nx.valid[0], (uint32_t)nx.valid[1], (uint32_t)e0, (uint32_t)e1);
          mbar_arrive(sh.bar(ITEM_FULL + (int)(n & 3u)));
          return true;
        };
        locate((int64_t)atomicAdd(work_counter, 1));
        ok = announce(0);
        for (uint32_t n = 0; ok; ++n) {
          const Slot it = read_slot(n);                    // (its own announcement)
          if (it.len < 0) break;
          int ja = it.first[0], jb = it.first[1];
          const int64_t w = (int64_t)atomicAdd(work_counter, 1);
          const int tiles = it.tiles(), g = it.h / m.group;
          if (tiles == 0) { locate(w); ok = announce(n + 1); continue; }
          const uint32_t qb = nitem & 1u, qf = sh.bar(Q_FULL + (int)qb);
          if (!mbar_wait(sh, Q_EMPTY + (int)qb, ((nitem >> 1) & 1u) ^ 1u, status)) break;
          mbar_expect_tx(qf, it.valid[0] > 0 && it.valid[1] > 0 ? kQBytes : kQBytes / 2);
#pragma unroll
          for (int half = 0; half < 2; ++half)
            if (it.valid[half] > 0)
#pragma unroll
              for (int dh = 0; dh < 2; ++dh)
                tma_load_3d(sh.base + kOffQ + qb * kQBytes + (uint32_t)(2 * dh + half) * kHalfTile, &map_q, qf, 64 * dh, it.h, it.tok0 + 64 * half);
          ++nitem;
          for (int t = 0; t < tiles; ++t) {
            const int ra = entry(it, 2 * t + 2), rb = entry(it, 2 * t + 3);   // next pair
            const bool has_b = jb >= 0;
            const int ta = it.s0 + ja * kBlock, tb = it.s0 + jb * kBlock;
            if (!mbar_wait(sh, K_EMPTY + (int)ku, kph ^ 1u, status)) { ok = false; break; }
            const uint32_t fb = sh.bar(K_FULL + (int)ku), dst = sh.base + kOffK + ku * kUnit;
            mbar_expect_tx(fb, has_b ? kUnit : kUnit / 2);
#pragma unroll
            for (int dh = 0; dh < 2; ++dh) {
              tma_load_3d(dst + (uint32_t)dh * 2 * kHalfTile, &map_k, fb, 64 * dh, g, ta);
              if (has_b) tma_load_3d(dst + (uint32_t)dh * 2 * kHalfTile + kHalfTile, &map_k, fb, 64 * dh, g, tb);
            }
            if (++ku == kKUnits) { ku = 0; kph ^= 1u; }
            ja = ra; jb = rb;
            if (t == 0) locate(w);
            if (t == min(1, tiles - 1) && !announce(n + 1)) { ok = false; break; }
          }
        }
      }
    }
    // ========================================================================================== producer of V (TMA)
    else if (warp == 2) {
      if (elect_one()) {
        uint32_t vu = 0, vph = 0, cnt = 0;
        bool ok = true;
        for (uint32_t n = 0; ok; ++n) {
          if (!mbar_wait(sh, ITEM_FULL + (int)(n & 3u), (n >> 2) & 1u, status)) break;
          const Slot it = read_slot(n);
          mbar_arrive(sh.bar(ITEM_EMPTY + (int)(n & 3u)));
          if (it.len < 0) break;
          const int g = it.h / m.group;
          int j0 = it.first[0], j1 = it.first[1];
          for (int p = 0; p < it.len && ok; p += 2) {
            const int ra = entry(it, p + 2), rb = entry(it, p + 3);   // next pair
            const int last = it.len - 1 - p;                // the tile's position that is the list's last: 0, 1 or beyond
            const bool lone = last < 2 && it.lone();
            const int whole = lone ? last : min(last + 1, 2);   // blocks for both query blocks
            const int ta = it.s0 + j0 * kBlock, tb = it.s0 + j1 * kBlock;
            if (whole > 0) {
              if (!mbar_wait(sh, V_EMPTY + (int)vu, vph ^ 1u, status)) { ok = false; break; }
              const uint32_t fb = sh.bar(V_FULL + (int)vu), dst = sh.base + kOffV + vu * kUnit;
              // test hook: one V copy that is never issued, so that the issuer's wait for it runs out
              if (blockIdx.x != 0 || m.lose_v_copy < 0 || cnt != (uint32_t)m.lose_v_copy) {
                mbar_expect_tx(fb, (uint32_t)whole * kVBlock);
                tma_load_3d(dst, &map_v, fb, 0, g, ta);
                tma_load_3d(dst + kHalfTile, &map_v, fb, 64, g, ta);
                if (whole > 1) {
                  tma_load_3d(dst + kVBlock, &map_v, fb, 0, g, tb);
                  tma_load_3d(dst + kVBlock + kHalfTile, &map_v, fb, 64, g, tb);
                }
              }
              if (++vu == kVUnits) { vu = 0; vph ^= 1u; }
            }
            if (lone) {
              // [0 | V] by key halves: zeros, which a copy from past the last token brings, for the first block's rows
              if (!mbar_wait(sh, V_EMPTY + (int)vu, vph ^ 1u, status)) { ok = false; break; }
              const uint32_t fb = sh.bar(V_FULL + (int)vu), dst = sh.base + kOffV + vu * kUnit;
              const int tok = last == 0 ? ta : tb;
              mbar_expect_tx(fb, kUnit);
#pragma unroll
              for (int kh = 0; kh < 2; ++kh) {
                tma_load_3d(dst + (uint32_t)kh * kVBlock, &map_v32, fb, 0, g, m.total_tokens);
                tma_load_3d(dst + (uint32_t)kh * kVBlock + 4096, &map_v32, fb, 64, g, m.total_tokens);
                tma_load_3d(dst + (uint32_t)kh * kVBlock + 8192, &map_v32, fb, 0, g, tok + 32 * kh);
                tma_load_3d(dst + (uint32_t)kh * kVBlock + 12288, &map_v32, fb, 64, g, tok + 32 * kh);
              }
              if (++vu == kVUnits) { vu = 0; vph ^= 1u; }
            }
            j0 = ra; j1 = rb;
            ++cnt;
          }
        }
      }
    }
    // ========================================================================================== MMA issuer
    else if (warp == 1) {
      if (elect_one()) {
        const uint64_t hi = make_desc(0, 16, 1024) & 0xffffffff00000000ull;
        const uint32_t kd_lo = (uint32_t)make_desc(sh.base + kOffK, 16, 1024), qd_lo = (uint32_t)make_desc(sh.base + kOffQ, 16, 1024);
        const uint32_t vd_lo = (uint32_t)make_desc(sh.base + kOffV, kHalfTile, 1024), vd4_lo = (uint32_t)make_desc(sh.base + kOffV, 4096, 1024);
        uint32_t cs = 0, cp = 0, ku = 0, kph = 0, vu = 0, vph = 0;   // tiles whose S and whose P V are issued, ring positions
        uint32_t n = 0, nitem = 0, nfirst = 0, qlo = 0, kinds = 0;   // next ring slot, items with tiles, items whose P V is begun; four bits a tile (tile & 3):
        int left = 0, len = 0;                                       // first, two positions, first position / second position for the second block alone
        bool ok = true, done = false, lone = false;
        while (ok) {
          // ---- S, up to two tiles ahead of P V.  With P V work pending the next item is not waited for: its announcement may
          // need the softmax groups to get on, and they that P V.
          while (!done && cs - cp < 2u) {
            uint32_t kind = 0;
            if (left == 0) {
              const uint32_t par = (n >> 2) & 1u;
              if (cs != cp) { if (!mbar_test(sh.bar(ITEM_FULL + (int)(n & 3u)), par)) break; }
              else if (!mbar_wait(sh, ITEM_FULL + (int)(n & 3u), par, status)) { ok = false; break; }
              const Slot it = read_slot(n);
              mbar_arrive(sh.bar(ITEM_EMPTY + (int)(n & 3u)));
              ++n;
              if (it.len < 0) { done = true; break; }
              len = it.len; lone = it.lone();
              left = it.tiles();
              if (left == 0) continue;
              qlo = qd_lo + (nitem & 1u) * (kQBytes >> 4);
              if (!mbar_wait(sh, Q_FULL + (int)(nitem & 1u), (nitem >> 1) & 1u, status)) { ok = false; break; }
              ++nitem;
              kind = 1u;
            }
            const bool two = left > 1 || (len & 1) == 0;
            kind |= (two ? 2u : 0u) | (left == 1 && lone ? (two ? 8u : 4u) : 0u);
            kinds = (kinds & ~(15u << (4 * (cs & 3u)))) | kind << (4 * (cs & 3u));
            // (P V of tile cs - 2, which reads P from the same columns, is ahead on the pipe, which takes the MMAs of one thread and shape in turn, as in
            // attn_tc_kernel.  A wait for its commit: 65 536 tokens in 128-token blocks, the whole pass, 3729 -> 3821 us, 16 384 dense with the map 2927 -> 2972)
            const uint32_t d = tmem + col_s(cs & 1u, 0), klo = kd_lo + ku * (kUnit >> 4);
            if (!mbar_wait(sh, K_FULL + (int)ku, kph, status)) { ok = false; break; }
            tc_fence_after();
#pragma unroll
            for (int kk = 0; kk < 8; ++kk) {
              const uint32_t off = (uint32_t)((kk >> 2) * (2 * kHalfTile >> 4) + (kk & 3) * 2);
              tc_mma_ss(d, hi | (uint64_t)(qlo + off), hi | (uint64_t)(klo + off), kIdescS, kk != 0 ? 1u : 0u);
            }
            tc_commit(sh.bar(S_FULL + (int)(cs & 1u)));
            tc_commit(sh.bar(K_EMPTY + (int)ku));
            if (++ku == kKUnits) { ku = 0; kph ^= 1u; }
            if (--left == 0) tc_commit(sh.bar(Q_EMPTY + (int)((nitem - 1) & 1u)));
            ++cs;
          }
          if (!ok) break;
          if (cp == cs) { if (done) break; continue; }
          // ---- P V of tile cp, one group after the other
          const uint32_t kind = kinds >> (4 * (cp & 3u)), pbuf = cp & 1u, keep = (kind & 1u) ^ 1u, ppar = (cp >> 1) & 1u;
          if ((kind & 1u) != 0u) {                           // the groups have read the O of the item before
            if (!mbar_wait(sh, O_FREE, (nfirst & 1u) ^ 1u, status)) break;
            ++nfirst;
          }
          const bool whole = (kind & 4u) == 0u;              // (a tile of the lone block alone has no unit of whole ones)
          if (whole && !mbar_wait(sh, V_FULL + (int)vu, vph, status)) break;
          uint32_t vlo = vd_lo + vu * (kUnit >> 4);
#pragma unroll
          for (int g = 0; g < 2; ++g) {
            if (!mbar_wait(sh, P_FULL + 2 * g + (int)pbuf, ppar, status)) { ok = false; break; }
            tc_fence_after();
            if ((kind & (g == 0 ? 4u : 8u)) != 0u) {         // for the second block alone
              if (g == 1) {
                tc_commit(sh.bar(V_EMPTY + (int)vu));
                if (++vu == kVUnits) { vu = 0; vph ^= 1u; }
              }
              if (!mbar_wait(sh, V_FULL + (int)vu, vph, status)) { ok = false; break; }
              // The tile before (lone() sees that there is one) has accumulated on the same O in another form and shape: MMAs of one
              // accumulator keep their order by themselves only within a shape.
              if (!mbar_wait(sh, PV_DONE + (int)(pbuf ^ 1u), ((cp - 1u) >> 1) & 1u, status)) { ok = false; break; }
              tc_fence_after();
              const uint32_t v4lo = vd4_lo + vu * (kUnit >> 4);
#pragma unroll
              for (int kk = 0; kk < 4; ++kk)
                tc_mma_ws_ts(tmem + col_o(g), tmem + col_s(pbuf, g) + (uint32_t)kk * 8u, hi | (uint64_t)(v4lo + (uint32_t)((kk >> 1) * (kVBlock >> 4) + (kk & 1) * 128)), kIdescLone, 1u);
            } else if (g == 0 || (kind & 2u) != 0u) {
#pragma unroll
              for (int kk = 0; kk < 4; ++kk)                 // 16 keys (2048 bytes of 128-byte rows, 8 columns of P) per step
                tc_mma_ts(tmem + col_o(g), tmem + col_s(pbuf, g) + (uint32_t)kk * 8u, hi | (uint64_t)(vlo + (uint32_t)(g * (kVBlock >> 4) + kk * 128)), kIdescPV, kk != 0 ? 1u : keep);
            }
          }
          if (!ok) break;
          tc_commit(sh.bar(PV_DONE + (int)pbuf));
          tc_commit(sh.bar(V_EMPTY + (int)vu));
          if (++vu == kVUnits) { vu = 0; vph ^= 1u; }
          ++cp;
        }
      }
    }
  }
  // ============================================================================================ softmax groups
  else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kSoftmaxRegs));
    const int g = (warp - 4) >> 2;                          // list positions of this parity
    const int quad = warp & 3, half = quad >> 1;            // TMEM lane quadrant; which of the item's query blocks
    const int r = quad * 32 + lane, row = r & 63;
    const uint32_t lane_addr = (uint32_t)(quad * 32) << 16;
    const float sl2 = m.softmax_scale * 1.4426950408889634f;
    const uint32_t ml = sh.base + kOffMl, o_addr = tmem + lane_addr + col_o(g);
    const int64_t lse_stride = kChunk ? m.total_q_tokens : m.total_tokens;
    constexpr int bar_vote = 1, kBoth = 256;
    uint32_t cnt = 0;                                       // tiles
    for (uint32_t n = 0;; ++n) {
      // a lost wait does not simply leave: both groups meet in every item, and all warps have to get there
      bool fail = !mbar_wait(sh, ITEM_FULL + (int)(n & 3u), (n >> 2) & 1u, status);
      Slot it{};
      if (!fail) it = read_slot(n);
      __syncwarp();
      if (lane == 0 && !fail) mbar_arrive(sh.bar(ITEM_EMPTY + (int)(n & 3u)));
      fail = __any_sync(0xffffffffu, fail);
      if (fail || it.len < 0) { named_bar_or(bar_vote, kBoth, fail); break; }
      const int tiles = it.tiles(), mine_n = half ? it.n[1] : it.n[0], valid = half ? it.valid[1] : it.valid[0];
      uint16_t* orow = o + (((int64_t)it.tok0 + 64 * half + row) * m.num_q_heads + it.h) * kHeadDim + g * 64;
      const int64_t lrow = (int64_t)it.h * lse_stride + it.tok0 + 64 * half + row;
      if (tiles == 0) {                                     // no visible key: o = 0, lse = -inf
        if (row < valid) {
#pragma unroll
          for (int c = 0; c < 8; ++c) reinterpret_cast<uint4*>(orow)[c] = make_uint4(0u, 0u, 0u, 0u);
          if (g == 0 && lse != nullptr) lse[lrow] = -CUDART_INF_F;
        }
        continue;
      }
      float R = kNoRef, l = 0.f;
      int t = 0;
      // tiles that this half lists, up to its diagonal
      for (const int plain = ((half ? it.plain[1] : it.plain[0]) + 1 - g) >> 1; t < plain; ++t, ++cnt) {
        const uint32_t buf = cnt & 1u, s_addr = tmem + lane_addr + col_s(buf, g);
        fail = !mbar_wait_warp(sh, S_FULL + (int)buf, (cnt >> 1) & 1u, status);
        if (fail) break;
        tc_fence_after();
        if (t == 0) {
          const float mx = row_max<false>(s_addr, 63);
          if (fabsf(mx) < 3.0e38f) R = mx * sl2;
        }
        uint32_t pk[32];
        const float sum = row_pass<false>(s_addr, sl2, R, 63, pk);
        if (!__any_sync(0xffffffffu, !(sum < kRise))) {
          l = __fadd_rn(l, sum);
          tc_st32(s_addr, pk);                              // P over the scores this thread has read
          tc_wait_st();
          tc_fence_before();
        } else {
          const float4 x = other_tile(sh, s_addr, o_addr, sl2, R, l, 63, false, t, PV_DONE + (int)(buf ^ 1u), ((cnt - 1) >> 1) & 1u, status);
          R = x.x; l = x.y; fail = x.z != 0.f;
          if (fail) break;
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(sh.bar(P_FULL + 2 * g + (int)buf));
      }
      // its diagonal, and tiles of the other half alone
      for (; t < tiles && !fail; ++t, ++cnt) {
        const uint32_t buf = cnt & 1u;
        fail = !mbar_wait_warp(sh, S_FULL + (int)buf, (cnt >> 1) & 1u, status);
        if (fail) break;
        tc_fence_after();
        const float4 x = other_tile(sh, tmem + lane_addr + col_s(buf, g), o_addr, sl2, R, l, 2 * t + g < mine_n ? row : -1, t == 0, t, PV_DONE + (int)(buf ^ 1u),
                                    ((cnt - 1) >> 1) & 1u, status);
        R = x.x; l = x.y; fail = x.z != 0.f;
        if (fail) break;
        __syncwarp();
        if (lane == 0) mbar_arrive(sh.bar(P_FULL + 2 * g + (int)buf));
      }
      // ---------------------------------------------------------------------------------------- merge of the two groups, store
      st_shared_v2(ml + (uint32_t)(g * 128 + r) * 8u, __float_as_uint(R), __float_as_uint(l));
      if (named_bar_or(bar_vote, kBoth, fail)) break;
      const bool two = mine_n > 1;                          // both groups have something of this row
      const uint32_t at = ml + (uint32_t)((g ^ 1) * 128 + r) * 8u;
      const float Ro = ld_shared_f32(at), lo = ld_shared_f32(at + 4u);
      float sc, sco, lse_row;                               // factors of this group's and the other's partial row
      if (two) {
        // out = (2^(R_0 - R) O_0 + 2^(R_1 - R) O_1) / l, R = max(R_0, R_1)
        const float Rm = fmaxf(R, Ro);
        const float f = l == 0.f ? 0.f : ex2f(R - Rm), fo = lo == 0.f ? 0.f : ex2f(Ro - Rm);
        const float la = __fmul_rn(l, f), lb = __fmul_rn(lo, fo), total = __fadd_rn(la, lb);
        sc = total > 0.f ? f / total : 0.f;
        sco = total > 0.f ? fo / total : 0.f;
        lse_row = total > 0.f ? (Rm + log2f(total)) * 0.6931471805599453f : -CUDART_INF_F;
      } else {
        sc = l > 0.f ? 1.f / l : 0.f;
        sco = lo > 0.f ? 1.f / lo : 0.f;
        lse_row = l > 0.f ? (R + log2f(l)) * 0.6931471805599453f : -CUDART_INF_F;
      }
      fail = !mbar_wait_warp(sh, PV_DONE + (int)((cnt - 1) & 1u), ((cnt - 1) >> 1) & 1u, status);
      fail = named_bar_or(bar_vote, kBoth, fail);           // no row is stored by halves
      if (fail) break;
      tc_fence_after();
      // this group's thread makes d columns 64 g .. of its row, from both groups' O
      uint32_t mine[2][32], other[2][32];
      const uint32_t m_addr = o_addr + (uint32_t)g * 64u, x_addr = tmem + lane_addr + col_o(g ^ 1) + (uint32_t)g * 64u;
      tc_ld32(m_addr, mine[0]); tc_ld32(x_addr, other[0]);
      tc_ld32(m_addr + 32, mine[1]); tc_ld32(x_addr + 32, other[1]);
      tc_wait_ld32(mine[0]); tc_wait_ld32(other[0]); tc_wait_ld32(mine[1]); tc_wait_ld32(other[1]);
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(sh.bar(O_FREE));
      if (row < valid) {
        const float2 sc2 = make_float2(sc, sc), sco2 = make_float2(sco, sco);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          uint32_t out[8];
#pragma unroll
          for (int c = 0; c < 8; ++c) {
            const int e = (q & 1) * 16 + 2 * c;
            const float2 a = make_float2(__uint_as_float(mine[q >> 1][e]), __uint_as_float(mine[q >> 1][e + 1]));
            const float2 b = __fmul2_rn(make_float2(__uint_as_float(other[q >> 1][e]), __uint_as_float(other[q >> 1][e + 1])), sco2);
            const float2 x = two ? __ffma2_rn(a, sc2, b) : g == 0 ? __fmul2_rn(a, sc2) : b;
            out[c] = mine_n > 0 ? pack_bf16(x.x, x.y) : 0u;
          }
          st_global_32(orow + q * 16, out, kO32);
        }
        if (g == 0 && lse != nullptr) lse[lrow] = lse_row;
      }
    }
  }

  // After a lost wait give copies and MMAs still in flight time to land before shared memory and TMEM go away.
  if (ld_shared_u32(sh.abort_flag()) != 0u)
    for (int k = 0; k < 2000; ++k) __nanosleep(1000);
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
  }
}

using Kernel = void(CUtensorMap, CUtensorMap, CUtensorMap, CUtensorMap, SeqMeta, const int32_t*, const int32_t*, uint16_t*, float*, int*, int*, const int*, int, int);

}  // namespace tp

static cudaError_t ready(seer_ctx* ctx) {
  if (ctx->pair_kernels) return cudaSuccess;
  cudaError_t e = cudaSuccess;
  for (tp::Kernel* k : {tp::attn_pair_kernel<false, false>, tp::attn_pair_kernel<false, true>, tp::attn_pair_kernel<true, false>, tp::attn_pair_kernel<true, true>})
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)tp::kSmemBytes);
  ctx->pair_kernels = e == cudaSuccess;
  return e;
}

int launch_pair_check(seer_ctx* ctx, const SeqMeta& m, const int32_t* row_ptr, const int32_t* col_idx, int* counter, const PairAnswer& a, cudaStream_t stream) {
  cudaError_t e = ready(ctx);
  if (e != cudaSuccess) return -(int)e;
  e = launch_next(m.chunked ? tp::check_kernel<true> : tp::check_kernel<false>, (unsigned)a.nwords, tp::kCheckWarps * 32, 0, stream, m, row_ptr, col_idx, counter, a.words, a.epoch);
  return e == cudaSuccess ? 1 : -(int)e;
}

int launch_attn_pair(seer_ctx* ctx, const SeqMeta& m, const CUtensorMap& mq, const CUtensorMap& mk, const CUtensorMap& mv, const CUtensorMap& mv32, const int32_t* row_ptr,
                     const int32_t* col_idx, void* o, float* lse, int* counter, const PairAnswer& a, cudaStream_t stream) {
  const bool o32 = ((uintptr_t)o & 31) == 0;
  tp::Kernel* kernel = m.chunked ? (o32 ? tp::attn_pair_kernel<true, true> : tp::attn_pair_kernel<true, false>)
                                 : (o32 ? tp::attn_pair_kernel<false, true> : tp::attn_pair_kernel<false, false>);
  const cudaError_t e = launch_next(kernel, (unsigned)min((int64_t)ctx->num_sms, m.pair_units), tp::kThreads, tp::kSmemBytes, stream, mq, mk, mv, mv32, m, row_ptr,
                                    col_idx, (uint16_t*)o, lse, ctx->d_status, counter, (const int*)a.words, a.nwords, a.epoch);
  return e == cudaSuccess ? 1 : -(int)e;
}

}  // namespace seer
