// Block-sparse causal GQA attention (Sec. 3.3) on the Blackwell tensor path, two work items in flight per CTA.
//
// What bounds it.  Long lists: the copies of K and V into shared memory (64 KB per pair of listed 64 x 64 blocks, about 885 clocks
// at the 74 bytes a clock that an SM takes from L2, of 960 that a pair takes with one in ten of 128k tokens), close before the MMA pipe (8 x 48 + 4 x 76 =
// 688 clocks: 75 % active on dense lists of 16k tokens), and in launches of more than a few milliseconds the board's power limit.
// Short lists: an item's start and end, about 5300 clocks beside 1730 for a stream's tile (instrumented).  Of them the wait for the last P V 1250, merge and
// stores 3400; everything that needs no O is done during the wait, and an item's row pointers and first list
// entries are fetched while the item before it is copied.  With those after the wait, the entries fetched at the item's start, and
// producers that slept between their polls: 6000 clocks; the launch by itself, both in turn: 24 prompts of 16 900 tokens 174 us where this
// takes 166, 32k tokens 1232 and 1174, 48k 2557 and 2480, 128k 16.7 and 16.1 ms; dense 2000-token prompts 435 and 432.  (A whole pass, which runs
// hotter: 3 % on short prompts, 1 to 2 on long ones.)
//
// Tiles.  A query block is 64 rows and every (head, query block) has its own list, so no two items share their keys.
// The MMAs are the weight-stationary form (tcgen05.mma.ws) with M = 64: the 128 lanes of tensor memory hold two 64-row
// halves, lanes 0-63 belong to the first half of the N columns and lanes 64-127 to the second, and an A operand in tensor
// memory is read by every lane from its own row.  A tile is two listed KV blocks a and b:
//     S[64 q x 128 keys] = Q (smem) * [K_a; K_b]^T      N = 128: lanes 0-63 get the scores of block a, 64-127 those of b
//     O_a += P_a V_a and O_b += P_b V_b                 N = 256: the same instruction, A = P in tensor memory (64 keys),
//                                                       B = [V_a | V_b]: lanes 0-63 accumulate O_a, lanes 64-127 O_b
// so all 128 lanes work for arbitrary lists at 82 % of the full MMA rate (K = 16 in 48 clocks for N = 128, 76 for 256; the
// ordinary M = 64 form takes 64 and 128).  A thread owns a query row and all 64 keys of one block: the softmax needs no
// other thread.  The two halves are two partial results with their own references and sums (as in split-KV decoding), merged
// once per item.  The transposed product (S^T = K Q^T, a thread per key, a vote of the group per tile, P^T through shared memory)
// takes 17 MMAs of 48 clocks per tile and 20.5 ms where this takes 15.3 (128k tokens, one block in ten).
//
// References.  p = 2^(s * scale * log2(e) - R), R the row's maximum over the half's first live block.  P is bf16 and the sums are
// fp32, so p may grow to 2^60 before R has to move: the sum of a tile's 64 probabilities says so, without a maximum.  O
// holds the values at that scale, so values up to 2^50 stay finite however a row's scores rise.  (2^30 here, for values up to 2^80:
// short prompts 253.6 us against 252.1, long ones alike; 2^20: 264; 2^10: 338 and long ones 10 to 30 % more.)
// When it does, the warp waits for the previous P V, rescales its rows of O and its sums and takes the tile again.
//
// Arrangement.  A CTA runs two independent streams; a stream owns a whole work item (head, query block) from its first
// tile to its stores: two Q buffers, rings of K and V units, two S buffers and O in tensor memory (2 x 64 + 128 columns;
// P(t) overwrites the first 32 columns of S(t)).  A K unit is a d half of a tile (2 x 64 keys x 64 d), a V unit a key half
// (2 x 32 keys x 128 d), 16 KB each, given back to the producer as soon as its MMAs have read it.  Roles (512 threads):
// warps 0 / 2 = producer of Q and K of stream 0 / 1, warps 12 / 13 = producer of V, warps 1 / 3 = MMA issuer (warp 1 owns
// tensor memory), warps 4-7 / 8-11 = softmax group.  The issuer computes S two tiles ahead of P V, across items, so that a
// group that ends an item finds the next item's scores waiting.  The Q / K producer draws the work items, decodes them and
// passes them on through a ring of four slots.  Every wait is bounded; a wait that runs out raises SEER_ERR_TIMEOUT and
// the CTA drains and exits.
#include <cuda.h>
#include <math_constants.h>

#include "block_max_pair.cuh"

namespace seer {
namespace tc {

using namespace tcc;

constexpr int kThreads = 512;
// Registers of the helpers' and the softmax warpgroups, two each: 2 * (helper + softmax) * 128 = 65536.  (The softmax pass wants 200; the
// block maxima want less, and their producer spills with 56.)
template <bool kBlockMax> constexpr int kHelperRegs = kBlockMax ? 64 : 56;
template <bool kBlockMax> constexpr int kSoftmaxRegs = 256 - kHelperRegs<kBlockMax>;
constexpr int kGroupThreads = 128;
constexpr uint32_t kHalfQ = 64 * 128;            // bytes of one d half of a 64-row tile (8 KB)
constexpr uint32_t kQBytes = 2 * kHalfQ;         // 16 KB
constexpr uint32_t kUnit = 16384;                // a K or V unit
// Ring depths per stream: three K units and two V units (two and three: 128k tokens 16.33 ms where this takes 16.15 to 16.25, 32k 1201 and 1174 us,
// dense 16k 2481 and 2450, short prompts 0.5 % slower; the launch by itself).
constexpr uint32_t kKUnits = 3, kVUnits = 2;
// shared memory map (offsets from a 1024-byte aligned base); the big buffers of a stream are contiguous
constexpr uint32_t kStQ = 0, kStK = 2 * kQBytes, kStV = kStK + kKUnits * kUnit;
constexpr uint32_t kStreamBytes = kStV + kVUnits * kUnit;         // 112 KB
constexpr uint32_t kOffMl = 2 * kStreamBytes;                     // per stream: (reference, sum) of 128 rows; block maxima
constexpr uint32_t kMlBytes = 1024;
constexpr uint32_t kOffBar = kOffMl + 2 * kMlBytes;               // mbarriers
constexpr int kBarsPerStream = 40;
constexpr uint32_t kOffRing = kOffBar + 2 * kBarsPerStream * 8;   // per stream: four item slots of 32 bytes
constexpr uint32_t kOffMisc = kOffRing + 2 * 4 * 32;              // tmem base, abort flag
constexpr uint32_t kSmemBytes = kOffMisc + 64;                    // (no slack: the kernel checks the base's alignment)
static_assert(kSmemBytes <= 232448, "shared memory budget of one CTA");

enum Bar { Q_FULL = 0 /* + buf */, Q_EMPTY = 2, K_FULL = 4 /* + unit */, K_EMPTY = 7, V_FULL = 10, V_EMPTY = 13,
           S_FULL = 16 /* + buf */, P_FULL = 18, PV_DONE = 20, ITEM_FULL = 22 /* + slot */, ITEM_EMPTY = 26, kBars = 30,
           // the block maxima have no V, no P and no O: five K units, four S buffers (M_TAKEN: the group has its maxima)
           M_KEMPTY = 30, M_TAKEN = 10, kBarsMax = 35 };
static_assert(kBarsMax <= kBarsPerStream && kKUnits <= 3 && kVUnits <= 3, "barrier map");
static_assert(tp::kMaxEnd <= kOffBar, "the maxima by pairs have barriers of their own");

constexpr uint32_t kTmemCols = 512;
// TMEM columns of a stream: two S buffers (P in their first 32 columns), O
__device__ __forceinline__ uint32_t col_s(int s, uint32_t buf) { return (uint32_t)s * 256u + buf * 64u; }
__device__ __forceinline__ uint32_t col_o(int s) { return (uint32_t)s * 256u + 128u; }

constexpr uint32_t kIdescS = make_idesc(false, false, 128u, 64u);
constexpr uint32_t kIdescPV = make_idesc(false, true, 256u, 64u);

// What the roles need to know of a work item (decoded once, by the stream's Q / K producer).
struct Slot {
  int h, i, l0, nlist, q_valid, s0, tok0;   // tok0: first row of the item in q / o / lse
  int first[2];                             // the list's first two entries (not for the block maxima)
  __device__ __forceinline__ int ntiles() const { return (nlist + 1) >> 1; }
};
__device__ __forceinline__ int slot_block(const Slot& it, const int32_t* col_idx, int p) {
  return p < it.nlist ? (int)ld_global(reinterpret_cast<const uint32_t*>(col_idx) + it.l0 + p) : -1;
}
// Block index of a list entry: -1 past the end of the list, -2 outside [0, i].
__device__ __forceinline__ int slot_check(const Slot& it, int p, int raw) {
  if (p >= it.nlist) return -1;
  return (raw < 0 || raw > it.i) ? -2 : raw;
}

// ------------------------------------------------------------------------------------------------ kernel
// kBlockMax: the same pipeline without V: instead of softmax(S) V the kernel writes, for every list entry, the largest
// probability exp(scale * s - lse) of its 64 x 64 tile (Sec. 3.2, Eq. 2 on the listed blocks), `lse` being an input: a
// thread takes the maximum of its row, a block's maximum is one redux per warp and a word from its neighbour.
// Without V and O a stream has five K units and four S buffers: with two of each it waits for copies and MMAs in turn (16k tokens, 32
// heads, all causal blocks: 1277 us and 1060 so when both were timed on a cool board, 520 clocks a tile; 440 are its 32 KB from L2, 384 its
// MMAs; 1160 to 1210 us behind an attention launch).
// kO32: o begins on 32 bytes.  (A test of the address in the kernel instead: 32k tokens 1392 -> 1404 us.)
template <bool kTrace, bool kChunk, bool kBlockMax = false, bool kO32 = true>
__global__ void __launch_bounds__(kThreads, 1)
attn_tc_kernel(const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_k,
                const __grid_constant__ CUtensorMap map_v, SeqMeta m,
                const int32_t* row_ptr, const int32_t* col_idx,
                uint16_t* __restrict__ o, float* lse, int* __restrict__ status,
                unsigned long long* __restrict__ trace, float* block_max = nullptr,
                int* __restrict__ work_counter = nullptr, const int* words = nullptr, int nwords = 0, int epoch = 0, bool pairs = false) {
  extern __shared__ __align__(1024) unsigned char smem[];
  Shared sh;
  sh.base = smem_u32(smem);
  sh.bar0 = sh.base + kOffBar;
  sh.abort_addr = sh.base + kOffMisc + 8;
  sh.limit_us = m.wait_limit_us;
  if (!kBlockMax && words != nullptr) {                    // (a way out from further in costs a launch of 32k tokens 2 %)
    grid_wait();
    if (tp::lists_agree(words, nwords, epoch)) return;      // attn_pair_kernel does the work
  }
  if ((sh.base & 1023u) != 0u) {                           // the swizzled tiles need the alignment
    grid_wait();
    if (threadIdx.x == 0) atomicCAS(status, 0, (int)SEER_ERR_CUDA);
    return;
  }
  const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0), lane = threadIdx.x & 31;   // (warp-uniform for the compiler)
  volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(smem + kOffMisc);

  if (threadIdx.x == 0) {
    for (int s = 0; s < 2; ++s) {
      const int b = s * kBarsPerStream;
      for (int i = 0; i < (kBlockMax ? kBarsMax : kBars); ++i) {
        // Q_EMPTY, P_FULL: one arrival per warp of the softmax group; ITEM_EMPTY: those, the V producer (block maxima: the K producer) and the issuer
        const bool group = (i >= Q_EMPTY && i < Q_EMPTY + 2) || (kBlockMax ? i >= M_TAKEN && i < M_TAKEN + 4 : i >= P_FULL && i < P_FULL + 2);
        mbar_init(sh.bar(b + i), i >= ITEM_EMPTY && i < ITEM_EMPTY + 4 ? 6 : group ? 4 : 1);
      }
    }
    st_shared_u32(sh.abort_flag(), 0u);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(sh.base + kOffMisc), "r"(kTmemCols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (kBlockMax && pairs && warp == 2) tp::max_init(sh.base, lane);
  tc_fence_before();
  bool by_pairs = false;
  if constexpr (kBlockMax) {
    if (pairs) {
      __syncwarp();                                        // (thread 0 has set up the barriers)
      grid_wait();
      by_pairs = tp::share_agrees<kChunk>(m, row_ptr, col_idx, warp, lane);   // (meets as below)
    }
  }
  if (!(kBlockMax && pairs)) __syncthreads();
  tc_fence_after();
  grid_wait();
  const uint32_t tmem = *tmem_slot;
  const unsigned long long cta_t0 = kTrace ? global_ns() : 0ull;
  const long long cta_c0 = kTrace ? clock64() : 0ll;

  // Work items.  Without a counter a stream takes the items CTA + stream * grid, + 2 * grid, ... (static deal: as long as there are no
  // more items than CTAs each has an SM to itself: 128 items 12.3 us, two to an SM 15.2).  With one
  // (`work_counter`, zero at launch) the next item number is drawn from it.  Either way the stream's Q / K producer decodes
  // the item and passes it to the other roles through a ring of four slots, each with a full and an empty mbarrier: a slot
  // is rewritten only when every other role has read it.  nlist < 0 ends the stream.  Results do not depend on which
  // stream runs an item.
  constexpr uint32_t ring_k = kBlockMax ? kKUnits + kVUnits : kKUnits;   // without V its units are K's, without O its columns S buffers
  constexpr int empty_k = kBlockMax ? M_KEMPTY : K_EMPTY;
  const bool dyn = work_counter != nullptr;
  auto ring_addr = [&](int s, uint32_t n) -> uint32_t { return sh.base + kOffRing + (uint32_t)s * 128u + (n & 3u) * 32u; };
  auto read_slot = [&](int s, uint32_t n) -> Slot {
    const uint4 a = ld_shared_v4(ring_addr(s, n)), b = ld_shared_v4(ring_addr(s, n) + 16u);
    Slot it;
    it.h = (int)a.x; it.i = (int)(a.y >> 7); it.q_valid = (int)(a.y & 127u);   // (a batch has at most 2^25 blocks)
    it.l0 = (int)a.z; it.nlist = (int)a.w;
    it.s0 = (int)b.x; it.tok0 = (int)b.y; it.first[0] = (int)b.z; it.first[1] = (int)b.w;
    return it;
  };
  auto first_entry = [&](const Slot& it, int p) -> int { return kBlockMax ? slot_block(it, col_idx, p) : it.first[p]; };
  auto item_full = [&](int s, uint32_t n) -> int { return s * kBarsPerStream + ITEM_FULL + (int)(n & 3u); };
  auto put_item = [&](int s, uint32_t n, const Item& nx, bool more, int e0, int e1) -> bool {
    // the slot's previous content (item n - 4) has been read by everyone
    if (!mbar_wait(sh, s * kBarsPerStream + ITEM_EMPTY + (int)(n & 3u), ((n >> 2) & 1u) ^ 1u, status)) return false;
    const int tok0 = nx.s0 + nx.i * kBlock + (kChunk ? nx.dq : 0);
    st_shared_v4(ring_addr(s, n), (uint32_t)nx.h, (uint32_t)nx.i << 7 | (uint32_t)nx.q_valid, (uint32_t)nx.l0, more ? (uint32_t)nx.nlist : 0xffffffffu);
    st_shared_v4(ring_addr(s, n) + 16u, (uint32_t)nx.s0, (uint32_t)tok0, (uint32_t)e0, (uint32_t)e1);
    mbar_arrive(sh.bar(item_full(s, n)));
    return true;
  };
  auto release_item = [&](int s, uint32_t n) { mbar_arrive(sh.bar(s * kBarsPerStream + ITEM_EMPTY + (int)(n & 3u))); };

  if (by_pairs) {
    if constexpr (kBlockMax)
      tp::block_max_pairs<kChunk, kHelperRegs<true>, kSoftmaxRegs<true>>(map_q, map_k, m, sh, smem, tmem, warp, lane, row_ptr, col_idx, lse, status, block_max);
  } else if (warp < 4 || warp >= 12) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kHelperRegs<kBlockMax>));
    // ========================================================================================== producer of Q and K (TMA)
    if (warp == 0 || warp == 2) {
      if (elect_one()) {
        const int s = warp >> 1, bb = s * kBarsPerStream;
        const uint32_t sbase = sh.base + (uint32_t)s * kStreamBytes;
        Tracer<kTrace> tr; tr.init(s == 0 ? trace : nullptr, 0);
        const int64_t w_step = 2 * (int64_t)gridDim.x;
        int64_t w_static = (int64_t)blockIdx.x + (int64_t)s * gridDim.x;
        auto draw = [&]() -> int64_t {
          if (dyn) return (int64_t)atomicAdd(work_counter, 1);
          const int64_t w = w_static;
          w_static += w_step;
          return w;
        };
        uint32_t nitem = 0, cnt = 0, ku = 0, kph = 0;
        bool ok = true;
        // An item is decoded and announced while the one before it is copied: its row pointers and its first list entries are two
        // trips to L2, one after the other, that every role of the stream would wait for at the item's start.  (The block maxima have warps to spare for it.)
        Item nx{};
        bool more = false;
        auto locate = [&](int64_t w) {                     // which item comes next
          more = w < m.q_rows;
          nx = Item{};
          if (more) nx = decode_item<kChunk, true>(m, row_ptr, w);
        };
        auto announce = [&](uint32_t n) -> bool {
          const int na0 = 0 < nx.nlist ? (int)ld_global(reinterpret_cast<const uint32_t*>(col_idx) + nx.l0) : -1;
          const int nb0 = 1 < nx.nlist ? (int)ld_global(reinterpret_cast<const uint32_t*>(col_idx) + nx.l0 + 1) : -1;
          return put_item(s, n, nx, more, na0, nb0);
        };
        if (!kBlockMax) {
          locate(draw());
          ok = announce(0);
        }
        for (uint32_t n = 0; ok; ++n) {
          if (kBlockMax && !mbar_wait(sh, item_full(s, n), (n >> 2) & 1u, status)) break;
          const Slot it = read_slot(s, n);                 // (its own announcement: two items in 56 registers are 1 % of a long launch)
          if (kBlockMax) release_item(s, n);
          if (it.nlist < 0) break;
          int ja = slot_check(it, 0, first_entry(it, 0)), jb = slot_check(it, 1, first_entry(it, 1));
          const int64_t w = kBlockMax ? 0 : draw();        // the next one is on its way while this one is copied
          const int ntiles = it.ntiles(), g = it.h / m.group;
          if (ntiles == 0) {
            if (!kBlockMax) { locate(w); ok = announce(n + 1); }
            continue;
          }
          const uint32_t qb = nitem & 1u;
          if (!mbar_wait(sh, bb + Q_EMPTY + (int)qb, ((nitem >> 1) & 1u) ^ 1u, status)) break;
          mbar_expect_tx(sh.bar(bb + Q_FULL + (int)qb), kQBytes);
          tma_load_3d(sbase + kStQ + qb * kQBytes, &map_q, sh.bar(bb + Q_FULL + (int)qb), 0, it.h, it.tok0);
          tma_load_3d(sbase + kStQ + qb * kQBytes + kHalfQ, &map_q, sh.bar(bb + Q_FULL + (int)qb), 64, it.h, it.tok0);
          ++nitem;
          for (int t = 0; t < ntiles; ++t, ++cnt) {
            const int ra = slot_block(it, col_idx, 2 * t + 2), rb = slot_block(it, col_idx, 2 * t + 3);   // next pair
            if (ja == -2 || jb == -2) atomicCAS(status, 0, (int)SEER_ERR_INVALID_INDEX);
            const bool has_b = jb != -1;
            // a rejected entry: any valid block, masked out in the softmax
            const int ta = it.s0 + (ja < 0 ? 0 : ja) * kBlock, tb = it.s0 + (jb < 0 ? 0 : jb) * kBlock;
            tr.sample(cnt); tr.ev(1);
            // test hook of the block maxima: one K copy that is never issued, so that the issuer's wait for it runs out
            const bool lost = kBlockMax && s == 0 && blockIdx.x == 0 && m.lose_v_copy >= 0 && cnt == (uint32_t)m.lose_v_copy;
#pragma unroll
            for (int dh = 0; dh < 2; ++dh) {
              if (!mbar_wait(sh, bb + empty_k + (int)ku, kph ^ 1u, status)) { ok = false; break; }
              const uint32_t fb = sh.bar(bb + K_FULL + (int)ku), dst = sbase + kStK + ku * kUnit;
              if (!lost) {
                mbar_expect_tx(fb, has_b ? kUnit : kUnit / 2);   // (an odd list's last tile: the scores of the missing block are not looked at)
                tma_load_3d(dst, &map_k, fb, 64 * dh, g, ta);
                if (has_b) tma_load_3d(dst + kHalfQ, &map_k, fb, 64 * dh, g, tb);
              }
              if (++ku == ring_k) { ku = 0; kph ^= 1u; }
            }
            tr.ev(2);
            if (!ok) break;
            ja = slot_check(it, 2 * t + 2, ra); jb = slot_check(it, 2 * t + 3, rb);
            if (!kBlockMax && t == 0) locate(w);
            if (!kBlockMax && t == min(1, ntiles - 1) && !announce(n + 1)) { ok = false; break; }
          }
        }
      }
    }
    // ========================================================================================== producer of V (TMA)
    else if (warp == 12 || warp == 13) {
      if (kBlockMax) {
        // The block maxima: items are decoded and announced ahead of the copies.  Where lists have a few blocks the producer has no time for it
        // (24 sequences of 2048 tokens, 64 heads, one in twenty: 273 us behind an item's last copy, 257 so).
        if (elect_one()) {
          const int s = warp - 12;
          bool more = true;
          for (uint32_t n = 0; more; ++n) {
            Item nx{};
            if (pairs) {                                   // the blocks of the pairs dealt to this CTA (share_agrees), a stream each
              const int64_t w = tp::dealt_pair(m, n);
              more = w >= 0;
              if (more) {
                const tp::PairItem u = tp::decode_pair<kChunk, true>(m, row_ptr, w);
                nx.h = u.h; nx.i = u.i0 + s; nx.s0 = u.s0; nx.dq = u.tok0 - u.s0 - u.i0 * kBlock;
                nx.l0 = s ? u.l[1] : u.l[0]; nx.nlist = s ? u.n[1] : u.n[0]; nx.q_valid = s ? u.valid[1] : u.valid[0];
              }
            } else {
              const int64_t w = (int64_t)blockIdx.x + (2 * (int64_t)n + s) * gridDim.x;
              more = w < m.q_rows;
              if (more) nx = decode_item<kChunk, kChunk>(m, row_ptr, w);
            }
            if (!put_item(s, n, nx, more, -1, -1)) break;
          }
        }
      } else if (elect_one()) {
        const int s = warp - 12, bb = s * kBarsPerStream;
        const uint32_t sbase = sh.base + (uint32_t)s * kStreamBytes;
        Tracer<kTrace> tr; tr.init(s == 0 ? trace : nullptr, 2);
        uint32_t cnt = 0, vu = 0, vph = 0;
        bool ok = true;
        for (uint32_t n = 0; ok; ++n) {
          if (!mbar_wait(sh, item_full(s, n), (n >> 2) & 1u, status)) break;
          const Slot it = read_slot(s, n);
          release_item(s, n);
          if (it.nlist < 0) break;
          const int g = it.h / m.group;
          int ja = slot_check(it, 0, it.first[0]), jb = slot_check(it, 1, it.first[1]);
          for (int t = 0; t < it.ntiles() && ok; ++t, ++cnt) {
            const int ra = slot_block(it, col_idx, 2 * t + 2), rb = slot_block(it, col_idx, 2 * t + 3);   // next pair
            const int ta = it.s0 + (ja < 0 ? 0 : ja) * kBlock;
            // the last tile of an odd list: the second half multiplies zeros by zeros, which a copy from past the last token brings
            // (values of another block, or what else lies in the buffer, might not be finite); a list of one block has no second
            // half to spoil
            const int tb = jb == -1 ? m.total_tokens : it.s0 + (jb < 0 ? 0 : jb) * kBlock;
            const bool two = it.nlist > 1;
            tr.sample(cnt); tr.ev(1);
            // test hook: one V copy that is never issued, so that the issuer's wait for it runs out
            const bool lost = s == 0 && blockIdx.x == 0 && m.lose_v_copy >= 0 && cnt == (uint32_t)m.lose_v_copy;
#pragma unroll
            for (int kh = 0; kh < 2; ++kh) {
              if (!mbar_wait(sh, bb + V_EMPTY + (int)vu, vph ^ 1u, status)) { ok = false; break; }
              const uint32_t fb = sh.bar(bb + V_FULL + (int)vu), dst = sbase + kStV + vu * kUnit;
              if (!lost) {
                mbar_expect_tx(fb, two ? kUnit : kUnit / 2);
                tma_load_3d(dst, &map_v, fb, 0, g, ta + 32 * kh);
                tma_load_3d(dst + 4096, &map_v, fb, 64, g, ta + 32 * kh);
                if (two) {
                  tma_load_3d(dst + 8192, &map_v, fb, 0, g, tb + 32 * kh);
                  tma_load_3d(dst + 12288, &map_v, fb, 64, g, tb + 32 * kh);
                }
              }
              if (++vu == kVUnits) { vu = 0; vph ^= 1u; }
            }
            tr.ev(2);
            ja = slot_check(it, 2 * t + 2, ra); jb = slot_check(it, 2 * t + 3, rb);
          }
        }
      }
    }
    // ========================================================================================== MMA issuer of a stream
    else if (warp == 1 || warp == 3) {
      if (elect_one()) {
        const int s = warp >> 1, bb = s * kBarsPerStream;
        const uint32_t sbase = sh.base + (uint32_t)s * kStreamBytes;
        Tracer<kTrace> tr; tr.init(trace, s == 0 ? 1 : 3);
        // (the low word of a descriptor holds the start address and the leading-dimension offset, the high word is constant)
        const uint64_t desc_hi_k = make_desc(0, 16, 1024) & 0xffffffff00000000ull;
        const uint64_t desc_hi_v = make_desc(0, 4096, 1024) & 0xffffffff00000000ull;
        const uint32_t kd_lo = (uint32_t)make_desc(sbase + kStK, 16, 1024), qd_lo = (uint32_t)make_desc(sbase + kStQ, 16, 1024);
        const uint32_t vd_lo = (uint32_t)make_desc(sbase + kStV, 4096, 1024);
        const uint32_t d_o = tmem + col_o(s);
        uint32_t cs = 0, cp = 0, ku = 0, kph = 0, vu = 0, vph = 0;   // S tiles and P V tiles issued, ring positions
        uint32_t n = 0, nitem = 0, first_bits = 0;           // next ring slot, items with tiles, first-of-item flags by tile & 3
        int left = 0;                                        // S tiles still to come of the current item
        bool ok = true, done = false;
        while (ok) {
          // ---- S, up to two tiles ahead of P V.  With P V work pending the next item is not waited for: its announcement may
          // need the softmax group to get on, and the group that P V.
          while (!done && cs - cp < 2u) {
            if (left == 0) {
              const uint32_t par = (n >> 2) & 1u;
              if (cs != cp) { if (!mbar_test(sh.bar(item_full(s, n)), par)) break; }
              else if (!mbar_wait(sh, item_full(s, n), par, status)) { ok = false; break; }
              const Slot it = read_slot(s, n);
              release_item(s, n);
              ++n;
              if (it.nlist < 0) { done = true; break; }
              left = it.ntiles();
              if (left == 0) continue;
              if (!mbar_wait(sh, bb + Q_FULL + (int)(nitem & 1u), (nitem >> 1) & 1u, status)) { ok = false; break; }
              ++nitem;
              first_bits |= 1u << (cs & 3u);
            } else first_bits &= ~(1u << (cs & 3u));
            tr.sample(cs); tr.ev(10);
            if constexpr (kBlockMax) {
              // the group has taken the maxima of this S buffer's previous tile
              if (cs >= 4 && !mbar_wait(sh, bb + M_TAKEN + (int)(cs & 3u), ((cs - 4) >> 2) & 1u, status)) { ok = false; break; }
            }
            const uint32_t sbuf = cs & (kBlockMax ? 3u : 1u), d = tmem + col_s(s, sbuf);     // (P V of tile cs - 2, which read P from it, is ahead on the pipe)
#pragma unroll
            for (int dh = 0; dh < 2 && ok; ++dh) {
              if (!mbar_wait(sh, bb + K_FULL + (int)ku, kph, status)) { ok = false; break; }
              tc_fence_after();
              const uint32_t klo = kd_lo + ku * (kUnit >> 4), qlo = qd_lo + ((nitem - 1) & 1u) * (kQBytes >> 4) + (uint32_t)dh * (kHalfQ >> 4);
#pragma unroll
              for (int kk = 0; kk < 4; ++kk)
                tc_mma_ws(d, desc_hi_k | (uint64_t)(qlo + (uint32_t)kk * 2u), desc_hi_k | (uint64_t)(klo + (uint32_t)kk * 2u), kIdescS, (dh | kk) != 0 ? 1u : 0u);
              tc_commit(sh.bar(bb + empty_k + (int)ku));
              if (++ku == ring_k) { ku = 0; kph ^= 1u; }
            }
            if (!ok) break;
            tc_commit(sh.bar(bb + S_FULL + (int)sbuf));
            tr.ev(12);
            ++cs; --left;
            if constexpr (kBlockMax) ++cp;
          }
          if (!ok) break;
          if (cp == cs) { if (done) break; continue; }
          if constexpr (kBlockMax) continue;
          // ---- P V of tile cp: P is in its S buffer, and the group has finished with the O of the previous item
          tr.sample(cp); tr.ev(13);
          if (!mbar_wait(sh, bb + P_FULL + (int)(cp & 1u), (cp >> 1) & 1u, status)) break;
          tr.ev(15);
          const uint32_t a = tmem + col_s(s, cp & 1u);
          const uint32_t keep = ((first_bits >> (cp & 3u)) & 1u) ^ 1u;
#pragma unroll
          for (int kh = 0; kh < 2 && ok; ++kh) {
            if (!mbar_wait(sh, bb + V_FULL + (int)vu, vph, status)) { ok = false; break; }
            tc_fence_after();
            const uint32_t vlo = vd_lo + vu * (kUnit >> 4);
#pragma unroll
            for (int kk = 0; kk < 2; ++kk)                   // 16 keys (2048 bytes of 128-byte rows, 8 columns of P) per step
              tc_mma_ws_ts(d_o, a + (uint32_t)(kh * 2 + kk) * 8u, desc_hi_v | (uint64_t)(vlo + (uint32_t)kk * 128u), kIdescPV, (kh | kk) != 0 ? 1u : keep);
            tc_commit(sh.bar(bb + V_EMPTY + (int)vu));
            if (++vu == kVUnits) { vu = 0; vph ^= 1u; }
          }
          if (!ok) break;
          tc_commit(sh.bar(bb + PV_DONE + (int)(cp & 1u)));
          tr.ev(16);
          ++cp;
        }
      }
    }
  }   // helper warpgroups
  // ============================================================================================ softmax groups
  else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kSoftmaxRegs<kBlockMax>));
    const int s = (warp - 4) >> 2, bb = s * kBarsPerStream;
    const int quad = warp & 3;                              // TMEM lane quadrant this warp may access
    const int half = quad >> 1;                             // which of a tile's two blocks this warp works on
    const int r = quad * 32 + lane;                         // TMEM lane of this thread
    const int row = r & 63;                                 // query row within the block
    const uint32_t lane_addr = (uint32_t)(quad * 32) << 16;
    const int bar_vote = 1 + s, bar_merge = 3 + s;
    const float sl2 = m.softmax_scale * 1.4426950408889634f;
    const uint32_t ml = sh.base + kOffMl + (uint32_t)s * kMlBytes;
    const uint32_t o_addr = tmem + lane_addr + col_o(s);
    const int64_t lse_stride = kChunk ? m.total_q_tokens : m.total_tokens;
    const bool o32 = kTrace ? (reinterpret_cast<uintptr_t>(o) & 31) == 0 : kO32;
    Tracer<kTrace> tr; tr.init(r == 0 ? trace : nullptr, 4 + s);
    uint32_t cnt = 0, nitem = 0;                            // tiles and items with tiles this stream has processed
    bool lost = false;                                      // block maxima: this warp, or its neighbour, has given up
    for (uint32_t n = 0;; ++n) {
      tr.sample(0);
      // a lost wait does not simply leave: the warps of a group meet once per item with tiles (block maxima: before every item), and all of
      // them have to get there; a warp that gives up votes early, the others find its vote at their next meeting
      bool fail = (kBlockMax && lost) || !mbar_wait(sh, item_full(s, n), (n >> 2) & 1u, status);
      Slot it{};
      if (!fail) it = read_slot(s, n);
      __syncwarp();
      if (lane == 0 && !fail) release_item(s, n);
      fail = __any_sync(0xffffffffu, fail);
      if constexpr (kBlockMax) {
        // a warp with an item waits in it for its neighbour: so either all warps of the group have the item, or none goes on
        if (named_bar_or(bar_vote, kGroupThreads, fail) || it.nlist < 0) break;
      } else if (fail || it.nlist < 0) { named_bar_or(bar_vote, kGroupThreads, fail); break; }
      const int ntiles = it.ntiles();
      if (ntiles == 0) {                                    // no visible key: o = 0, lse = -inf
        if constexpr (!kBlockMax) {
          for (int idx = r; idx < 64 * 16; idx += kGroupThreads) {
            const int qrow = idx >> 4, chunk = idx & 15;
            if (qrow < it.q_valid)
              *reinterpret_cast<uint4*>(o + (((int64_t)it.tok0 + qrow) * m.num_q_heads + it.h) * kHeadDim + chunk * 8) = make_uint4(0u, 0u, 0u, 0u);
          }
          if (lse != nullptr && r < it.q_valid) lse[(int64_t)it.h * lse_stride + it.tok0 + r] = -CUDART_INF_F;
        }
        continue;
      }
      int raw = kBlockMax ? slot_block(it, col_idx, half) : half ? it.first[1] : it.first[0];
      tr.ev(36);
      if constexpr (kBlockMax) {
        int* wmax = reinterpret_cast<int*>(smem + kOffMl + s * kMlBytes);   // [2 tile parities][4 warps]: maxima as order-preserving integers
        float L = row < it.q_valid ? lse[(int64_t)it.h * lse_stride + it.tok0 + row] : 0.f;
        if (!(fabsf(L) < 3.0e38f)) L = 0.f;                 // a query without a key has no probabilities to report
        const float L2 = L * 1.4426950408889634f;
        for (int t = 0; t < ntiles; ++t, ++cnt) {
          const uint32_t buf = cnt & 1u, sbuf = cnt & 3u;
          const int p = 2 * t + half, j = slot_check(it, p, raw);
          raw = slot_block(it, col_idx, p + 2);
          fail = fail || !mbar_wait(sh, bb + S_FULL + (int)sbuf, (cnt >> 2) & 1u, status);
          if (__any_sync(0xffffffffu, fail)) { fail = true; break; }
          tc_fence_after();
          const uint32_t s_addr = tmem + lane_addr + col_s(s, sbuf);
          float mx = j == it.i ? row_max<true>(s_addr, row) : row_max<false>(s_addr, 63);
          if (j < 0 || row >= it.q_valid || !(mx == mx)) mx = -CUDART_INF_F;
          else mx = fmaf(mx, sl2, -L2);
          int key = __float_as_int(mx);
          key ^= (key >> 31) & 0x7fffffff;                  // order-preserving map float -> int
          key = __reduce_max_sync(0xffffffffu, key);
          if (lane == 0) wmax[buf * 4 + quad] = key;
          // this warp is done with the S buffer (four arrivals free it); the two warps of a key block meet to combine
          // their maxima, the group as a whole does not
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(sh.bar(bb + M_TAKEN + (int)sbuf));
          if (named_bar_or(5 + 2 * s + half, 64, false)) { lost = true; break; }
          if ((quad & 1) == 0 && lane == 0 && p < it.nlist) {
            int kx = max(wmax[buf * 4 + quad], wmax[buf * 4 + quad + 1]);
            kx ^= (kx >> 31) & 0x7fffffff;
            block_max[it.l0 + p] = exp2f(__int_as_float(kx));   // 2^(-inf) = 0: no causal pair, or a rejected entry
          }
        }
        if (fail) { named_bar_or(5 + 2 * s + half, 64, true); lost = true; }   // (the neighbour is waiting there, or will)
        if (lost) continue;
        if (lane == 0) mbar_arrive(sh.bar(bb + Q_EMPTY + (int)(nitem & 1u)));
        ++nitem;
        continue;
      }
      float R = kNoRef, l = 0.f;
      for (int t = 0; t < ntiles; ++t, ++cnt) {
        const uint32_t buf = cnt & 1u;
        tr.sample(cnt);
        const int here = raw;                               // (uniform in the warp; -1 past the list's end)
        raw = slot_block(it, col_idx, 2 * t + 2 + half);    // the next tile's list entry: looked at when its turn comes
        tr.ev(31);
        fail = !mbar_wait_warp(sh, bb + S_FULL + (int)buf, (cnt >> 1) & 1u, status);
        if (fail) break;
        tr.ev(32);
        tc_fence_after();
        const uint32_t s_addr = tmem + lane_addr + col_s(s, buf);
        // Each kind of tile to its own end: where the paths join the plain pass's results, or share its registers, every tile pays for them (a
        // launch of 32k tokens 1426 us with all in one, 1240 with the plain pass alone and a call for everything else).  The call is for tiles
        // whose reference moves, which are few.  With it for absent tiles and the diagonal too, lists of a few blocks, which have one in six
        // of these, were slower than with all in one.  The launch by itself, 32 heads, all in one, call for all but the plain pass, and so:
        // one in twenty, 11 584 tokens 142.5, 146.3 and 139.8 us, 16 384 236.1, 238.1 and 235.2; one in ten, 65 536 4291, 4175 and 4134.  48
        // sequences of up to 4, 8, 16 and 30 blocks, one in ten, the whole pass: all in one 109.7, 184.9, 305.1 and 535.6 us, so 108.3, 182.9, 299.8 and 524.6.
        if ((uint32_t)here < (uint32_t)it.i) {              // the plain pass: a block before the diagonal
          if (t == 0) {
            const float mx = row_max<false>(s_addr, 63);
            if (fabsf(mx) < 3.0e38f) R = mx * sl2;
          }
          uint32_t pk[32];
          const float sum = row_pass<false>(s_addr, sl2, R, 63, pk);
          if (!__any_sync(0xffffffffu, !(sum < kRise))) {
            l = __fadd_rn(l, sum);
            tr.ev(33);
            tc_st32(s_addr, pk);                            // P over the scores this thread has read
            tc_wait_st();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(sh.bar(bb + P_FULL + (int)buf));
            tr.ev(34);
            continue;
          }
        }
        if ((uint32_t)here > (uint32_t)it.i) {              // absent (every odd list ends with one) or rejected: contributes nothing
          uint32_t pk[32];
#pragma unroll
          for (int i = 0; i < 32; ++i) pk[i] = 0u;
          tc_st32(s_addr, pk);
          tc_wait_st();
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(sh.bar(bb + P_FULL + (int)buf));
          tr.ev(34);
          continue;
        }
        if (here == it.i) {
          if (t == 0) {
            const float mx = row_max<true>(s_addr, row);
            if (fabsf(mx) < 3.0e38f) R = mx * sl2;
          }
          uint32_t pk[32];
          const float sum = row_pass<true>(s_addr, sl2, R, row, pk);
          if (!__any_sync(0xffffffffu, !(sum < kRise))) {
            l = __fadd_rn(l, sum);
            tr.ev(35);
            tc_st32(s_addr, pk);
            tc_wait_st();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(sh.bar(bb + P_FULL + (int)buf));
            tr.ev(34);
            continue;
          }
        }
        // some row's reference has to move
        const float4 x = other_tile(sh, s_addr, o_addr, sl2, R, l, here == it.i ? row : 63, false, t, bb + PV_DONE + (int)(buf ^ 1u), ((cnt - 1) >> 1) & 1u, status);
        R = x.x; l = x.y; fail = x.z != 0.f;
        if (fail) break;
        __syncwarp();
        if (lane == 0) mbar_arrive(sh.bar(bb + P_FULL + (int)buf));
        tr.ev(40);                                          // (a moved reference)
      }
      if constexpr (!kBlockMax) {
        // ---------------------------------------------------------------------------------------- epilogue: merge, store
        tr.sample(0); tr.ev(36);
        const bool two = it.nlist > 1;                      // the second half has something to contribute
        if (two) st_shared_v2(ml + (uint32_t)r * 8u, __float_as_uint(R), __float_as_uint(l));
        if (named_bar_or(bar_vote, kGroupThreads, fail)) break;
        uint16_t* orow = o + (((int64_t)it.tok0 + row) * m.num_q_heads + it.h) * kHeadDim;
        const uint32_t qbuf = nitem & 1u;
        float sc, lse_row;
        if (two) {
          // out = (2^(R_a - R) O_a + 2^(R_b - R) O_b) / l, R = max(R_a, R_b)
          const float Ro = ld_shared_f32(ml + (uint32_t)(r ^ 64) * 8u), lo = ld_shared_f32(ml + (uint32_t)(r ^ 64) * 8u + 4u);
          const float Rm = fmaxf(R, Ro);
          const float f = l == 0.f ? 0.f : ex2f(R - Rm), fo = lo == 0.f ? 0.f : ex2f(Ro - Rm);
          const float la = __fmul_rn(l, f), lb = __fmul_rn(lo, fo), total = __fadd_rn(la, lb);   // (the same in both threads)
          sc = total > 0.f ? f / total : 0.f;
          lse_row = total > 0.f ? (Rm + log2f(total)) * 0.6931471805599453f : -CUDART_INF_F;
        } else {
          sc = l > 0.f ? 1.f / l : 0.f;
          lse_row = l > 0.f ? (R + log2f(l)) * 0.6931471805599453f : -CUDART_INF_F;
        }
        // The last P V of the item.  A warp whose wait for it is lost keeps the group's barriers and leaves afterwards.  Warps that hand each other
        // partial rows agree on the outcome between their first exchange and their first store: one lost wait and none of them stores.  (A
        // one-block list's rows are each a warp's own.)
        fail = !mbar_wait(sh, bb + PV_DONE + (int)((cnt - 1) & 1u), ((cnt - 1) >> 1) & 1u, status);
        fail = __any_sync(0xffffffffu, fail);
        bool store = row < it.q_valid && !fail;
        tc_fence_after();
        tr.ev(37);
        auto store_lse = [&] { if (half == 0 && lse != nullptr && store) lse[(int64_t)it.h * lse_stride + it.tok0 + row] = lse_row; };
        if (two) {
          // The thread of lane r ends with d columns 64 * half ..: it hands the other 64 of its partial row to lane r ^ 64 through the
          // item's Q buffer (Q has been read: the last S is done), 32 columns at a time, 16-byte chunks XOR (row % 8)
          uint32_t mine[2][32], other[2][32];
          tc_ld32(o_addr + (half ^ 1) * 64, other[0]);
          tc_wait_ld32(other[0]);
          tc_ld32(o_addr + half * 64, mine[0]);
          tc_ld32(o_addr + (half ^ 1) * 64 + 32, other[1]); tc_ld32(o_addr + half * 64 + 32, mine[1]);
          const uint32_t buf = sh.base + (uint32_t)s * kStreamBytes + kStQ + qbuf * kQBytes;
          const uint32_t wr = buf + (uint32_t)r * 128u, rd = buf + (uint32_t)(r ^ 64) * 128u;
          const float2 sc2 = make_float2(sc, sc);
#pragma unroll
          for (int i = 0; i < 2; ++i) {
#pragma unroll
            for (int c = 0; c < 8; ++c) {
              const float2 x = __fmul2_rn(make_float2(__uint_as_float(other[i][4 * c]), __uint_as_float(other[i][4 * c + 1])), sc2);
              const float2 y = __fmul2_rn(make_float2(__uint_as_float(other[i][4 * c + 2]), __uint_as_float(other[i][4 * c + 3])), sc2);
              st_shared_v4(wr + (uint32_t)((c ^ (r & 7)) << 4), __float_as_uint(x.x), __float_as_uint(x.y), __float_as_uint(y.x), __float_as_uint(y.y));
            }
            if (i == 0) { tc_wait_ld32(mine[0]); tc_wait_ld32(other[1]); tc_wait_ld32(mine[1]); }
            named_bar_sync(bar_merge, kGroupThreads);
            uint32_t out[16];
#pragma unroll
            for (int c = 0; c < 8; ++c) {
              const float4 v = ld_shared_f4(rd + (uint32_t)((c ^ (r & 7)) << 4));
              const float2 x = __ffma2_rn(make_float2(__uint_as_float(mine[i][4 * c]), __uint_as_float(mine[i][4 * c + 1])), sc2, make_float2(v.x, v.y));
              const float2 y = __ffma2_rn(make_float2(__uint_as_float(mine[i][4 * c + 2]), __uint_as_float(mine[i][4 * c + 3])), sc2, make_float2(v.z, v.w));
              out[2 * c] = pack_bf16(x.x, x.y);
              out[2 * c + 1] = pack_bf16(y.x, y.y);
            }
            if (i == 0) {                                   // (the vote on the first barrier: short lists 1 to 3 % slower)
              fail = named_bar_or(bar_merge, kGroupThreads, fail);
              store = store && !fail;
              store_lse();
            }
            if (store) {
              const uint32_t o0[8] = {out[0], out[1], out[2], out[3], out[4], out[5], out[6], out[7]};
              const uint32_t o1[8] = {out[8], out[9], out[10], out[11], out[12], out[13], out[14], out[15]};
              st_global_32(orow + half * 64 + i * 32, o0, o32);
              st_global_32(orow + half * 64 + i * 32 + 16, o1, o32);
            }
          }
          fence_async_smem();                               // before the next Q copy into this buffer
        } else if (half == 0) {
          store_lse();
#pragma unroll
          for (int ch = 0; ch < 4; ++ch) {
            uint32_t ov[32];
            tc_ld32(o_addr + ch * 32, ov);
            tc_wait_ld32(ov);
            uint32_t out[16];
#pragma unroll
            for (int c = 0; c < 16; ++c) out[c] = pack_bf16(__uint_as_float(ov[2 * c]) * sc, __uint_as_float(ov[2 * c + 1]) * sc);
            if (store) {
              const uint32_t o0[8] = {out[0], out[1], out[2], out[3], out[4], out[5], out[6], out[7]};
              const uint32_t o1[8] = {out[8], out[9], out[10], out[11], out[12], out[13], out[14], out[15]};
              st_global_32(orow + ch * 32, o0, o32);
              st_global_32(orow + ch * 32 + 16, o1, o32);
            }
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(sh.bar(bb + Q_EMPTY + (int)qbuf));
        ++nitem;
        tr.ev(38);
        if (fail) { named_bar_or(bar_vote, kGroupThreads, true); break; }
      }
    }
  }

  // ------------------------------------------------------------------------------------------------ teardown
  // After a lost wait give copies and MMAs still in flight time to land before shared memory and TMEM go away.
  if (ld_shared_u32(sh.abort_flag()) != 0u)
    for (int i = 0; i < 2000; ++i) __nanosleep(1000);
  tc_fence_before();
  __syncthreads();
  if (kTrace && trace != nullptr && threadIdx.x == 0) { trace[6 * 8192 + blockIdx.x] = global_ns() - cta_t0; trace[6 * 8192 + 256 + blockIdx.x] = (unsigned long long)(clock64() - cta_c0); }  // wall time of this CTA: ns, SM clocks
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
  }
}

using Kernel = void(CUtensorMap, CUtensorMap, CUtensorMap, SeqMeta, const int32_t*, const int32_t*, uint16_t*, float*, int*, unsigned long long*, float*, int*, const int*, int, int, bool);

__global__ void zero_kernel(int* __restrict__ word) {
  grid_wait();
  if (threadIdx.x == 0) *word = 0;
}

// ------------------------------------------------------------------------------------------------ host side
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                                  const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// [T, H, 128] bf16 viewed as (d, head, token); box = 64 d x 1 head x `rows` tokens, 128-byte swizzle, zero fill past T.
static bool make_map(seer_ctx* ctx, CUtensorMap* map, const void* base, int64_t tokens, int heads, uint32_t rows) {
  EncodeTiledFn fn = (EncodeTiledFn)ctx->tmap_encode;
  const cuuint64_t dims[3] = {(cuuint64_t)kHeadDim, (cuuint64_t)heads, (cuuint64_t)tokens};
  const cuuint64_t strides[2] = {(cuuint64_t)kHeadDim * 2, (cuuint64_t)heads * kHeadDim * 2};
  const cuuint32_t box[3] = {64, 1, rows};
  const cuuint32_t estr[3] = {1, 1, 1};
  return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace tc

seer_status init_attn_tc(seer_ctx* ctx) {
  void* fn = nullptr;
  cudaDriverEntryPointQueryResult qres;
  if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &qres) != cudaSuccess || !fn ||
      qres != cudaDriverEntryPointSuccess)
    return SEER_ERR_CUDA;
  ctx->tmap_encode = fn;
  for (tc::Kernel* k : {tc::attn_tc_kernel<false, false>, tc::attn_tc_kernel<false, true>, tc::attn_tc_kernel<true, false>,
                        tc::attn_tc_kernel<false, false, false, false>, tc::attn_tc_kernel<false, true, false, false>,
                        tc::attn_tc_kernel<false, false, true>, tc::attn_tc_kernel<false, true, true>})
    if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)tc::kSmemBytes) != cudaSuccess) return SEER_ERR_CUDA;
  return SEER_OK;
}

int launch_attn_tc(seer_ctx* ctx, const SeqMeta& m, const void* q, const void* k, const void* v,
                    const int32_t* row_ptr, const int32_t* col_idx, void* o, float* lse, int* work_counter,
                    cudaStream_t stream) {
  if (m.q_rows == 0) return 0;
  CUtensorMap mq, mk, mv;
  if (!tc::make_map(ctx, &mq, q, m.total_q_tokens, m.num_q_heads, 64) || !tc::make_map(ctx, &mk, k, m.total_tokens, m.num_kv_heads, 64) ||
      !tc::make_map(ctx, &mv, v, m.total_tokens, m.num_kv_heads, 32))
    return -(int)cudaErrorInvalidValue;
  const unsigned grid = (unsigned)min((int64_t)ctx->num_sms, m.q_rows);
  // The counter the streams draw their work items from lies in the caller's workspace; without one, or with an item a stream at
  // most, the deal is static.  (Its zero by a kernel: a memset would make this launch wait for all that precedes it.)
  cudaError_t e = cudaSuccess;
  int launched = 0;
  if (m.q_rows <= 2 * (int64_t)grid) work_counter = nullptr;
  // Whether pairs of query blocks share their lists is known on the device only.  Asking takes 3.5 to 5 us: the check, and the kernel that then has
  // nothing to do.  The launch without and with it, 32 heads, every block, one in ten, one in twenty: 16 384 tokens 2356 and 2082, 353.5 and 356.3, 226.7
  // and 231.3 us; 13 760 tokens 1685 and 1502, 265.5 and 270.8, 175.4 and 178.1; 8192 tokens 632 and 569, 118.7 and 120.5, 89.4 and 90.7.  Most
  // launches are of sparse lists, and this one loses at most 2 % of them: it is asked from 2^20 causal blocks on (16 384 tokens, 32 heads).
  const bool pairs = work_counter != nullptr && ctx->trace == nullptr && m.score_tiles >= (1 << 20) / (128 * kScoreTile);
  const PairAnswer answer(ctx, m, pairs ? work_counter + 1 : nullptr);
  if (pairs) {
    launched = launch_pair_check(ctx, m, row_ptr, col_idx, work_counter, answer, stream);
    if (launched < 0) return launched;
  } else if (work_counter != nullptr) {
    e = launch_next(tc::zero_kernel, 1, 32, 0, stream, work_counter);
    if (e != cudaSuccess) return -(int)e;
    launched = 1;
  }
  unsigned long long* tb = (unsigned long long*)ctx->trace;
  const bool o32 = ((uintptr_t)o & 31) == 0;
  tc::Kernel* kernel = m.chunked ? (o32 ? tc::attn_tc_kernel<false, true> : tc::attn_tc_kernel<false, true, false, false>)   // (never instrumented)
                     : tb != nullptr ? tc::attn_tc_kernel<true, false>
                     : o32 ? tc::attn_tc_kernel<false, false> : tc::attn_tc_kernel<false, false, false, false>;
  e = launch_next(kernel, grid, tc::kThreads, tc::kSmemBytes, stream, mq, mk, mv, m, row_ptr, col_idx, (uint16_t*)o, lse, ctx->d_status, tb, nullptr, work_counter,
                  (const int*)answer.words, answer.nwords, answer.epoch, false);
  if (e != cudaSuccess) return -(int)e;
  ++launched;
  if (pairs) {
    CUtensorMap mv64;
    if (!tc::make_map(ctx, &mv64, v, m.total_tokens, m.num_kv_heads, 64)) return -(int)cudaErrorInvalidValue;
    const int n = launch_attn_pair(ctx, m, mq, mk, mv64, mv, row_ptr, col_idx, o, lse, work_counter, answer, stream);
    if (n < 0) return n;
    launched += n;
  }
  return launched;
}

// Max-pooled attention map on the listed blocks (Sec. 3.2, Eq. 2): the attention pipeline without V.
int launch_block_max_tc(seer_ctx* ctx, const SeqMeta& m, const void* q, const void* k, const int32_t* row_ptr,
                        const int32_t* col_idx, const float* lse, float* out, cudaStream_t stream) {
  if (m.q_rows == 0) return 0;
  CUtensorMap mq, mk;
  if (!tc::make_map(ctx, &mq, q, m.total_q_tokens, m.num_q_heads, 64) || !tc::make_map(ctx, &mk, k, m.total_tokens, m.num_kv_heads, 64))
    return -(int)cudaErrorInvalidValue;
  const unsigned grid = (unsigned)min((int64_t)ctx->num_sms, m.q_rows);
  float* lse_in = const_cast<float*>(lse);   // read only in this mode
  // From 2^18 causal blocks on (8k tokens, 32 heads) a CTA's share of the work is pairs of query blocks: it takes them by pairs where all of them list the
  // same blocks (block_max_pair.cuh), and otherwise as single blocks.  To ask takes 2 us.  Without and with: 8192 tokens, 32 heads, every block 276 and
  // 197 us, one in eight 45.9 and 46.4, one in twenty 30.6 and 32.7; 16 384 tokens 1146 and 797, one in eight 164 and 160; below, the 2 us weigh more (5824
  // tokens, one in twenty, 19.3), and the map is taken of dense lists above all.  (As a check and a kernel for pairs of their own: 37.7 for the 32.7, 53.3 for the 46.4.)
  const bool pairs = m.score_tiles >= (1 << 18) / (128 * kScoreTile);
  const cudaError_t e = launch_next(m.chunked ? tc::attn_tc_kernel<false, true, true> : tc::attn_tc_kernel<false, false, true>, grid, tc::kThreads, tc::kSmemBytes, stream,
                                    mq, mk, mk, m, row_ptr, col_idx, nullptr, lse_in, ctx->d_status, nullptr, out, nullptr, nullptr, 0, 0, pairs);
  return e == cudaSuccess ? 1 : -(int)e;
}

}  // namespace seer
