// Block-sparse attention forward on the 5th-generation tensor cores (Sec. 3.3):
//   O_i = softmax(Q_i K_{S_i}^T * scale) V_{S_i}
// for every (head, query block i), iterating only the listed key blocks.
//
// Persistent kernel, one CTA per SM, work items (h, i) in head-major order so
// that the CTAs in flight share one head's K/V in L2.  The key tiles of a CTA's
// items form one stream; tile n of the stream belongs to softmax warpgroup
// n & 1 and to S buffer n & 1.  Roles (384 threads, three warpgroups, registers
// rebalanced with setmaxnreg):
//   warps 0, 2  TMA producers, one lane each: warp 0 streams the items' Q tiles
//               and the K tiles, warp 2 the V tiles, K and V each into a 3-stage
//               ring of 128B-swizzled shared tiles.  A K stage is released by
//               the MMA that consumed it (S = Q K^T), a V stage by O += P V.
//   warp 1      TMEM owner and MMA issuer: O += P_u V_u (P from TMEM, V from
//               shared memory), then S_{u+2} = Q K_{u+2}^T (Q from TMEM, K from
//               shared memory) into the buffer P_u was just read from.
//   warps 4-11  two softmax warpgroups, thread = query row = TMEM lane.  Per
//               tile: read S from TMEM, mask the ragged last key block, keep a
//               running row maximum (rescaling O in TMEM only when the maximum
//               grew by more than 2^8, so the exponentials stay bounded), write
//               P as bf16 pairs over the columns of S it was computed from, in
//               two halves so that P V starts after the first.
// What bounds it, and why this split: the two 128 x 128 x 128 products of a key
// tile take 1,024 cycles, one warpgroup's serial pass over a tile (barrier, TMEM
// load, maximum, 128 exponentials a thread at 8 a cycle and quarter, store,
// barrier) about 1,700.  With one warpgroup the launch ran at that pace (a clock
// trace: 1,720 cycles per tile); two of them on alternate tiles overlap one
// pass with the other's and with the products.  The row maximum goes from tile
// to tile through shared memory (each tile's warp publishes it before the
// exponentials, the warp of the next tile reads it), so the rescaling rule and
// P are those of one pass in tile order; each warpgroup sums its own tiles' row
// normalisers and the two are added at the end of the item.
// P over S leaves 64 TMEM columns: they double-buffer Q, so the next item's
// first S follows the current item's last but one P V without a gap.
// Reading Q from TMEM halves the shared-memory operand traffic of S = Q K^T;
// per key block the shared memory then serves K and V to the tensor core and
// their TMA writes (128 KB), about what the two products take.
// TMEM columns: S0 [0,128), S1 [128,256) (P over the first 64 of each),
// O [256,256+D), Q [384,384+D/2) and [448,448+D/2).
// Measured against one warpgroup, same clocks: 2048 canvas, Top-K 0.12, 7,545 ->
// 7,384 us in a loop (6,972 -> 6,783 after a pause: in a loop the card is at its
// 1.4 kW cap, and what the kernel gains in cycles the clock gives back, 1,815 ->
// 1,732 MHz); d = 64 forward and backward at 512 418 -> 398 us.  With the two
// producers apart (below) 7,130 and 6,350 us at 2048, 203 -> 193 at 512.
// Blocks of 64 rows (b_q or b_kv) are served by the same 128 x 128 tiles:
//   b_kv = 64:  two listed 64-row key blocks fill one 128-row key tile (two
//               TMA boxes per operand, PairList): consecutive entries of the
//               list for b_q = 128 (nothing discarded), the two 64-row query
//               blocks' lists in lockstep for b_q = 64 (rows 0-63 see the low
//               half of the tile, rows 64-127 the high half);
//   b_q = 64, b_kv = 128:  the item's two lists are merged into 128-row key
//               tiles with a mask of the listed 64 x 64 sub-blocks (TileList).
// The softmax sets the scores of sub-blocks a row does not see to -inf.  Rows
// that see no key end with O = 0 and LSE = -inf.
// Every wait is bounded; on expiry the kernel records UT_ERR_TIMEOUT,
// drains its own copies and MMAs, frees TMEM and returns.
#include "common.cuh"
#include "kernels.h"

namespace ut {

constexpr int kBM = 128;  // query rows per tile
constexpr int kBN = 128;  // key rows per tile
constexpr int kFwdThreads = 384;
// registers per thread after setmaxnreg: control warpgroup and the two softmax
// warpgroups; the sum is what the launch allocates (3 x 168), so every
// increase is covered by the decrease
constexpr int kFwdRegLaunch = 168, kFwdRegCtl = 88, kFwdRegSm = 208;
static_assert(kFwdRegCtl + 2 * kFwdRegSm == 3 * kFwdRegLaunch, "setmaxnreg split must match the launch");
constexpr int kStages = 3;                       // K and V ring depth
constexpr int kRowSlots = 8;                     // key tiles whose row counts are kept
constexpr uint32_t kTileChunkBytes = 128 * 128;  // 128 rows x 128 bytes (64 bf16)
constexpr uint32_t kColO = 256, kColQ = 384;     // TMEM column bases (Q: two buffers of 64 columns)

// Static schedule of lists of unequal length.  Dealt out in index order, round
// by round, the busiest of 152 CTAs has 244 steps against a mean of 199 at the
// 512 canvas (structured lists, reference kept in full) and up to 1.8 times the
// mean on smaller ones.  The entry point has no workspace for a common counter
// or order, so every CTA computes the same order for itself, in its still unused
// K ring: items by length, longest first, equal ones by index, dealt out
// boustrophedon (202 steps there).  Only where it pays: a few items per CTA
// (the more there are the better index order evens out; the scratch holds 4,096
// in all), index order at least 5% off the mean, 128-row blocks on both sides, and
// K and V of all heads within 96 MiB, since the order gives up that neighbours
// share a head in L2.  512 canvas: 219 -> 207 us when it
// was made (193 now).  Sorted against index order, d = 128, 24 heads, lists of
// 20%, K + V of 59 / 91 / 105 / 117 / 152 / 199 MiB: lists that differ by chance
// only 0.94 / 0.97 / 1.01 / 1.03 / 1.11 / 1.11 of the time, lists of which some
// are six times as long 0.70 / 0.73 / 0.66 / 0.80 / 0.75 / 0.82: the line is where
// the first kind stops gaining.
constexpr int kSortItems = 4096, kSortBins = 1024, kSortRounds = 32;
constexpr int64_t kSortKvBytes = 96ll << 20;
struct FwdSort {
  uint16_t length[kSortItems];
  uint16_t bin[kSortItems];  // 0: the longest
  int32_t start[kSortBins];  // entries per bin, then the rank of its first item
  int32_t longest, busiest, total;
};

template <int D>
struct FwdSmem {
  static constexpr int kChunks = D / 64;
  static constexpr uint32_t kQBytes = kBM * D * 2;
  static constexpr uint32_t kKVBytes = kBN * D * 2;
  alignas(1024) uint8_t q[kQBytes];
  alignas(1024) uint8_t k[kStages][kKVBytes];
  alignas(1024) uint8_t v[kStages][kKVBytes];
  // shared Q tile: TMA landed, by item & 1 (a warpgroup may pass over one item
  // without waiting for its Q, never over two, so it always waits for the phase
  // after one it knows to be complete) / copied into TMEM
  uint64_t q_full[2], q_empty;
  uint64_t qt_full[2];         // TMEM Q written by the softmax warps, by item & 1
  uint64_t k_full[kStages], v_full[kStages], k_empty[kStages], v_empty[kStages];
  uint64_t s_full[2];          // S tile in its buffer
  uint64_t p_full[2][2];       // [buffer][half of the key columns]
  uint64_t pv_done[2];         // O += P V of a tile finished, by tile & 1
  uint64_t o_empty, mma_done;
  uint64_t m_full[2][4];       // [tile & 1][lane quarter]: row maxima published
  uint64_t l_full[2][4];       // [item & 1][lane quarter]: the other warpgroup's normalisers
  // existing rows of the key tiles, by tile % kRowSlots (128-row blocks).  The K
  // producer is at most three tiles ahead of S and S two ahead of P V, whose P
  // needs the row maxima of every tile before it: a slot is read long before
  // it is written again.
  int32_t k_rows[kRowSlots];
  int32_t mine[kSortRounds];   // this CTA's items, where they are sorted
  // row maximum used by tile (tile & 1): tile n + 2 writes it after its warp has read
  // the maximum of tile n + 1, published after that tile's warp had read tile n's
  float m_row[2][kBM];
  // normaliser handed over, per item & 1.  Item i + 2's comes after item i's was
  // read: since item i the warpgroup that hands over has either finished item i +
  // 1, and waited there for the other's half, handed over after the epilogue of
  // item i; or the other finished item i + 1 too, and the first tile of item i + 2,
  // here, has waited for the maximum of that item's last tile, published after it.
  float l_row[2][kBM];
  uint32_t tmem_base;
  int abort_flag;
};

struct FwdParams {
  const int32_t* row_ptr;   // fine lists: nq_fine rows per head
  const int32_t* col_idx;
  int nq_fine;              // query blocks per head in the lists
  int q_rows_per_tile;      // 1 (b_q = 128) or 2 (b_q = 64)
  int list_shift;           // 0 (b_kv = 128) or 1 (b_kv = 64)
  __nv_bfloat16* o;
  float* lse;
  int32_t* status;
  int64_t N;
  int64_t rs;  // elements between tokens
  int H, nq;         // nq: 128-row query tiles per head
  int n_items;
  float scale_log2;  // softmax scale * log2(e)
  uint64_t timeout_ns;
};

// Fills mine[] with this CTA's items, longest first over all CTAs; false (in
// every CTA alike) if index order is even enough.  All threads call it.
UT_DEV bool sort_items(const FwdParams& prm, FwdSort& st, int32_t* mine) {
  const int n = prm.n_items, G = gridDim.x, tid = threadIdx.x;
  if (tid == 0) st.longest = st.busiest = st.total = 0;
  for (int b = tid; b < kSortBins; b += kFwdThreads) st.start[b] = 0;
  __syncthreads();
  int mx = 0;
  for (int x = tid; x < n; x += kFwdThreads) {  // listed blocks of item x
    const int len = min(65535, prm.row_ptr[x + 1] - prm.row_ptr[x]);
    st.length[x] = (uint16_t)len;
    mx = max(mx, len);
  }
  atomicMax(&st.longest, mx);
  __syncthreads();
  for (int b = tid; b < G; b += kFwdThreads) {
    int sum = 0;
    for (int x = b; x < n; x += G) sum += st.length[x];
    atomicMax(&st.busiest, sum);
    atomicAdd(&st.total, sum);
  }
  __syncthreads();
  if ((int64_t)st.busiest * G * 20 <= (int64_t)st.total * 21) return false;
  const uint32_t longest = (uint32_t)max(1, st.longest);
  for (int x = tid; x < n; x += kFwdThreads) {
    const uint32_t b = (kSortBins - 1) - st.length[x] * (uint32_t)(kSortBins - 1) / longest;
    st.bin[x] = (uint16_t)b;
    atomicAdd(&st.start[b], 1);
  }
  __syncthreads();
  const int lane = tid & 31;
  if (tid < 32) {  // exclusive prefix, 32 bins a lane
    int c[kSortBins / 32], local = 0;
#pragma unroll
    for (int e = 0; e < kSortBins / 32; ++e) {
      c[e] = st.start[lane * (kSortBins / 32) + e];
      local += c[e];
    }
    int run = local;
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, run, o);
      if (lane >= o) run += v;
    }
    run -= local;
#pragma unroll
    for (int e = 0; e < kSortBins / 32; ++e) {
      st.start[lane * (kSortBins / 32) + e] = run;
      run += c[e];
    }
  }
  __syncthreads();
  for (int k = tid >> 5; k < kSortRounds; k += kFwdThreads / 32) {  // a warp finds the item of one round
    int rank = k * G + (k & 1 ? G - 1 - (int)blockIdx.x : (int)blockIdx.x);
    if (rank >= n) continue;
    int lo = 0, hi = kSortBins - 1;  // the last bin that starts at or before the rank
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (st.start[mid] <= rank) lo = mid;
      else hi = mid - 1;
    }
    rank -= st.start[lo];
    for (int x0 = 0; x0 < n; x0 += 32) {
      const uint32_t m = __ballot_sync(0xffffffffu, x0 + lane < n && st.bin[x0 + lane] == lo);
      if (rank < __popc(m)) {
        if ((m >> lane & 1u) && __popc(m & ((1u << lane) - 1u)) == rank) mine[k] = x0 + lane;
        break;
      }
      rank -= __popc(m);
    }
  }
  return true;
}

template <int D, int kMode, bool kSort>  // kSort: sizes allow the sorted schedule
__global__ void __launch_bounds__(kFwdThreads, 1)
    attn_fwd_tc_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k,
                       const __grid_constant__ CUtensorMap tm_v, const __grid_constant__ CUtensorMap tm_k64,
                       const __grid_constant__ CUtensorMap tm_v64, const FwdParams prm) {
  constexpr bool kSub = kMode != 0;  // 64-row blocks on at least one side
  // Exponentials ahead of the tile's maximum (below): they pay where the two
  // products are as long as the softmax (d = 128: 7,597 -> 7,411 us at the 2048
  // canvas); with d = 64, and with halves that a row may not see, the maximum
  // first is faster (d = 64 training layer 397 against 408 us, 64-row blocks
  // 13.2 against 14.0 ms), since the exponentials then do not stand between one
  // tile's maximum and the next's.
  constexpr bool kAhead = kMode == 0 && D == 128;
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  FwdSmem<D>& sm = *reinterpret_cast<FwdSmem<D>*>(smem_raw);
  constexpr int C = FwdSmem<D>::kChunks;
  const uint32_t warp = warp_id();
  const uint32_t lane = lane_id();
  volatile int* abort_flag = &sm.abort_flag;
  if ((smem_u32(smem_raw) & 1023u) != 0) {
    if (threadIdx.x == 0) set_status(prm.status, UT_ERR_INVALID_ARG);
    return;
  }

  if (threadIdx.x == 0) {
    mbar_init(&sm.q_full[0], 1);
    mbar_init(&sm.q_full[1], 1);
    mbar_init(&sm.q_empty, 4);
    mbar_init(&sm.qt_full[0], 4);
    mbar_init(&sm.qt_full[1], 4);
    for (int s = 0; s < kStages; ++s) {
      mbar_init(&sm.k_full[s], 1);
      mbar_init(&sm.v_full[s], 1);
      mbar_init(&sm.k_empty[s], 1);
      mbar_init(&sm.v_empty[s], 1);
    }
    for (int s = 0; s < 2; ++s) {
      mbar_init(&sm.s_full[s], 1);
      mbar_init(&sm.pv_done[s], 1);
      mbar_init(&sm.p_full[s][0], 4);
      mbar_init(&sm.p_full[s][1], 4);
      for (int x = 0; x < 4; ++x) {
        mbar_init(&sm.m_full[s][x], 1);
        mbar_init(&sm.l_full[s][x], 1);
      }
    }
    mbar_init(&sm.o_empty, 4);
    mbar_init(&sm.mma_done, 1);
    sm.abort_flag = 0;
    fence_barrier_init();
  }
  if (warp == 1) {
    tmem_alloc(&sm.tmem_base, 512);
    tmem_relinquish();
  }
  const int G = gridDim.x;
  bool sorted = false;
  if constexpr (kSort) {
    const int in_order = !sort_items(prm, *reinterpret_cast<FwdSort*>(&sm.k[0][0]), sm.mine);
    fence_proxy_async_smem();  // the K ring is written by TMA next
    sorted = uniform(in_order) == 0;
  }
  // this CTA's items: first_item(k), then next_item(w, k) until n_items or more
  auto item_at = [&](int k) -> int {
    if (!sorted) return blockIdx.x + k * G;
    return k * G + (k & 1 ? G - 1 - (int)blockIdx.x : (int)blockIdx.x) < prm.n_items && k < kSortRounds ? sm.mine[k]
                                                                                                        : prm.n_items;
  };
  auto first_item = [&](int& k) -> int {
    k = 0;
    if constexpr (kSort) return item_at(0);
    else return blockIdx.x;
  };
  auto next_item = [&](int w, int& k) -> int {
    if constexpr (kSort) return item_at(++k);
    else return w + G;
  };
  // with items from shared memory the compiler has to be told what is uniform
  auto same = [](auto x) {
    if constexpr (kSort) return uniform(x);
    else return x;
  };
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = sm.tmem_base;

  if (warp < 4) {
  setmaxnreg_dec<kFwdRegCtl>();
  if (warp == 0 || warp == 2) {
    // ----------------------------------------------------------- producers
    // Warp 0 streams Q and K, warp 2 streams V, one lane each: each ring is
    // released by the MMA that consumes it (K after S = Q K^T, V after O += P V),
    // so neither waits for the other.  As two lanes of one warp they did, wherever
    // the compiler let the lanes meet again: 7,780 tokens, 24 heads, lists of 20%
    // 139.6 -> 129.8 us, 512 canvas with d = 64 117 -> 111, 64-row blocks 2,360 ->
    // 2,234 (85,202 tokens, 4 heads); a branch on the lane in the loop made it
    // 20% slower.
    if (lane == 0) {
      const bool is_k = warp == 0;
      if (is_k) {
        tma_prefetch_desc(&tm_q);
        tma_prefetch_desc(&tm_k);
        if (kMode >= 2) tma_prefetch_desc(&tm_k64);
      } else {
        tma_prefetch_desc(&tm_v);
        if (kMode >= 2) tma_prefetch_desc(&tm_v64);
      }
      const uint64_t pol_kv = policy_evict_last();
      const uint64_t pol_q = policy_evict_first();
      uint64_t* full = is_k ? sm.k_full : sm.v_full;
      uint64_t* empty = is_k ? sm.k_empty : sm.v_empty;
      uint8_t* ring = is_k ? &sm.k[0][0] : &sm.v[0][0];
      const void* tmap = is_k ? static_cast<const void*>(&tm_k) : static_cast<const void*>(&tm_v);
      const void* tmap64 = is_k ? static_cast<const void*>(&tm_k64) : static_cast<const void*>(&tm_v64);
      uint32_t qi = 0, kv = 0;
      const int cut_block = prm.N % kBN ? prm.nq - 1 : -1;
      bool ok = true;
      int k;
      for (int w = first_item(k); w < prm.n_items && ok; w = next_item(w, k)) {
        const int h = w / prm.nq, i = w % prm.nq;
        BlockSteps<kMode> tl;
        tl.init(prm.row_ptr, prm.col_idx, h, i, prm.nq_fine, prm.q_rows_per_tile, prm.list_shift);
        if (tl.empty()) continue;
        if (is_k) {
          if (!(ok = mbar_wait(&sm.q_empty, (qi & 1) ^ 1, abort_flag, prm.status, prm.timeout_ns))) break;
          mbar_expect_tx(&sm.q_full[qi & 1], FwdSmem<D>::kQBytes);
          for (int c = 0; c < C; ++c)
            tma_load_2d(sm.q + c * kTileChunkBytes, &tm_q, &sm.q_full[qi & 1], h * D + c * 64, i * kBM, pol_q);
          ++qi;
        }
        int j, jh;
        uint32_t bits;
        bool held = false;  // 128-row blocks: the block that N cuts off, met before the end of the list
        for (; tl.next(j, jh, bits); ++kv) {
          const uint32_t st = kv % kStages, n = kv / kStages;
          if (kMode == 0) {
            // lists in any order: that block changes places with the last one, so
            // that the softmax warps mask columns in an item's last tile only
            const bool last = tl.tl.pa == tl.tl.na;
            if (last && held) j = cut_block;
            else if (!last && j == cut_block) {
              held = true;
              j = tl.tl.a[tl.tl.na - 1];
            }
          }
          if (!(ok = mbar_wait(&empty[st], (n & 1) ^ 1, abort_flag, prm.status, prm.timeout_ns))) break;
          if (kMode == 0 && is_k)
            *const_cast<volatile int*>(&sm.k_rows[kv % kRowSlots]) = j == cut_block ? (int)(prm.N % kBN) : kBN;
          mbar_expect_tx(&full[st], FwdSmem<D>::kKVBytes);
          uint8_t* dst = ring + st * FwdSmem<D>::kKVBytes;
          if (tl.pair) {  // two 64-row boxes: rows 0-63 and 64-127 of each 128-row sub-tile
            const int b0 = PairList::load_lo(j, jh), b1 = PairList::load_hi(j, jh);
            for (int c = 0; c < C; ++c) {
              tma_load_2d(dst + c * kTileChunkBytes, tmap64, &full[st], h * D + c * 64, b0 * 64, pol_kv);
              tma_load_2d(dst + c * kTileChunkBytes + 64 * 128, tmap64, &full[st], h * D + c * 64, b1 * 64, pol_kv);
            }
          } else {
            for (int c = 0; c < C; ++c)
              tma_load_2d(dst + c * kTileChunkBytes, tmap, &full[st], h * D + c * 64, j * kBN, pol_kv);
          }
        }
      }
      // Drain: every copy this thread issued has landed before the CTA may exit.
      auto drain = [&](uint64_t* bar, uint32_t parity) {
        if (!mbar_drain(bar, parity, kDrainTimeoutNs)) set_status(prm.status, UT_ERR_TIMEOUT);
      };
      if (qi > 0) drain(&sm.q_full[(qi - 1) & 1], ((qi - 1) >> 1) & 1);
      for (uint32_t u = (kv >= kStages ? kv - kStages : 0); u < kv; ++u)
        drain(&full[u % kStages], (u / kStages) & 1);
    }
  } else if (warp == 1) {
    // ---------------------------------------------------------- MMA issuer
    // The whole warp runs this loop converged; every MMA and commit is issued
    // by one elected lane (see mma_bf16_ss_w), waits are warp-uniform.
    // S runs two tiles ahead of P V over the stream of tiles.  S_{u+2} needs no
    // wait for its buffer: it is issued after P V_u, the last reader, and MMAs
    // of one thread execute in order.
    constexpr uint32_t idesc_s = idesc_bf16_f32(kBM, kBN, false, false);
    constexpr uint32_t idesc_o = idesc_bf16_f32(kBM, D, false, true);
    uint32_t sc = 0, pc = 0;  // tiles of the stream: S issued, P V issued
    uint32_t qi = 0, oi = 0;  // items: S started, P V started
    uint32_t firsts = 0;      // bit (tile & 3): the tile is the first of its item
    bool ok = true;
    // item of the S cursor: index, round, tiles, next tile; the list bounds of the
    // following item are loaded an item ahead (128-row blocks)
    int ck, cw = same(first_item(ck)), cL = 0, ct = 0;
    int n_lo = 0, n_hi = 0;
    auto load_bounds = [&](int w) {
      if (kMode == 0 && w < prm.n_items) {
        n_lo = prm.row_ptr[w];
        n_hi = prm.row_ptr[w + 1];
      }
    };
    auto count_from = [&]() {  // cw, cL: the first item from cw on that lists something (cL = 0: none)
      for (cL = 0; same(cw < prm.n_items); cw = same(next_item(cw, ck))) {
        if (kMode == 0) {
          cL = same(n_hi - n_lo);
          int k = ck;
          load_bounds(same(next_item(cw, k)));
        } else {
          BlockSteps<kMode> tl;
          tl.init(prm.row_ptr, prm.col_idx, cw / prm.nq, cw % prm.nq, prm.nq_fine, prm.q_rows_per_tile,
                  prm.list_shift);
          cL = tl.count_warp();
        }
        if (same(cL > 0)) return;
      }
      cL = 0;
    };
    auto wait_k = [&]() -> bool {  // K of the next S tile in its stage
      return warp_wait(&sm.k_full[sc % kStages], (sc / kStages) & 1, abort_flag, prm.status, prm.timeout_ns);
    };
    auto issue_s = [&]() -> bool {
      sc = same((int)sc);
      qi = same((int)qi);
      const uint32_t st = sc % kStages, sb = sc & 1;
      const bool first = same(ct == 0);
      if (first && !warp_wait(&sm.qt_full[qi & 1], (qi >> 1) & 1, abort_flag, prm.status, prm.timeout_ns)) return false;
      if (same(sc < 2) && !wait_k()) return false;
      tc_fence_after();
      const uint32_t k_addr = smem_u32(sm.k[st]);
      const uint32_t q_col = tmem + kColQ + (qi & 1) * 64;
#pragma unroll
      for (int kk = 0; kk < D / 16; ++kk) {
        const uint32_t off = (kk >> 2) * kTileChunkBytes + (kk & 3) * 32;
        mma_bf16_ts_w(tmem + sb * 128, q_col + kk * 8, sdesc_sw128(k_addr + off, 16, 1024), idesc_s, kk > 0);
      }
      mma_commit_w(&sm.s_full[sb]);
      mma_commit_w(&sm.k_empty[st]);
      firsts = (firsts & ~(1u << (sc & 3))) | ((first ? 1u : 0u) << (sc & 3));
      ++sc;
      if (same(++ct == cL)) {
        cw = same(next_item(cw, ck));
        ct = 0;
        ++qi;
        count_from();
      }
      return true;
    };
    auto issue_pv = [&]() -> bool {
      pc = same((int)pc);
      const uint32_t st = pc % kStages, n = pc / kStages, sb = pc & 1, ph = (pc >> 1) & 1;
      const bool first = same(((firsts >> (pc & 3)) & 1u) != 0);
      if (!warp_wait(&sm.v_full[st], n & 1, abort_flag, prm.status, prm.timeout_ns)) return false;
      if (first) {  // O is free once the previous item's was read
        if (!warp_wait(&sm.o_empty, (oi & 1) ^ 1, abort_flag, prm.status, prm.timeout_ns)) return false;
        ++oi;
      }
      // K of the S tile that follows: ready long before P, and waited for here
      // it does not stand between P V and S
      if (same(cL > 0) && !wait_k()) return false;
      const uint32_t v_addr = smem_u32(sm.v[st]);
#pragma unroll
      for (int hc = 0; hc < 2; ++hc) {
        if (!warp_wait(&sm.p_full[sb][hc], ph, abort_flag, prm.status, prm.timeout_ns)) return false;
        tc_fence_after();
#pragma unroll
        for (int kk = hc * (kBN / 32); kk < (hc + 1) * (kBN / 32); ++kk)
          mma_bf16_ts_w(tmem + kColO, tmem + sb * 128 + kk * 8, sdesc_sw128(v_addr + kk * 2048, kTileChunkBytes, 1024),
                        idesc_o, (!first || kk > 0));
      }
      mma_commit_w(&sm.pv_done[sb]);
      mma_commit_w(&sm.v_empty[st]);
      ++pc;
      return true;
    };
    load_bounds(cw);
    count_from();
    for (int x = 0; x < 2 && same(ok && cL > 0); ++x) ok = issue_s();
    while (same(ok && pc < sc)) {
      if (!(ok = issue_pv())) break;
      if (same(cL > 0)) ok = issue_s();
    }
    // Drain: all MMAs issued by this warp complete before TMEM is freed.
    mma_commit_w(&sm.mma_done);
    if (!mbar_drain(&sm.mma_done, 0, kDrainTimeoutNs)) set_status(prm.status, UT_ERR_TIMEOUT);
  }
  } else {
    setmaxnreg_inc<kFwdRegSm>();
    // ------------------------------------------------------------- softmax
    const uint32_t wgi = (warp >> 2) - 1;  // warpgroup 0 / 1: even / odd tiles of the stream
    const uint32_t quarter = warp & 3;
    const uint32_t row = quarter * 32 + lane;
    const uint32_t lane_base = (quarter * 32) << 16;
    const float c = prm.scale_log2;
    uint32_t sc0 = 0, it = 0;  // tiles and (non-empty) items so far
    bool ok = true;
    const uint32_t rh = row >> 6;  // which 64-row half of the query tile
    // Q tile of an item: shared memory (128B-swizzled, as TMA wrote it) ->
    // registers -> TMEM, this thread's row, bf16 pairs (element 2u in the low
    // half of column u), the A-operand layout of S = Q K^T.  The buffer was
    // last read by item it - 2, whose S this warpgroup's previous tile
    // (or a later one) has waited for.
    auto load_q = [&]() -> bool {
      if (!warp_wait(&sm.q_full[it & 1], (it >> 1) & 1, abort_flag, prm.status, prm.timeout_ns)) return false;
      tc_fence_after();
#pragma unroll
      for (int cc = 0; cc < C; ++cc) {
        uint32_t qv[32];
        const uint32_t base = smem_u32(sm.q) + cc * kTileChunkBytes + row * 128;
#pragma unroll
        for (int u = 0; u < 8; ++u)
          asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];"
                       : "=r"(qv[4 * u]), "=r"(qv[4 * u + 1]), "=r"(qv[4 * u + 2]), "=r"(qv[4 * u + 3])
                       : "r"(base + ((u ^ (row & 7)) << 4)));
        tmem_st32(tmem + lane_base + kColQ + (it & 1) * 64 + cc * 32, qv);
      }
      tmem_wait_st();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) {
        mbar_arrive(&sm.qt_full[it & 1]);
        mbar_arrive(&sm.q_empty);
      }
      return true;
    };
    int k;
    for (int w = same(first_item(k)); w < prm.n_items && ok; w = same(next_item(w, k))) {
      const int h = w / prm.nq, i = w % prm.nq;
      BlockSteps<kMode> tl;
      tl.init(prm.row_ptr, prm.col_idx, h, i, prm.nq_fine, prm.q_rows_per_tile, prm.list_shift);
      const int L = same(tl.count_warp());
      const int64_t grow = (int64_t)i * kBM + row;
      const bool row_ok = grow < prm.N;
      __nv_bfloat16* orow = prm.o + grow * prm.rs + (int64_t)h * D;
      if (L <= 0) {
        if (wgi == 0 && row_ok) {
          for (int e = 0; e < D; e += 8) *reinterpret_cast<uint4*>(orow + e) = make_uint4(0, 0, 0, 0);
          prm.lse[(int64_t)h * prm.N + grow] = -INFINITY;
        }
        continue;
      }
      const uint32_t t0 = (sc0 ^ wgi) & 1;  // this warpgroup's first tile of the item
      if (t0 == 0 && !(ok = load_q())) break;
      int j = 0, jh = -1;
      uint32_t bits = 15u;
      if (kMode != 0 && t0) tl.next(j, jh, bits);
      float m_before = 0.f;  // the maximum the previous tile of the stream used
      float m = 0.f, l = 0.f;  // row maximum in use and this warpgroup's part of the normaliser under it
      for (int t = t0; t < L; t += 2) {
        if (kMode != 0) {
          if (t > (int)t0) tl.next(j, jh, bits);  // the other warpgroup's tile
          tl.next(j, jh, bits);
        }
        const uint32_t sc = sc0 + t, sb = sc & 1, ns = sc >> 1;
        const uint32_t s_col = tmem + lane_base + sb * 128;
        if (!(ok = warp_wait(&sm.s_full[sb], ns & 1, abort_flag, prm.status, prm.timeout_ns))) break;
        tc_fence_after();
        // ragged last key block: columns past N do not exist.  They are set to
        // -inf in TMEM, in a short loop: selects on all 128 registers, skipped
        // or not, sit in the middle of every tile's instruction stream.
        if (kMode != 0 || t == L - 1) {
          const int e0 = tl.pair ? 64 : kBN;  // columns that belong to the low (or only) listed block
          int64_t nv0, nv1 = 64;
          if constexpr (kMode == 0) {
            nv0 = *const_cast<volatile int*>(&sm.k_rows[sc % kRowSlots]);
          } else {
            nv0 = prm.N - (tl.pair ? 64 * (int64_t)PairList::load_lo(j, jh) : (int64_t)j * kBN);
            nv1 = tl.pair ? prm.N - 64 * (int64_t)PairList::load_hi(j, jh) : 64;
          }
          if (__builtin_expect(nv0 < e0 || nv1 < 64, 0)) {
            for (int x = (int)nv0; x < e0; ++x) tmem_st1(s_col + x, 0xff800000u);
            for (int x = (int)nv1; x < 64; ++x) tmem_st1(s_col + 64 + x, 0xff800000u);
            tmem_wait_st();
          }
        }
        // the maximum that the previous tile used, from its warp (waited for on
        // an item's first tile too: it also says that the slot written below
        // was read)
        float m_new = -INFINITY;
        auto previous_max = [&]() -> bool {
          if (sc > 0 && !warp_wait(&sm.m_full[(sc - 1) & 1][quarter], ((sc - 1) >> 1) & 1, abort_flag, prm.status,
                                   prm.timeout_ns))
            return false;
          if (t > 0) m_new = m_before = *const_cast<volatile float*>(&sm.m_row[(sc - 1) & 1][row]);
          return true;
        };
        // all four 32-column loads in flight before one wait
        uint32_t r[kBN];
#pragma unroll
        for (int g = 0; g < kBN / 32; ++g) tmem_ld32(s_col + g * 32, *reinterpret_cast<uint32_t(*)[32]>(&r[g * 32]));
        if (kAhead) ok = previous_max();
        tmem_wait_ld();  // also when that wait gave up: the loads must not land in registers or TMEM reused since
        if (!ok) break;
        float s[kBN];
#pragma unroll
        for (int x = 0; x < kBN; ++x) s[x] = __uint_as_float(r[x]);
        // 64-column halves of the tile not listed for this row's half do not
        // count (the same for the whole warp: rh is per warp)
        const uint32_t cols = kSub ? (bits >> (2 * rh)) & 3u : 3u;
        // P = exp2(s * c - m) of one half's 64 columns, rounded to bf16 for the
        // P V MMA, and its part of the normaliser
        float2 l4[4] = {{0.f, 0.f}, {0.f, 0.f}, {0.f, 0.f}, {0.f, 0.f}};
        uint32_t pk[kBN / 4];
        auto exp_pair = [&](int hc, int x) {
          const float2 e = ffma2(make_float2(s[hc * 64 + x], s[hc * 64 + x + 1]), make_float2(c, c),
                                 make_float2(-m_new, -m_new));
          const float2 p = make_float2(ex2_approx(e.x), ex2_approx(e.y));
          l4[(x >> 1) & 3] = add2(l4[(x >> 1) & 3], p);
          pk[x / 2] = pack_bf16x2(p.x, p.y);
        };
        auto exp_half = [&](int hc) {
          if (kSub && !((cols >> hc) & 1u)) {  // a masked half: P = 0 without the exponentials
#pragma unroll
            for (int x = 0; x < kBN / 4; ++x) pk[x] = 0u;
          } else {
#pragma unroll
            for (int x = 0; x < kBN / 2; x += 2) exp_pair(hc, x);
          }
        };
        // Row maximum, eight chains of three-input maxima.  Ahead: the first
        // half of P is computed under the previous tile's maximum in the same
        // instructions' shadow (exponentials and maxima run on different
        // units) and done over in the rare tile that has to raise it, and in an
        // item's first (m_new = -inf).
        float mx = -INFINITY;
        {
          float m8[8];
#pragma unroll
          for (int q = 0; q < 8; ++q) m8[q] = -INFINITY;
          if constexpr (kAhead) {
#pragma unroll
            for (int x = 0; x < kBN / 2; x += 2) {
              exp_pair(0, x);
              m8[(x >> 1) & 3] = max3(m8[(x >> 1) & 3], s[x], s[x + 1]);
              m8[4 + ((x >> 1) & 3)] = max3(m8[4 + ((x >> 1) & 3)], s[64 + x], s[64 + x + 1]);
            }
          } else {
#pragma unroll
            for (int hc = 0; hc < 2; ++hc) {
              if (kSub && !((cols >> hc) & 1u)) continue;
#pragma unroll
              for (int x = 0; x < kBN / 2; x += 16)
#pragma unroll
                for (int q = 0; q < 8; ++q) m8[q] = max3(m8[q], s[hc * 64 + x + q], s[hc * 64 + x + q + 8]);
            }
          }
          mx = max3(max3(m8[0], m8[1], m8[2]), max3(m8[3], m8[4], m8[5]), fmaxf(m8[6], m8[7]));
        }
        // a row may see nothing in this tile: keep the reference maximum
        // finite so that exp2(-inf - m) stays 0 (not NaN)
        mx = kSub ? fmaxf(mx * c, -1e30f) : mx * c;
        if (!kAhead && !(ok = previous_max())) break;
        const bool need = t == 0 || mx > m_new + 8.0f;
        if (__builtin_expect(__any_sync(0xffffffffu, need), 0)) {
          if (t > 0) {
            // O holds P V up to the previous tile once that MMA finished
            if (!(ok = warp_wait(&sm.pv_done[(sc - 1) & 1], ((sc - 1) >> 1) & 1, abort_flag, prm.status,
                                 prm.timeout_ns)))
              break;
            tc_fence_after();
            const float alpha = need ? ex2_approx(m_new - mx) : 1.0f;
#pragma unroll 1
            for (int g = 0; g < D / 16; ++g) {
              uint32_t o[16];
              tmem_ld16(tmem + lane_base + kColO + g * 16, o);
              tmem_wait_ld();
#pragma unroll
              for (int x = 0; x < 16; ++x) o[x] = __float_as_uint(__uint_as_float(o[x]) * alpha);
              tmem_st16(tmem + lane_base + kColO + g * 16, o);
            }
            tmem_wait_st();
          }
          if (need) m_new = mx;
          if (kAhead) {
#pragma unroll
            for (int q = 0; q < 4; ++q) l4[q] = make_float2(0.f, 0.f);
            exp_half(0);
          }
        }
        *const_cast<volatile float*>(&sm.m_row[sc & 1][row]) = m_new;
        __syncwarp();
        if (lane == 0) mbar_arrive(&sm.m_full[sc & 1][quarter]);
        if (t > (int)t0) l *= ex2_approx(m - m_new);
        m = m_new;
        // P goes over S's own columns (this thread has read its whole row of S)
#pragma unroll
        for (int hc = 0; hc < 2; ++hc) {
          if (!kAhead || hc == 1) exp_half(hc);
          tmem_st32(s_col + hc * 32, pk);
          tmem_wait_st();
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(&sm.p_full[sb][hc]);
        }
        const float2 lt = add2(add2(l4[0], l4[1]), add2(l4[2], l4[3]));
        l += lt.x + lt.y;
      }
      if (!ok) break;
      const uint32_t last = sc0 + L - 1, is = it & 1;
      if ((last & 1) != wgi) {
        // the other warpgroup finishes the item: hand it this one's normaliser
        *const_cast<volatile float*>(&sm.l_row[is][row]) = l;
        __syncwarp();
        if (lane == 0) mbar_arrive(&sm.l_full[is][quarter]);
      } else {
        // epilogue: O / l -> bf16, LSE (natural log)
        if (!(ok = warp_wait(&sm.l_full[is][quarter], (it >> 1) & 1, abort_flag, prm.status, prm.timeout_ns))) break;
        const float l_o = *const_cast<volatile float*>(&sm.l_row[is][row]);
        // it is under the maximum that the last tile but one used, <= m (0 where
        // there was none; a NaN has to come through)
        if (l_o != 0.f) l += l_o * ex2_approx(m_before - m);
        if (!(ok = warp_wait(&sm.pv_done[last & 1], (last >> 1) & 1, abort_flag, prm.status, prm.timeout_ns))) break;
        tc_fence_after();
        uint32_t o[D];
#pragma unroll
        for (int g = 0; g < D / 32; ++g)
          tmem_ld32(tmem + lane_base + kColO + g * 32, *reinterpret_cast<uint32_t(*)[32]>(&o[g * 32]));
        tmem_wait_ld();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&sm.o_empty);
        const float inv = (!kSub || l > 0.f) ? 1.0f / l : 0.f;  // a row that saw no key: O = 0, LSE = -inf
        if (row_ok) {
#pragma unroll
          for (int x = 0; x < D; x += 8) {
            uint4 v;
            v.x = pack_bf16x2(__uint_as_float(o[x + 0]) * inv, __uint_as_float(o[x + 1]) * inv);
            v.y = pack_bf16x2(__uint_as_float(o[x + 2]) * inv, __uint_as_float(o[x + 3]) * inv);
            v.z = pack_bf16x2(__uint_as_float(o[x + 4]) * inv, __uint_as_float(o[x + 5]) * inv);
            v.w = pack_bf16x2(__uint_as_float(o[x + 6]) * inv, __uint_as_float(o[x + 7]) * inv);
            *reinterpret_cast<uint4*>(orow + x) = v;
          }
          prm.lse[(int64_t)h * prm.N + grow] = (!kSub || l > 0.f) ? (m + log2f(l)) * 0.69314718055994531f : -INFINITY;
        }
      }
      sc0 += L;
      ++it;
    }
  }

  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 1) tmem_dealloc(tmem, 512);
}

static_assert(sizeof(FwdSmem<128>) <= 232448, "forward shared layout exceeds the per-block limit");
static_assert(sizeof(FwdSort) <= kStages * FwdSmem<64>::kKVBytes, "the sort's scratch must fit the K ring");

template <int D, int kMode, bool kSort = false>
static cudaError_t launch_d(const AttnProblem& p, const CUtensorMap& tq, const CUtensorMap& tk,
                            const CUtensorMap& tv, const CUtensorMap& tk64, const CUtensorMap& tv64,
                            const FwdParams& prm, int grid, cudaStream_t stream) {
  const size_t smem = sizeof(FwdSmem<D>);
  cudaError_t e =
      cudaFuncSetAttribute(attn_fwd_tc_kernel<D, kMode, kSort>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  // the setmaxnreg split assumes exactly kFwdRegLaunch registers per thread at
  // launch: with fewer, the increases would wait for registers that never come
  cudaFuncAttributes fa;
  e = cudaFuncGetAttributes(&fa, attn_fwd_tc_kernel<D, kMode, kSort>);
  if (e != cudaSuccess) return e;
  if (fa.numRegs != kFwdRegLaunch) return cudaErrorInvalidConfiguration;
  attn_fwd_tc_kernel<D, kMode, kSort><<<grid, kFwdThreads, smem, stream>>>(tq, tk, tv, tk64, tv64, prm);
  return cudaGetLastError();
}

cudaError_t launch_attn_fwd_tc(const AttnProblem& p, const void* q, const void* k, const void* v,
                               const int32_t* row_ptr, const int32_t* col_idx, void* o, float* lse, int32_t* status,
                               uint64_t timeout_ns, int sms, cudaStream_t stream) {
  const int nt = (int)((p.N + kBM - 1) / kBM);  // 128-row tiles
  const int n_items = p.H * nt;
  if (n_items == 0) return cudaSuccess;
  // 0: 128-row blocks on both sides; 1: 64-row query blocks, 128-row key
  // blocks (merged lists); 2: 128-row query blocks, 64-row key blocks paired
  // into 128-row tiles; 3: 64-row blocks on both sides, merged or paired per item
  const int mode = p.block == 128 ? (p.block_k == 128 ? 0 : 2) : (p.block_k == 128 ? 1 : 3);
  CUtensorMap tq, tk, tv, tk64, tv64;  // K / V as 128-row and as 64-row boxes
  const uint64_t inner = (uint64_t)p.H * p.d;
  const uint64_t stride = (uint64_t)p.row_stride * 2;
  if (!encode_tmap_2d_bf16(&tq, q, inner, p.N, stride, 64, kBM) ||
      !encode_tmap_2d_bf16(&tk, k, inner, p.N, stride, 64, kBN) ||
      !encode_tmap_2d_bf16(&tv, v, inner, p.N, stride, 64, kBN) ||
      !encode_tmap_2d_bf16(&tk64, k, inner, p.N, stride, 64, 64) ||
      !encode_tmap_2d_bf16(&tv64, v, inner, p.N, stride, 64, 64))
    return cudaErrorInvalidValue;
  FwdParams prm{};
  prm.row_ptr = row_ptr;
  prm.col_idx = col_idx;
  prm.o = static_cast<__nv_bfloat16*>(o);
  prm.lse = lse;
  prm.status = status;
  prm.N = p.N;
  prm.rs = p.row_stride;
  prm.H = p.H;
  prm.nq = nt;
  prm.nq_fine = p.nq;
  prm.q_rows_per_tile = p.block == 64 ? 2 : 1;
  prm.list_shift = p.block_k == 64 ? 1 : 0;
  prm.n_items = n_items;
  prm.scale_log2 = p.scale * 1.4426950408889634f;
  prm.timeout_ns = timeout_ns;
  const int grid = n_items < sms ? n_items : sms;
  const bool sort = mode == 0 && n_items > grid && n_items <= kSortItems && n_items <= kSortRounds * grid &&
             (int64_t)p.H * p.N * p.d * 4 <= kSortKvBytes;
#define UT_FWD_LAUNCH(DD, MM) launch_d<DD, MM>(p, tq, tk, tv, tk64, tv64, prm, grid, stream)
#define UT_FWD_MODES(DD)                                                                    \
  (sort ? launch_d<DD, 0, true>(p, tq, tk, tv, tk64, tv64, prm, grid, stream)               \
   : mode == 0 ? UT_FWD_LAUNCH(DD, 0)                                                       \
             : (mode == 1 ? UT_FWD_LAUNCH(DD, 1) : (mode == 2 ? UT_FWD_LAUNCH(DD, 2) : UT_FWD_LAUNCH(DD, 3))))
  if (p.d == 64) return UT_FWD_MODES(64);
  return UT_FWD_MODES(128);
#undef UT_FWD_MODES
#undef UT_FWD_LAUNCH
}

}  // namespace ut
