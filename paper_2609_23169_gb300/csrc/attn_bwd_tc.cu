// Block-sparse attention backward on the tcgen05 tensor cores.
//
// With P = exp(S - LSE) recomputed from the forward's row normalisers and
// D_r = dO_r . O_r:
//   dV = P^T dO,   dS = P o (dO V^T - D),   dQ = scale * dS K,   dK = scale * dS^T Q
// over the retained block pairs only:
//
//   bwd_pre_kernel          -D_r and -LSE_r * log2(e) per (head, row) into a
//                           padded [H, N_t*128] workspace (padding rows: 0 and
//                           -inf so that they contribute P = 0), the dQ
//                           accumulator cleared, the order of the items.
//   bwd_fused_kernel        item (h, 128-row key tile j) over the transposed
//                           lists: S^T and dP^T once per pair, dK and dV
//                           accumulated in TMEM, dQ^T partials added into an
//                           fp32 accumulator (below).
//   bwd_dq_finalize_kernel  dQ = scale * accumulator, bf16.
//
// Blocks of 64 rows (b_q or b_kv) are served by the same 128 x 128 tiles:
//   b_q = 64:   two listed 64-row query blocks fill one 128-row query tile
//               (Q and dO loaded as two 64-row TMA boxes, PairList):
//               consecutive entries of the key block's list for b_kv = 128
//               (nothing discarded), the two 64-row key blocks' lists in
//               lockstep for b_kv = 64 (key rows 0-63 see the low half of the
//               query tile, key rows 64-127 the high half); the dQ^T drain
//               adds each half into its own query block;
//   b_q = 128, b_kv = 64:  the item's two lists are merged into 128-row query
//               tiles with a mask of the listed 64 x 64 sub-blocks (TileList).
// P of the sub-blocks a key row does not see is zero.
// All waits are bounded (UT_ERR_TIMEOUT on expiry, then drain and return).
#include "common.cuh"
#include "kernels.h"

namespace ut {

constexpr int kTile = 128;
constexpr uint32_t kChunk = 128 * 128;  // one 128-row x 128-byte swizzled sub-tile

// ------------------------------------------------------------- preprocess
// Order in which the fused kernel's items (128-row key tiles) are handed out:
// groups of heads one after another, inside a group the longest lists first.
// Structured lists differ a lot in length (at the 512 canvas the reference
// image's key blocks list 61 query blocks, most others 11), and an item taken
// last holds one CTA while the others are done: handed out in index order the
// busiest of 152 CTAs had 242 steps against a mean of 199 there (1,516 against
// 1,388 at 1024), longest first 205 (1,407); a training layer at 1024 went from
// 5,316 to 5,151 us, at 512 with d = 64 from 440 to 419, this kernel also
// clearing the accumulator in place of a memset.  A group is as many heads as keep
// Q, dO and the dQ accumulator (8 N d bytes a head) within kOrderGroupBytes, so
// that the CTAs in flight still share one group's tiles in L2.
constexpr int64_t kOrderGroupBytes = 64ll << 20;
constexpr int kOrderBins = 1024;

struct OrderParams {
  const int32_t* ptr;  // transposed fine lists
  int32_t* order;      // [H * nt] (nullptr: index order)
  int32_t* counter;    // item counter, zeroed here
  int H, nt, nk_fine, k_rows_per_tile, heads_per_group, groups;
};

// One CTA per group: a counting sort by list length (which of two equally long
// items comes first does not matter).
UT_DEV void order_group(const OrderParams& o, int g) {
  __shared__ int32_t bins[kOrderBins];
  __shared__ int32_t warp_tot[8], s_max;
  const int h0 = g * o.heads_per_group, h1 = min(o.H, h0 + o.heads_per_group);
  const int first = h0 * o.nt, n = (h1 - h0) * o.nt;
  auto length = [&](int x) {  // listed blocks of item first + x
    const int h = h0 + x / o.nt, j = x % o.nt;
    const int64_t r = (int64_t)h * o.nk_fine + j * o.k_rows_per_tile;
    const int rows = min(o.k_rows_per_tile, o.nk_fine - j * o.k_rows_per_tile);
    return o.ptr[r + rows] - o.ptr[r];
  };
  if (threadIdx.x == 0) s_max = 1;
  for (int b = threadIdx.x; b < kOrderBins; b += blockDim.x) bins[b] = 0;
  __syncthreads();
  int mx = 1;
  for (int x = threadIdx.x; x < n; x += blockDim.x) mx = max(mx, length(x));
  atomicMax(&s_max, mx);
  __syncthreads();
  const float inv = (float)(kOrderBins - 1) / (float)s_max;
  auto bin = [&](int x) { return kOrderBins - 1 - min(kOrderBins - 1, (int)((float)length(x) * inv)); };
  for (int x = threadIdx.x; x < n; x += blockDim.x) atomicAdd(&bins[bin(x)], 1);
  __syncthreads();
  // exclusive prefix of the bins, four per thread (256 threads)
  const int b0 = threadIdx.x * (kOrderBins / 256), lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
  int c[kOrderBins / 256], local = 0;
#pragma unroll
  for (int e = 0; e < kOrderBins / 256; ++e) {
    c[e] = bins[b0 + e];
    local += c[e];
  }
  int incl = local;
  for (int off = 1; off < 32; off <<= 1) {
    const int v = __shfl_up_sync(0xffffffffu, incl, off);
    if (lane >= off) incl += v;
  }
  if (lane == 31) warp_tot[wp] = incl;
  __syncthreads();
  int run = incl - local;
  for (int i = 0; i < wp; ++i) run += warp_tot[i];
#pragma unroll
  for (int e = 0; e < kOrderBins / 256; ++e) {
    bins[b0 + e] = run;
    run += c[e];
  }
  __syncthreads();
  for (int x = threadIdx.x; x < n; x += blockDim.x) o.order[first + atomicAdd(&bins[bin(x)], 1)] = first + x;
}

// Where row o of a 64-row block stands in the row vectors: the elementwise
// threads read S^T and dP^T in accumulator fragments, so a thread needs columns
// 8 g + 2 a + {0, 1} with a = its lane % 4; they lie next to each other.
UT_DEV int vec_pos(int o) { return ((o >> 1) & 3) * 16 + (o >> 3) * 2 + (o & 1); }

// -D_r = -dO_r . O_r and -LSE_r * log2(e) into the padded [H, Np] workspace, and the
// dQ accumulator's row cleared; one warp per row r of Np.  The first
// o.groups blocks write the item order instead.
__global__ void __launch_bounds__(256) bwd_pre_kernel(const __nv_bfloat16* __restrict__ o,
                                                      const __nv_bfloat16* __restrict__ dout,
                                                      const float* __restrict__ lse, int64_t N, int64_t Np, int H,
                                                      int d, int64_t rs, float* __restrict__ lse2,
                                                      float* __restrict__ dsum, float* __restrict__ dq_acc,
                                                      const OrderParams op) {
  if (blockIdx.x == 0 && threadIdx.x == 0) *op.counter = 0;
  if ((int)blockIdx.x < op.groups) {
    order_group(op, blockIdx.x);
    return;
  }
  const int64_t r = (int64_t)(blockIdx.x - op.groups) * 8 + (threadIdx.x >> 5);
  if (r >= Np) return;
  const int lane = threadIdx.x & 31;
  const int lanes_per_head = d / 8;           // 16 (d=128) or 8 (d=64)
  const int heads_per_iter = 32 / lanes_per_head;
  for (int h0 = 0; h0 < H; h0 += heads_per_iter) {
    const int h = h0 + lane / lanes_per_head;
    float s = 0.f;
    if (r < N && h < H) {
      const int64_t off = r * rs + (int64_t)h * d + (lane % lanes_per_head) * 8;
      uint4 a = *reinterpret_cast<const uint4*>(o + off);
      uint4 b = *reinterpret_cast<const uint4*>(dout + off);
      const __nv_bfloat162* pa = reinterpret_cast<const __nv_bfloat162*>(&a);
      const __nv_bfloat162* pb = reinterpret_cast<const __nv_bfloat162*>(&b);
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        float2 x = __bfloat1622float2(pa[e]);
        float2 y = __bfloat1622float2(pb[e]);
        s = fmaf(x.x, y.x, s);
        s = fmaf(x.y, y.y, s);
      }
    }
    if (h < H) {
      uint4* acc = reinterpret_cast<uint4*>(dq_acc + ((int64_t)h * Np + r) * d + (lane % lanes_per_head) * 8);
      acc[0] = make_uint4(0, 0, 0, 0);
      acc[1] = make_uint4(0, 0, 0, 0);
    }
    for (int off = lanes_per_head / 2; off; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
    if ((lane % lanes_per_head) == 0 && h < H) {
      const int64_t at = (int64_t)h * Np + (r & ~(int64_t)63) + vec_pos((int)(r & 63));
      dsum[at] = r < N ? -s : 0.f;
      lse2[at] = r < N ? lse[(int64_t)h * N + r] * -1.4426950408889634f : -INFINITY;
    }
  }
}

struct BwdParams {
  const int32_t* ptr;   // transposed fine lists: per (head, key block) the query blocks
  const int32_t* idx;
  const float* lse2;    // [H, Np]  -LSE * log2(e) (padding rows: -inf, so that P = 0), rows in vec_pos order
  const float* dsum;    // [H, Np]  -D, likewise
  __nv_bfloat16* out0;  // dv
  __nv_bfloat16* out1;  // dk
  int32_t* status;
  int64_t N, Np, rs;
  int H, nq, n_items;   // nq: 128-row tiles per head (items = H * nq key tiles)
  int nk_fine;          // key blocks per head in the transposed lists
  int k_rows_per_tile;  // 1 (b_kv = 128) or 2 (b_kv = 64)
  int list_shift;       // 0 (b_q = 128) or 1 (b_q = 64)
  float scale, scale_log2;
  uint64_t timeout_ns;
  int32_t* item_counter;  // next item to hand out (zeroed before the launch)
  const int32_t* order;   // the items in the order they are handed out (nullptr: index order)
};

// 64 consecutive TMEM columns of this warp's 32 lanes, one wait.
UT_DEV void tmem_ld64(uint32_t taddr, uint32_t* r) {
  tmem_ld32(taddr, *reinterpret_cast<uint32_t(*)[32]>(r));
  tmem_ld32(taddr + 32, *reinterpret_cast<uint32_t(*)[32]>(r + 32));
  tmem_wait_ld();
}

// =========================================================================
//                       fused dK, dV and dQ (one kernel)
// =========================================================================
// Item = (head h, key block j); the pairs are the query blocks i of the
// transposed list.  Per pair, with the 128 key rows as TMEM lanes:
//   S^T  = K Q_i^T         -> TMEM R0            (A = K, B = Q_i; smem)
//   P^T  = exp2(S^T c - LSE_i log2 e)   -> bf16, shared tile PT
//   dP^T = V dO_i^T        -> TMEM R0 (after S^T was read)
//   dV  += P^T dO_i        (A = PT, B = dO_i)
//   dS^T = P^T o (dP^T - D_i)           -> bf16, shared tile DST
//   dK  += dS^T Q_i        (A = DST, B = Q_i)
//   dQ_i^T = K^T dS^T      -> TMEM RQ            (A = K read d-major, B = DST)
// and four drain warps add dQ_i^T into an fp32 [H, N_q*128, d] accumulator
// with coalesced reductions (lane = d, one 128-byte row segment per query
// row), off the elementwise warps' path; S and dP are computed once per pair.
// A final kernel scales the accumulator by the softmax scale and writes dQ in
// bf16.  Roles (512 threads, four warpgroups; the register file is rebalanced
// with setmaxnreg): warpgroup 0 = warp 0 TMA of K, V and Q, warp 1 TMEM owner +
// MMA issuer, warp 2 the row vectors and warp 3 TMA of dO (one lane each);
// warpgroups 1-2 = 8 elementwise warps; warpgroup 3 = 4 dQ drain warps.
// TMEM columns: R0 [0,128), RQ [128,256), dV [256,256+d), dK [384,384+d).
// For d = 64 the A operand K^T of the dQ product is padded to 128 rows with a
// zero sub-tile placed right after K, and the padding rows of RQ are ignored.
constexpr int kFuThreads = 512;
// registers per thread after setmaxnreg, per warpgroup; the sum equals the
// launch allocation (4 x 128) so that every increase is covered by decreases
constexpr int kFuRegLaunch = 128, kFuRegCtl = 96, kFuRegEw = 168, kFuRegDrain = 80;
static_assert(kFuRegCtl + 2 * kFuRegEw + kFuRegDrain == 4 * kFuRegLaunch, "setmaxnreg split must match the launch");
// Ring depths: Q is held from S^T to dK (late in the pair), dO only from dP^T
// to dV (early), so dO gets one stage and its 32 KB buy separate P^T and
// dS^T tiles: P^T of the next pair never waits for this pair's dK and dQ.
constexpr int kFuQStages = 2, kFuDoStages = 1;
constexpr uint32_t kColR0 = 0, kColRQ = 128, kColFuDv = 256, kColFuDk = 384;

// Items are handed out dynamically (the transposed lists differ in length:
// 36-153 query blocks per key block at the 2048 canvas, so a static
// round-robin leaves the busiest CTA ~5% above the mean), in the order that
// bwd_pre_kernel wrote.  kItemConsumers: the dO and row-vector producers,
// the MMA warp, 8 elementwise warps, 4 drain warps.
constexpr int kItemSlots = 4, kItemConsumers = 15;

template <int D>
struct FusedSmem {
  static constexpr int kC = D / 64;
  static constexpr uint32_t kTileBytes = kTile * D * 2;
  alignas(1024) uint8_t k[2 * kChunk];        // K (d/64 sub-tiles), then zeros up to 128 d-rows
  alignas(1024) uint8_t v[kTileBytes];
  alignas(1024) uint8_t pt[kTile * kTile * 2];   // P^T of the current pair
  alignas(1024) uint8_t dst[kTile * kTile * 2];  // dS^T of the current pair
  alignas(1024) uint8_t q[kFuQStages][kTileBytes];
  alignas(1024) uint8_t dout[kFuDoStages][kTileBytes];
  alignas(16) float lse2[2][kTile];           // -LSE log2 e and -D of the pair's query rows
  alignas(16) float dsum[2][kTile];
  uint64_t kv_full, kv_empty;
  uint64_t q_full[kFuQStages], q_empty[kFuQStages], do_full[kFuDoStages], do_empty[kFuDoStages];
  uint64_t s_full, s_empty, dp_full, dp_empty, pt_full, pt_done, dst_full, ds_done, dq_empty;
  uint64_t acc_full, acc_empty, mma_done;
  uint64_t vec_full[2], vec_empty[2];
  // the CTA's item sequence: warp 0 takes the next item from the global
  // counter and publishes it here; every other role reads the slots in order
  int32_t item[kItemSlots];
  uint64_t item_full[kItemSlots], item_empty[kItemSlots];
  uint32_t tmem_base;
  int abort_flag;
};

UT_DEV void red_add_f32(float* p, float v) {
  asm volatile("red.relaxed.gpu.global.add.f32 [%0], %1;" ::"l"(p), "f"(v) : "memory");
}

template <int D, int kMode>
__global__ void __launch_bounds__(kFuThreads, 1)
    bwd_fused_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k,
                     const __grid_constant__ CUtensorMap tm_v, const __grid_constant__ CUtensorMap tm_do,
                     const __grid_constant__ CUtensorMap tm_q64, const __grid_constant__ CUtensorMap tm_do64,
                     const BwdParams prm, float* __restrict__ dq_acc) {
  constexpr bool kSub = kMode != 0;  // 64-row blocks on at least one side
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  FusedSmem<D>& sm = *reinterpret_cast<FusedSmem<D>*>(smem_raw);
  constexpr int C = FusedSmem<D>::kC;
  constexpr uint32_t TB = FusedSmem<D>::kTileBytes;
  const uint32_t warp = warp_id(), lane = lane_id();
  volatile int* abort_flag = &sm.abort_flag;
  if ((smem_u32(smem_raw) & 1023u) != 0) {
    if (threadIdx.x == 0) set_status(prm.status, UT_ERR_INVALID_ARG);
    return;
  }
  if (D == 64) {  // zero padding sub-tile of K^T (rows d = 64..127 of the dQ product)
    uint4* z = reinterpret_cast<uint4*>(sm.k + kChunk);
    for (uint32_t x = threadIdx.x; x < kChunk / 16; x += blockDim.x) z[x] = make_uint4(0, 0, 0, 0);
    fence_proxy_async_smem();
  }
  if (threadIdx.x == 0) {
    mbar_init(&sm.kv_full, 1);
    mbar_init(&sm.kv_empty, 1);
    for (int s = 0; s < kFuQStages; ++s) {
      mbar_init(&sm.q_full[s], 1);
      mbar_init(&sm.q_empty[s], 1);
    }
    for (int s = 0; s < kFuDoStages; ++s) {
      mbar_init(&sm.do_full[s], 1);
      mbar_init(&sm.do_empty[s], 1);
    }
    mbar_init(&sm.s_full, 1);
    mbar_init(&sm.s_empty, 8);
    mbar_init(&sm.dp_full, 1);
    mbar_init(&sm.dp_empty, 8);
    mbar_init(&sm.pt_full, 8);
    mbar_init(&sm.pt_done, 1);
    mbar_init(&sm.dst_full, 8);
    mbar_init(&sm.ds_done, 1);
    mbar_init(&sm.dq_empty, 4);
    mbar_init(&sm.acc_full, 1);
    mbar_init(&sm.acc_empty, 8);
    mbar_init(&sm.mma_done, 1);
    for (int s = 0; s < 2; ++s) {
      mbar_init(&sm.vec_full[s], 1);
      mbar_init(&sm.vec_empty[s], 8);
    }
    for (int s = 0; s < kItemSlots; ++s) {
      mbar_init(&sm.item_full[s], 1);
      mbar_init(&sm.item_empty[s], kItemConsumers);
    }
    sm.abort_flag = 0;
    fence_barrier_init();
  }
  if (warp == 1) {
    tmem_alloc(&sm.tmem_base, 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = sm.tmem_base;
  const uint32_t wg = warp >> 2;
  // next item of this CTA's sequence (-1: none left); whole warp (converged)
  // or, with one = true, a single thread.  Returns false on timeout / abort.
  auto next_item = [&](uint32_t& kk, int& w, bool one) -> bool {
    const uint32_t s = kk % kItemSlots, n = kk / kItemSlots;
    const bool got = one ? mbar_wait(&sm.item_full[s], n & 1, abort_flag, prm.status, prm.timeout_ns)
                         : warp_wait(&sm.item_full[s], n & 1, abort_flag, prm.status, prm.timeout_ns);
    if (!got) return false;
    w = *reinterpret_cast<volatile int32_t*>(&sm.item[s]);
    if (one) {
      mbar_arrive(&sm.item_empty[s]);
    } else {
      __syncwarp();
      if (lane == 0) mbar_arrive(&sm.item_empty[s]);
    }
    ++kk;
    return true;
  };
  if (wg == 0) {
    setmaxnreg_dec<kFuRegCtl>();
    if (warp == 0 || warp == 3) {
      // Warp 0: K, V of the item and the Q ring (Q is freed after dK += dS^T Q);
      // warp 3: the dO ring (dO is freed after dV += P^T dO).  One lane each: two
      // lanes of one warp wait for each other wherever the compiler lets them meet
      // again (1024 canvas, d = 128: 1% of the launch).
      if (lane == 0) {
        const bool is_q = warp == 0;
        if (is_q) {
          tma_prefetch_desc(&tm_q);
          tma_prefetch_desc(&tm_k);
          tma_prefetch_desc(&tm_v);
          if (kMode >= 2) tma_prefetch_desc(&tm_q64);
        } else {
          tma_prefetch_desc(&tm_do);
          if (kMode >= 2) tma_prefetch_desc(&tm_do64);
        }
        const uint64_t pol_qd = policy_evict_last(), pol_kv = policy_evict_first();
        uint64_t* full = is_q ? sm.q_full : sm.do_full;
        uint64_t* empty = is_q ? sm.q_empty : sm.do_empty;
        uint8_t* ring = is_q ? &sm.q[0][0] : &sm.dout[0][0];
        const void* tmap = is_q ? static_cast<const void*>(&tm_q) : static_cast<const void*>(&tm_do);
        const void* tmap64 = is_q ? static_cast<const void*>(&tm_q64) : static_cast<const void*>(&tm_do64);
        const uint32_t nst = is_q ? kFuQStages : kFuDoStages;
        uint32_t ki = 0, qd = 0, kk = 0;
        bool ok = true;
        for (;;) {
          int w;
          if (is_q) {  // take the next item and publish it to the other roles
            const uint32_t s = kk % kItemSlots, n = kk / kItemSlots;
            if (!(ok = mbar_wait(&sm.item_empty[s], (n & 1) ^ 1, abort_flag, prm.status, prm.timeout_ns))) break;
            w = atomicAdd(prm.item_counter, 1);
            if (w >= prm.n_items) w = -1;
            else if (prm.order) w = prm.order[w];
            *reinterpret_cast<volatile int32_t*>(&sm.item[s]) = w;
            mbar_arrive(&sm.item_full[s]);
            ++kk;
          } else if (!(ok = next_item(kk, w, true))) {
            break;
          }
          if (w < 0) break;
          const int h = w / prm.nq, j = w % prm.nq;
          BlockSteps<kMode> tl;
          tl.init(prm.ptr, prm.idx, h, j, prm.nk_fine, prm.k_rows_per_tile, prm.list_shift);
          if (tl.empty()) continue;
          if (is_q) {
            if (!(ok = mbar_wait(&sm.kv_empty, (ki & 1) ^ 1, abort_flag, prm.status, prm.timeout_ns))) break;
            mbar_expect_tx(&sm.kv_full, 2 * TB);
            for (int c = 0; c < C; ++c) {
              tma_load_2d(sm.k + c * kChunk, &tm_k, &sm.kv_full, h * D + c * 64, j * kTile, pol_kv);
              tma_load_2d(sm.v + c * kChunk, &tm_v, &sm.kv_full, h * D + c * 64, j * kTile, pol_kv);
            }
            ++ki;
          }
          int i, ih;
          uint32_t bits;
          for (; tl.next(i, ih, bits); ++qd) {
            const uint32_t st = qd % nst, n = qd / nst;
            if (!(ok = mbar_wait(&empty[st], (n & 1) ^ 1, abort_flag, prm.status, prm.timeout_ns))) break;
            mbar_expect_tx(&full[st], TB);
            uint8_t* dst = ring + st * TB;
            if (tl.pair) {  // two 64-row boxes: rows 0-63 and 64-127 of each 128-row sub-tile
              const int b0 = PairList::load_lo(i, ih), b1 = PairList::load_hi(i, ih);
              for (int c = 0; c < C; ++c) {
                tma_load_2d(dst + c * kChunk, tmap64, &full[st], h * D + c * 64, b0 * 64, pol_qd);
                tma_load_2d(dst + c * kChunk + 64 * 128, tmap64, &full[st], h * D + c * 64, b1 * 64, pol_qd);
              }
            } else {
              for (int c = 0; c < C; ++c)
                tma_load_2d(dst + c * kChunk, tmap, &full[st], h * D + c * 64, i * kTile, pol_qd);
            }
          }
          if (!ok) break;
        }
        auto drain = [&](uint64_t* bar, uint32_t parity) {
          if (!mbar_drain(bar, parity, kDrainTimeoutNs)) set_status(prm.status, UT_ERR_TIMEOUT);
        };
        if (ki > 0) drain(&sm.kv_full, (ki - 1) & 1);
        for (uint32_t u = (qd >= nst ? qd - nst : 0); u < qd; ++u) drain(&full[u % nst], (u / nst) & 1);
      }
    } else if (warp == 2) {
      // row vectors of the pair's query rows, two pairs ahead (freed by the
      // elementwise warps): fetched by those warps themselves and handed round
      // through shared memory they cost ~480 of ~5,100 cycles of every pair
      // (2048 canvas, backward: 22.23 -> 21.6 ms)
      if (lane == 0) {
        uint32_t qd = 0, kk = 0;
        bool ok = true;
        while (ok) {
          int w;
          if (!(ok = next_item(kk, w, true)) || w < 0) break;
          const int64_t base = (int64_t)(w / prm.nq) * prm.Np;
          BlockSteps<kMode> tl;
          tl.init(prm.ptr, prm.idx, w / prm.nq, w % prm.nq, prm.nk_fine, prm.k_rows_per_tile, prm.list_shift);
          int i, ih;
          uint32_t bits;
          for (; tl.next(i, ih, bits); ++qd) {
            const uint32_t st = qd & 1;
            if (!(ok = mbar_wait(&sm.vec_empty[st], ((qd >> 1) & 1) ^ 1, abort_flag, prm.status, prm.timeout_ns))) break;
            const int64_t b0 = base + 64 * (int64_t)(tl.pair ? PairList::load_lo(i, ih) : 2 * i);
            const int64_t b1 = base + 64 * (int64_t)(tl.pair ? PairList::load_hi(i, ih) : 2 * i + 1);
            mbar_expect_tx(&sm.vec_full[st], 2 * kTile * sizeof(float));
            bulk_load(&sm.lse2[st][0], prm.lse2 + b0, 256, &sm.vec_full[st]);
            bulk_load(&sm.lse2[st][64], prm.lse2 + b1, 256, &sm.vec_full[st]);
            bulk_load(&sm.dsum[st][0], prm.dsum + b0, 256, &sm.vec_full[st]);
            bulk_load(&sm.dsum[st][64], prm.dsum + b1, 256, &sm.vec_full[st]);
          }
        }
        for (uint32_t u = (qd >= 2 ? qd - 2 : 0); u < qd; ++u)
          if (!mbar_drain(&sm.vec_full[u & 1], (u >> 1) & 1, kDrainTimeoutNs)) set_status(prm.status, UT_ERR_TIMEOUT);
      }
    } else if (warp == 1) {
      // whole warp, converged: waits are warp-uniform, MMAs/commits elect one lane.
      // Per pair t: dP^T_t, dV_t, S^T_{t+1}, dK_t, dQ_t^T.
      {
        constexpr uint32_t idesc_s = idesc_bf16_f32(kTile, kTile, false, false);
        constexpr uint32_t idesc_acc = idesc_bf16_f32(kTile, D, false, true);
        constexpr uint32_t idesc_dq = idesc_bf16_f32(kTile, kTile, true, true);
        const uint32_t k_addr = smem_u32(sm.k), v_addr = smem_u32(sm.v);
      const uint32_t pt_addr = smem_u32(sm.pt), dst_addr = smem_u32(sm.dst);
        uint32_t ki = 0, qd0 = 0, kk = 0;
        bool ok = true;
        for (;;) {
          int w;
          if (!(ok = next_item(kk, w, false)) || w < 0) break;
          BlockSteps<kMode> tl;
          tl.init(prm.ptr, prm.idx, w / prm.nq, w % prm.nq, prm.nk_fine, prm.k_rows_per_tile, prm.list_shift);
          const int L = uniform(tl.count_warp());
          if (L <= 0) continue;
          if (!(ok = warp_wait(&sm.kv_full, ki & 1, abort_flag, prm.status, prm.timeout_ns))) break;
          auto issue_st = [&](int t) -> bool {  // S^T_t = K Q_t^T into R0
            const uint32_t qd = qd0 + t, st = qd % kFuQStages, n = qd / kFuQStages;
            if (!warp_wait(&sm.q_full[st], n & 1, abort_flag, prm.status, prm.timeout_ns)) return false;
            if (!warp_wait(&sm.dp_empty, (qd & 1) ^ 1, abort_flag, prm.status, prm.timeout_ns)) return false;
            tc_fence_after();
            const uint32_t q_addr = smem_u32(sm.q[st]);
  #pragma unroll
            for (int kk = 0; kk < D / 16; ++kk) {
              const uint32_t off = (kk >> 2) * kChunk + (kk & 3) * 32;
              mma_bf16_ss_w(tmem + kColR0, sdesc_sw128(k_addr + off, 16, 1024), sdesc_sw128(q_addr + off, 16, 1024),
                            idesc_s, kk > 0);
            }
            mma_commit_w(&sm.s_full);
            return true;
          };
          if (!(ok = issue_st(0))) break;
          for (int t = 0; t < L && ok; ++t) {
            const uint32_t qd = qd0 + t, sq = qd % kFuQStages, sd = qd % kFuDoStages, nd = qd / kFuDoStages;
            const uint32_t do_addr = smem_u32(sm.dout[sd]), q_addr = smem_u32(sm.q[sq]);
            // dP^T_t = V dO_t^T into R0 once S^T_t has been read
            if (!(ok = warp_wait(&sm.do_full[sd], nd & 1, abort_flag, prm.status, prm.timeout_ns))) break;
            if (!(ok = warp_wait(&sm.s_empty, qd & 1, abort_flag, prm.status, prm.timeout_ns))) break;
            tc_fence_after();
  #pragma unroll
            for (int kk = 0; kk < D / 16; ++kk) {
              const uint32_t off = (kk >> 2) * kChunk + (kk & 3) * 32;
              mma_bf16_ss_w(tmem + kColR0, sdesc_sw128(v_addr + off, 16, 1024), sdesc_sw128(do_addr + off, 16, 1024),
                            idesc_s, kk > 0);
            }
            mma_commit_w(&sm.dp_full);
            // dV += P^T_t dO_t
            if (!(ok = warp_wait(&sm.pt_full, qd & 1, abort_flag, prm.status, prm.timeout_ns))) break;
            if (t == 0 && !(ok = warp_wait(&sm.acc_empty, (ki & 1) ^ 1, abort_flag, prm.status, prm.timeout_ns)))
              break;
            tc_fence_after();
  #pragma unroll
            for (int kk = 0; kk < kTile / 16; ++kk) {
              const uint32_t aoff = (kk >> 2) * kChunk + (kk & 3) * 32;
              mma_bf16_ss_w(tmem + kColFuDv, sdesc_sw128(pt_addr + aoff, 16, 1024),
                            sdesc_sw128(do_addr + kk * 2048, kChunk, 1024), idesc_acc, (t > 0 || kk > 0));
            }
            mma_commit_w(&sm.pt_done);
            mma_commit_w(&sm.do_empty[sd]);
            // S^T_{t+1} once dP^T_t has been read
            if (t + 1 < L && !(ok = issue_st(t + 1))) break;
            // dK += dS^T_t Q_t
            if (!(ok = warp_wait(&sm.dst_full, qd & 1, abort_flag, prm.status, prm.timeout_ns))) break;
            tc_fence_after();
  #pragma unroll
            for (int kk = 0; kk < kTile / 16; ++kk) {
              const uint32_t aoff = (kk >> 2) * kChunk + (kk & 3) * 32;
              mma_bf16_ss_w(tmem + kColFuDk, sdesc_sw128(dst_addr + aoff, 16, 1024),
                            sdesc_sw128(q_addr + kk * 2048, kChunk, 1024), idesc_acc, (t > 0 || kk > 0));
            }
            mma_commit_w(&sm.q_empty[sq]);
            // dQ_t^T = K^T dS^T_t into RQ once the previous pair's dQ^T was drained
            if (!(ok = warp_wait(&sm.dq_empty, (qd & 1) ^ 1, abort_flag, prm.status, prm.timeout_ns))) break;
            tc_fence_after();
  #pragma unroll
            for (int kk = 0; kk < kTile / 16; ++kk)
              mma_bf16_ss_w(tmem + kColRQ, sdesc_sw128(k_addr + kk * 2048, kChunk, 1024),
                            sdesc_sw128(dst_addr + kk * 2048, kChunk, 1024), idesc_dq, kk > 0);
            mma_commit_w(&sm.ds_done);
            if (t == L - 1) mma_commit_w(&sm.kv_empty);
          }
          if (!ok) break;
          mma_commit_w(&sm.acc_full);
          qd0 += L;
          ++ki;
        }
        mma_commit_w(&sm.mma_done);
        if (!mbar_drain(&sm.mma_done, 0, kDrainTimeoutNs)) set_status(prm.status, UT_ERR_TIMEOUT);
      }
  }
  } else if (wg == 1 || wg == 2) {
    setmaxnreg_inc<kFuRegEw>();
    // 8 elementwise warps: warps w and w+4 share TMEM lane quarter (w & 3),
    // i.e. the same 32 key rows, and split the 128 query columns (and the D
    // output columns) into halves.  A half is exactly one 128-byte swizzle
    // sub-tile of the shared P^T / dS^T tile.
    const uint32_t quarter = warp & 3;
    const uint32_t half = (warp - 4) >> 2;
    const uint32_t krow = quarter * 32 + lane;  // key row of the tile = TMEM lane (d index for dQ^T)
    const uint32_t lane_base = (quarter * 32) << 16;
    constexpr int HC = kTile / 2;               // query columns per half
    constexpr int HD = D / 2;                   // output columns per half
    const float c = prm.scale_log2;
    // S^T and dP^T are read as accumulator fragments (a thread: 4 rows x 16
    // columns instead of 1 x 64), so that a pair needs 8 shared reads of the row
    // vectors a thread, not 32: the dQ reductions keep the same load/store queue
    // full, and each read waits its turn there (2048 canvas, backward: 21.55 ->
    // 20.5 ms; training layer at 1024: 3.74 -> 3.54).  stmatrix puts the bf16 results
    // into the swizzled tiles: lane l gives row l % 16 of 16, chunk g + l / 16.
    const uint32_t srow = quarter * 32 + (lane & 15), chunk_hi = lane >> 4;
    const uint32_t pt_row = smem_u32(sm.pt) + half * kChunk + srow * 128;
    const uint32_t vec_at = half * HC + (lane & 3) * 16;
    auto load_vec = [](const float* src, float (&v)[16]) {
#pragma unroll
      for (int x = 0; x < 16; x += 4) {
        const float4 f = *reinterpret_cast<const float4*>(src + x);
        v[x] = f.x;
        v[x + 1] = f.y;
        v[x + 2] = f.z;
        v[x + 3] = f.w;
      }
    };
    uint32_t qd0 = 0, ki = 0, kk = 0;
    bool ok = true;
    const uint32_t kh = krow >> 6;  // which 64-row half of the key tile
    for (;;) {
      int w;
      if (!(ok = next_item(kk, w, false)) || w < 0) break;
      const int h = w / prm.nq, j = w % prm.nq;
      BlockSteps<kMode> tl;
      tl.init(prm.ptr, prm.idx, h, j, prm.nk_fine, prm.k_rows_per_tile, prm.list_shift);
      const int L = uniform(tl.count_warp());
      const int64_t gk = (int64_t)j * kTile + krow;
      const bool row_ok = gk < prm.N;
      // Key rows past N are zeros, so S = 0 there and P = exp(0 - LSE) is infinite
      // where LSE < -88.7: their rows of dS^T have to be zero, or dQ^T = K^T dS^T
      // sums 0 * inf.  In the last key tile they are cleared once, and what the
      // pairs compute for them goes over the same rows of P^T, which only reach
      // rows of dV that are not written.  Nothing is added to the loop over the
      // pairs but the choice of the row: selects on P or on dS^T, a test that is
      // never true, a copy of the loop, the clearing by the MMA warp or products
      // that leave those lanes out all cost more (1 to 14%; this -1 to 2%, and 4%
      // with d = 64 and 64-row blocks on both sides).
      const int key_rows = (int)min((int64_t)kTile, prm.N - (int64_t)j * kTile);
      const uint32_t to_dst = smem_u32(sm.dst) - smem_u32(sm.pt);
      const uint32_t ds_row[2] = {pt_row + ((int)srow < key_rows ? to_dst : 0),
                                  pt_row + ((int)srow + 16 < key_rows ? to_dst : 0) + 2048};
      __nv_bfloat16* dv_row = prm.out0 + gk * prm.rs + (int64_t)h * D + half * HD;
      __nv_bfloat16* dk_row = prm.out1 + gk * prm.rs + (int64_t)h * D + half * HD;
      if (L <= 0) {
        if (row_ok)
          for (int e = 0; e < HD; e += 8) {
            *reinterpret_cast<uint4*>(dv_row + e) = make_uint4(0, 0, 0, 0);
            *reinterpret_cast<uint4*>(dk_row + e) = make_uint4(0, 0, 0, 0);
          }
        continue;
      }
      if (key_rows < (int)quarter * 32 + 32) {  // (the tile is free: the item before has been written out)
        for (int x = max(key_rows - (int)quarter * 32, 0) * 8 + (int)lane; x < 32 * 8; x += 32)
          *reinterpret_cast<uint4*>(sm.dst + half * kChunk + quarter * (32 * 128) + x * 16) = make_uint4(0, 0, 0, 0);
        __syncwarp();
      }
      for (int t = 0; t < L; ++t) {
        const uint32_t qd = qd0 + t;
        // this half's 64 query columns and this thread's 64 key rows form one
        // 64 x 64 sub-block of the tile pair: listed or not
        bool listed = true;
        if (kSub) {
          int i, ih;
          uint32_t bits;
          tl.next(i, ih, bits);
          listed = (bits >> (2 * kh + half)) & 1u;
        }
        if (!(ok = warp_wait(&sm.vec_full[qd & 1], (qd >> 1) & 1, abort_flag, prm.status, prm.timeout_ns))) break;
        if (!(ok = warp_wait(&sm.s_full, qd & 1, abort_flag, prm.status, prm.timeout_ns))) break;
        tc_fence_after();
        float p[2][32];  // rows 0-15 and 16-31 of this warp's 32, accumulator fragments of 64 columns
        {
          uint32_t r[2][32];
          tmem_ld_16x64(tmem + lane_base + kColR0 + half * HC, r[0]);
          tmem_ld_16x64(tmem + lane_base + (16u << 16) + kColR0 + half * HC, r[1]);
          float ls[16];
          load_vec(sm.lse2[qd & 1] + vec_at, ls);
          tmem_wait_ld();
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(&sm.s_empty);
#pragma unroll
          for (int u = 0; u < 2; ++u)
#pragma unroll
            for (int x = 0; x < 32; x += 2) {
              if (listed) {
                const int g = x >> 2;
                const float2 e =
                    ffma2(make_float2(__uint_as_float(r[u][x]), __uint_as_float(r[u][x + 1])), make_float2(c, c),
                          make_float2(ls[2 * g], ls[2 * g + 1]));
                p[u][x] = ex2_approx(e.x);
                p[u][x + 1] = ex2_approx(e.y);
              } else {
                p[u][x] = p[u][x + 1] = 0.f;
              }
            }
        }
        // the P^T tile is free once the previous pair's dV MMA finished
        if (!(ok = warp_wait(&sm.pt_done, (qd & 1) ^ 1, abort_flag, prm.status, prm.timeout_ns))) break;
#pragma unroll
        for (int u = 0; u < 2; ++u)
#pragma unroll
          for (int g = 0; g < 8; g += 2)
            stmatrix_x4(pt_row + u * 2048 + (((g + chunk_hi) ^ (srow & 7)) << 4),
                        pack_bf16x2(p[u][4 * g], p[u][4 * g + 1]), pack_bf16x2(p[u][4 * g + 2], p[u][4 * g + 3]),
                        pack_bf16x2(p[u][4 * g + 4], p[u][4 * g + 5]), pack_bf16x2(p[u][4 * g + 6], p[u][4 * g + 7]));
        fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) mbar_arrive(&sm.pt_full);
        float dv[16];
        load_vec(sm.dsum[qd & 1] + vec_at, dv);
        if (!(ok = warp_wait(&sm.dp_full, qd & 1, abort_flag, prm.status, prm.timeout_ns))) break;
        tc_fence_after();
        // dS^T, 16 key rows at a time (fewer live registers); the dS^T tile is
        // free once the previous pair's dK and dQ^T MMAs finished
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          uint32_t r[32];
          tmem_ld_16x64(tmem + lane_base + ((16u * u) << 16) + kColR0 + half * HC, r);
          tmem_wait_ld();
          if (u == 1) {
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&sm.dp_empty);
          }
          uint32_t dsk[16];
#pragma unroll
          for (int x = 0; x < 32; x += 2) {
            const int g = x >> 2;
            const float2 a = mul2(make_float2(p[u][x], p[u][x + 1]),
                                  add2(make_float2(__uint_as_float(r[x]), __uint_as_float(r[x + 1])),
                                       make_float2(dv[2 * g], dv[2 * g + 1])));
            dsk[x / 2] = pack_bf16x2(a.x, a.y);
          }
          if (u == 0 && !(ok = warp_wait(&sm.ds_done, (qd & 1) ^ 1, abort_flag, prm.status, prm.timeout_ns))) break;
#pragma unroll
          for (int g = 0; g < 8; g += 2)
            stmatrix_x4(ds_row[u] + (((g + chunk_hi) ^ (srow & 7)) << 4), dsk[2 * g], dsk[2 * g + 1],
                        dsk[2 * g + 2], dsk[2 * g + 3]);
        }
        if (!ok) break;
        fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) {
          mbar_arrive(&sm.dst_full);
          mbar_arrive(&sm.vec_empty[qd & 1]);
        }
      }
      if (!ok) break;
      if (!(ok = warp_wait(&sm.acc_full, ki & 1, abort_flag, prm.status, prm.timeout_ns))) break;
      tc_fence_after();
#pragma unroll
      for (int part = 0; part < 2; ++part) {
        __nv_bfloat16* dst = part == 0 ? dv_row : dk_row;
        const float f = part == 0 ? 1.0f : prm.scale;
#pragma unroll
        for (int g = 0; g < HD / 32; ++g) {
          uint32_t r[32];
          tmem_ld32(tmem + lane_base + (part == 0 ? kColFuDv : kColFuDk) + half * HD + g * 32, r);
          tmem_wait_ld();
          if (row_ok) {
#pragma unroll
            for (int x = 0; x < 32; x += 8) {
              uint4 v;
              v.x = pack_bf16x2(__uint_as_float(r[x + 0]) * f, __uint_as_float(r[x + 1]) * f);
              v.y = pack_bf16x2(__uint_as_float(r[x + 2]) * f, __uint_as_float(r[x + 3]) * f);
              v.z = pack_bf16x2(__uint_as_float(r[x + 4]) * f, __uint_as_float(r[x + 5]) * f);
              v.w = pack_bf16x2(__uint_as_float(r[x + 6]) * f, __uint_as_float(r[x + 7]) * f);
              *reinterpret_cast<uint4*>(dst + g * 32 + x) = v;
            }
          }
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&sm.acc_empty);
      qd0 += L;
      ++ki;
    }
  } else {
    setmaxnreg_dec<kFuRegDrain>();
    // 4 dQ drain warps, one per TMEM lane quarter: for dQ_i^T the TMEM lane is
    // the d index.  Each thread adds its d of all 128 query rows of block i,
    // one fp32 reduction per row; the warp covers 32 consecutive d of a row
    // (one 128-byte segment).  RQ is released once both halves are read.
    const uint32_t quarter = warp & 3;
    const uint32_t dcol = quarter * 32 + lane;
    const uint32_t lane_base = (quarter * 32) << 16;
    uint32_t qd0 = 0, kk = 0;
    bool ok = true;
    for (;;) {
      int w;
      if (!(ok = next_item(kk, w, false)) || w < 0) break;
      const int h = w / prm.nq;
      BlockSteps<kMode> tl;
      tl.init(prm.ptr, prm.idx, h, w % prm.nq, prm.nk_fine, prm.k_rows_per_tile, prm.list_shift);
      const int L = uniform(tl.count_warp());
      if (L <= 0) continue;
      for (int t = 0; t < L; ++t) {
        const uint32_t qd = qd0 + t;
        int i, ih;
        uint32_t bits;
        tl.next(i, ih, bits);
        if (!(ok = warp_wait(&sm.ds_done, qd & 1, abort_flag, prm.status, prm.timeout_ns))) break;
        tc_fence_after();
#pragma unroll
        for (int g = 0; g < 2; ++g) {
          // query half g of the tile: rows of 64-row block lo / hi (paired), or
          // rows g * 64 .. of the 128-row query block; a missing block (-1)
          // has dS^T = 0 there and is not added
          const int blk = tl.pair ? (g ? ih : i) : 0;
          const int64_t row0 = tl.pair ? 64 * (int64_t)blk : (int64_t)i * kTile + 64 * g;
          float* dst = dq_acc + (((int64_t)h * prm.Np + row0) * D + dcol);
          uint32_t r[64];
          tmem_ld64(tmem + lane_base + kColRQ + g * 64, r);
          if (g == 1) {
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&sm.dq_empty);
          }
          if (dcol < (uint32_t)D && blk >= 0) {
#pragma unroll
            for (int x = 0; x < 64; ++x) red_add_f32(dst + (int64_t)x * D, __uint_as_float(r[x]));
          }
        }
      }
      if (!ok) break;
      qd0 += L;
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 1) tmem_dealloc(tmem, 512);
}

// dQ = scale * accumulator, bf16, rows < N: thread = 8 consecutive d of one (row, head)
__global__ void __launch_bounds__(256) bwd_dq_finalize_kernel(const float* __restrict__ acc, int64_t N, int64_t Np,
                                                              int H, int d, int64_t rs, float scale,
                                                              __nv_bfloat16* __restrict__ dq) {
  const int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int per_row = H * d / 8;
  if (g >= N * per_row) return;
  const int64_t r = g / per_row;
  const int e = (int)(g % per_row) * 8;
  const int h = e / d, c = e % d;
  const float4* src = reinterpret_cast<const float4*>(acc + ((int64_t)h * Np + r) * d + c);
  const float4 a = src[0], b = src[1];
  uint4 v;
  v.x = pack_bf16x2(a.x * scale, a.y * scale);
  v.y = pack_bf16x2(a.z * scale, a.w * scale);
  v.z = pack_bf16x2(b.x * scale, b.y * scale);
  v.w = pack_bf16x2(b.z * scale, b.w * scale);
  *reinterpret_cast<uint4*>(dq + r * rs + e) = v;
}

// ----------------------------------------------------------------- launcher
static size_t bwd_tiles(const AttnProblem& p) { return (size_t)((p.N + kTile - 1) / kTile); }

size_t attn_bwd_tc_ws(const AttnProblem& p) {
  const size_t Np = bwd_tiles(p) * kTile;
  return 2 * (size_t)p.H * Np * sizeof(float) + (size_t)p.H * Np * p.d * sizeof(float) + 16;  // + item counter
}

// With the item order after the counter; a smaller workspace (at least
// attn_bwd_tc_ws) hands the items out in index order.
size_t attn_bwd_tc_ws_ordered(const AttnProblem& p) {
  return attn_bwd_tc_ws(p) + (size_t)p.H * bwd_tiles(p) * sizeof(int32_t);
}

constexpr size_t kMaxDynSmem = 232448;  // 227 KB opt-in per block on sm_100/sm_103
static_assert(sizeof(FusedSmem<128>) <= kMaxDynSmem, "fused backward shared layout exceeds the per-block limit");

template <int D, int kMode>
static cudaError_t launch_bwd_fused(const AttnProblem& p, const CUtensorMap* tm, BwdParams prm, float* dq_acc,
                                   __nv_bfloat16* dq, int sms, cudaStream_t s) {
  const int n_items = prm.n_items;
  const int grid = n_items < sms ? n_items : sms;
  const size_t smem = sizeof(FusedSmem<D>);
  cudaError_t e =
      cudaFuncSetAttribute(bwd_fused_kernel<D, kMode>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  // the setmaxnreg split assumes exactly kFuRegLaunch registers per thread at
  // launch: with fewer, the increases would wait for registers that never come
  cudaFuncAttributes fa;
  e = cudaFuncGetAttributes(&fa, bwd_fused_kernel<D, kMode>);
  if (e != cudaSuccess) return e;
  if (fa.numRegs != kFuRegLaunch) return cudaErrorInvalidConfiguration;
  bwd_fused_kernel<D, kMode><<<grid, kFuThreads, smem, s>>>(tm[0], tm[1], tm[2], tm[3], tm[4], tm[5], prm, dq_acc);
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  const int64_t n8 = p.N * p.H * D / 8;
  bwd_dq_finalize_kernel<<<(unsigned)((n8 + 255) / 256), 256, 0, s>>>(dq_acc, p.N, prm.Np, p.H, D, p.row_stride,
                                                                      p.scale, dq);
  return cudaGetLastError();
}

cudaError_t launch_attn_bwd_tc(const AttnProblem& p, const void* q, const void* k, const void* v, const void* o,
                               const float* lse, const void* dout, const int32_t* row_ptr, const int32_t* col_idx,
                               const int32_t* col_ptr_t, const int32_t* row_idx_t, void* dq, void* dk, void* dv,
                               void* ws, size_t ws_bytes, int32_t* status, uint64_t timeout_ns, int sms,
                               cudaStream_t stream) {
  (void)row_ptr;
  (void)col_idx;  // the fused kernel walks the transposed lists only
  const int nt = (int)((p.N + kTile - 1) / kTile);  // 128-row tiles
  if (nt == 0) return cudaSuccess;
  const int64_t Np = (int64_t)nt * kTile;
  float* lse2 = static_cast<float*>(ws);
  float* dsum = lse2 + (size_t)p.H * Np;
  float* dq_acc = dsum + (size_t)p.H * Np;
  int32_t* item_counter = reinterpret_cast<int32_t*>(dq_acc + (size_t)p.H * Np * p.d);
  OrderParams op{};
  op.ptr = col_ptr_t;
  op.order = ws_bytes >= attn_bwd_tc_ws_ordered(p) ? item_counter + 4 : nullptr;
  op.counter = item_counter;
  op.H = p.H;
  op.nt = nt;
  op.nk_fine = p.nk;
  op.k_rows_per_tile = p.block_k == 64 ? 2 : 1;
  const int64_t per_group = kOrderGroupBytes / (8 * Np * p.d);
  op.heads_per_group = (int)(per_group < 1 ? 1 : (per_group > p.H ? p.H : per_group));
  op.groups = op.order ? (p.H + op.heads_per_group - 1) / op.heads_per_group : 0;
  bwd_pre_kernel<<<(unsigned)((Np + 7) / 8 + op.groups), 256, 0, stream>>>(
      static_cast<const __nv_bfloat16*>(o), static_cast<const __nv_bfloat16*>(dout), lse, p.N, Np, p.H, p.d,
      p.row_stride, lse2, dsum, dq_acc, op);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  // 0: 128-row blocks on both sides; 1: 128-row query blocks, 64-row key
  // blocks (merged lists); 2: 64-row query blocks, 128-row key blocks, paired
  // into 128-row tiles; 3: 64-row blocks on both sides, merged or paired per item
  const int mode = p.block == 128 ? (p.block_k == 128 ? 0 : 1) : (p.block_k == 128 ? 2 : 3);
  CUtensorMap tm[6];  // Q, K, V, dO as 128-row boxes, then Q and dO as 64-row boxes
  const uint64_t inner = (uint64_t)p.H * p.d, stride = (uint64_t)p.row_stride * 2;
  const void* bases[6] = {q, k, v, dout, q, dout};
  for (int x = 0; x < 6; ++x)
    if (!encode_tmap_2d_bf16(&tm[x], bases[x], inner, p.N, stride, 64, x < 4 ? kTile : 64))
      return cudaErrorInvalidValue;
  BwdParams a{};
  a.ptr = col_ptr_t;
  a.idx = row_idx_t;
  a.lse2 = lse2;
  a.dsum = dsum;
  a.out0 = static_cast<__nv_bfloat16*>(dv);
  a.out1 = static_cast<__nv_bfloat16*>(dk);
  a.status = status;
  a.N = p.N;
  a.Np = Np;
  a.rs = p.row_stride;
  a.H = p.H;
  a.nq = nt;
  a.n_items = p.H * nt;
  a.nk_fine = p.nk;
  a.k_rows_per_tile = op.k_rows_per_tile;
  a.list_shift = p.block == 64 ? 1 : 0;
  a.scale = p.scale;
  a.scale_log2 = p.scale * 1.4426950408889634f;
  a.timeout_ns = timeout_ns;
  a.item_counter = item_counter;
  a.order = op.order;
  __nv_bfloat16* dqb = static_cast<__nv_bfloat16*>(dq);
#define UT_BWD_LAUNCH(DD, MM) launch_bwd_fused<DD, MM>(p, tm, a, dq_acc, dqb, sms, stream)
#define UT_BWD_MODES(DD)                                                                    \
  (mode == 0 ? UT_BWD_LAUNCH(DD, 0)                                                         \
             : (mode == 1 ? UT_BWD_LAUNCH(DD, 1) : (mode == 2 ? UT_BWD_LAUNCH(DD, 2) : UT_BWD_LAUNCH(DD, 3))))
  if (p.d == 64) return UT_BWD_MODES(64);
  return UT_BWD_MODES(128);
#undef UT_BWD_MODES
#undef UT_BWD_LAUNCH
}

}  // namespace ut
