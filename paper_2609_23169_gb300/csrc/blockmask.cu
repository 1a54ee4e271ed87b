// Block mask M_c as key-block lists (Sec. 3.3).
//
// Top-K mode:
//   block_pool_kernel    pool(Q) over blocks of b_q rows, pool(K) over blocks
//                        of b_kv rows: fp32 mean over the valid rows of each
//                        block (one CTA per block and 128 16-byte columns).
//   score_select_kernel  S_c[i, :] = pool(Q)_i . pool(K)_j in fp32 for R query
//                        blocks of one head, then per row an exact select of
//                        the K_rho-th largest score over order-preserving keys;
//                        equal scores go to the smaller key-block index.
//                        Writes row_ptr, the ascending list and the row of a
//                        [H, N_q, N_k] bit mask (32 key blocks per word).
//   transpose_kernel     the lists per key block from the bit mask, by warp
//                        ballots.
// Bitmap mode, lists and transpose side by side in each launch:
//   bitmap_count_kernel  entries per row and per column (into the pointers),
//   scan_kernel          exclusive prefix in place -> row_ptr / col_ptr,
//   bitmap_fill_kernel   ascending lists by warp ballot.
#include "common.cuh"
#include "kernels.h"

namespace ut {

constexpr int kPoolThreads = 128;
constexpr int kSelThreads = 128;
constexpr int kSelCols = 256;      // key blocks per tile of scores
constexpr int kSelRows = 16;       // query blocks per CTA (fewer when N_k is large)

template <typename T>
struct Vec8;
template <>
struct Vec8<__nv_bfloat16> {
  static constexpr int kElems = 8;
  UT_DEV static void load(const __nv_bfloat16* p, float* f) {
    uint4 u = *reinterpret_cast<const uint4*>(p);
    const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&u);
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      float2 x = __bfloat1622float2(h[e]);
      f[2 * e] = x.x;
      f[2 * e + 1] = x.y;
    }
  }
};
template <>
struct Vec8<float> {
  static constexpr int kElems = 4;
  UT_DEV static void load(const float* p, float* f) {
    float4 u = *reinterpret_cast<const float4*>(p);
    f[0] = u.x; f[1] = u.y; f[2] = u.z; f[3] = u.w;
  }
};

// grid (max(nq, nk), 2, column slices): blockIdx.y selects Q (0, blocks of bq
// rows) or K (1, blocks of bk rows), a thread owns one 16-byte column of the
// slice.  out: pooled Q [H][nq][d], then pooled K [H][nk][d].  HBM-bound (Q and K
// are read once); one column a thread keeps every thread of a row busy whatever
// H * d is, and small problems get three times the CTAs.
// 2048 canvas (1.05 GB): 189 -> 160 us, 6.55 TB/s.
template <typename T>
__global__ void __launch_bounds__(kPoolThreads) block_pool_kernel(const T* __restrict__ q, const T* __restrict__ k,
                                                                  int64_t N, int H, int d, int64_t row_stride,
                                                                  int bq, int nq, int bk, int nk,
                                                                  float* __restrict__ out) {
  constexpr int E = Vec8<T>::kElems;
  const bool is_k = blockIdx.y == 1;
  const T* x = is_k ? k : q;
  const int block = is_k ? bk : bq, nb = is_k ? nk : nq;
  const int i = blockIdx.x;
  const int c0 = (blockIdx.z * kPoolThreads + threadIdx.x) * E;
  if (i >= nb || c0 >= H * d) return;
  const int64_t r0 = (int64_t)i * block;
  const int64_t r1 = min(N, r0 + block);
  float acc[E];
#pragma unroll
  for (int e = 0; e < E; ++e) acc[e] = 0.f;
  const T* p = x + r0 * row_stride + c0;
#pragma unroll 16
  for (int64_t r = r0; r < r1; ++r, p += row_stride) {
    float f[E];
    Vec8<T>::load(p, f);
#pragma unroll
    for (int e = 0; e < E; ++e) acc[e] += f[e];
  }
  float* dst = (is_k ? out + (size_t)H * nq * d : out) + ((int64_t)(c0 / d) * nb + i) * d + c0 % d;
#pragma unroll
  for (int e = 0; e < E; ++e) dst[e] = __fdiv_rn(acc[e], (float)(r1 - r0));
}

UT_DEV uint32_t order_key(float s) {
  s = s + 0.0f;  // -0 -> +0
  uint32_t u = __float_as_uint(s);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

// Score of a key (the inverse of order_key).
UT_DEV float key_score(uint32_t u) { return __uint_as_float((u & 0x80000000u) ? (u & 0x7FFFFFFFu) : ~u); }

// K-th largest of the warp's n_lo keys, lo and top the smallest and the largest:
// count_ge(lo) >= k > count_ge(hi) holds throughout and the bracket closes in on the largest value
// with at least k keys >= it.  Candidates alternate between the score that a
// straight line through the bracket's counts gives (scores near a quantile are
// nearly evenly spread: some eight steps, against 32 by bits) and the middle of
// the bracket, which bounds the steps whatever the scores are.  A candidate
// with exactly k keys at or above it ends the search.  On return every key >
// thr belongs, and the first `equal` keys (by index) that are equal to thr.
template <typename Count>
UT_DEV void select_kth(Count count_ge, int k, uint32_t lo, uint32_t top, int n_lo, uint32_t& thr, int& equal) {
  uint32_t hi = top;
  int n_hi = 0;
  if (top != 0xffffffffu) {
    hi = top + 1;
  } else {  // NaN scores (the largest key there is) stand first
    n_hi = __reduce_add_sync(0xffffffffu, count_ge(top));
    if (n_hi >= k) {
      thr = top;
      equal = k;
      return;
    }
  }
  if (n_lo == k && lo > 0) {  // every key
    thr = lo - 1;
    equal = 0;
    return;
  }
  for (int step = 0; hi - lo > 1; ++step) {
    uint32_t cand = lo + ((hi - lo) >> 1);
    if (!(step & 1)) {
      const float a = key_score(lo), b = key_score(hi);
      const float f = a + (b - a) * __fdividef((float)(n_lo - k) + 0.5f, (float)(n_lo - n_hi));
      const uint32_t c = order_key(f);  // (not finite: outside the bracket or harmless)
      if (c > lo && c < hi) cand = c;
    }
    const int n = __reduce_add_sync(0xffffffffu, count_ge(cand));
    if (n == k) {  // the keys >= cand are the answer: > cand - 1 (cand > 0)
      thr = cand - 1;
      equal = 0;
      return;
    }
    if (n > k) {
      lo = cand;
      n_lo = n;
    } else {
      hi = cand;
      n_hi = n;
    }
  }
  thr = lo;
  equal = k - n_hi;
}

// K-th largest of the keys of one row, kKeys per lane in registers (absent ones
// 0: below every score's key).
template <int kKeys>
UT_DEV void select_row(const float* srow, int nk, int k, int lane, uint32_t& thr, int& equal) {
  uint32_t key[kKeys], lo = 0xffffffffu, hi = 0u;
#pragma unroll
  for (int x = 0; x < kKeys; ++x) {
    const int j = 32 * x + lane;
    key[x] = j < nk ? order_key(srow[j]) : 0u;
    if (j < nk) {
      lo = min(lo, key[x]);
      hi = max(hi, key[x]);
    }
  }
  lo = __reduce_min_sync(0xffffffffu, lo);
  hi = __reduce_max_sync(0xffffffffu, hi);
  select_kth(
      [&](uint32_t cand) {
        int n = 0;
#pragma unroll
        for (int x = 0; x < kKeys; ++x) n += key[x] >= cand;
        return n;
      },
      k, lo, hi, nk, thr, equal);
}

// The same for rows that do not fit registers (N_k > 2048), where each of the
// search's passes would read the row from shared memory again: four passes by 8
// bits, counts of the warp in hw[256] (shared).  6,656 key blocks, 1 head: 3,700
// -> 2,530 us for the lists (the search 12 passes; these four were there before it
// and took 3,630 with the scores of that time); 1,332 key blocks, 24 heads of d =
// 64, 48 keys a lane in registers: 1,080 -> 848 (898 with these passes and the
// scores of that time).
UT_DEV void select_row_radix(const float* srow, int nk, int k, int lane, uint32_t* hw, uint32_t& thr, int& equal) {
  uint32_t prefix = 0, pmask = 0;
  for (int shift = 24; shift >= 0; shift -= 8) {
    for (int b = lane; b < 256; b += 32) hw[b] = 0;
    __syncwarp();
    for (int j = lane; j < nk; j += 32) {
      const uint32_t u = order_key(srow[j]);
      if ((u & pmask) == prefix) atomicAdd(&hw[(u >> shift) & 255u], 1u);
    }
    __syncwarp();
    // lane l owns bins 255 - 8 l .. 248 - 8 l; one lane finds the bin that holds rank k
    uint32_t cnt[8], local = 0;
#pragma unroll
    for (int x = 0; x < 8; ++x) {
      cnt[x] = hw[255 - 8 * lane - x];
      local += cnt[x];
    }
    uint32_t incl = local;
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t v = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += v;
    }
    uint32_t digit = 255 - 8 * lane, above = incl - local;
    const bool here = above < (uint32_t)k && (uint32_t)k <= incl;
#pragma unroll
    for (int x = 0; x < 7; ++x) {
      if (above + cnt[x] >= (uint32_t)k) break;
      above += cnt[x];
      --digit;
    }
    const int src = __ffs(__ballot_sync(0xffffffffu, here)) - 1;
    digit = __shfl_sync(0xffffffffu, digit, src);
    k -= (int)__shfl_sync(0xffffffffu, above, src);
    prefix |= digit << shift;
    pmask |= 0xFFu << shift;
    __syncwarp();
  }
  thr = prefix;
  equal = k;
}

// grid (H, ceil(nq / R)); dynamic smem: pooled query rows [d][kRows], a slice of
// pooled keys [kE][kSelCols], scores [R][nk].  Rows are query blocks (nq per
// head), columns key blocks (nk).
// The scores are bound by what shared memory can hand to the registers (128
// bytes a cycle, a broadcast counted in full): a thread that owned one key
// block and 16 rows read 68 bytes for 16 multiply-adds and the launch took 320
// us at the 2048 canvas; 8 rows x 4 key blocks read 48 for 32 (and with the
// search above instead of 32 passes by bits 263 -> 194; 282 with the keys read
// from global memory and a radix select over shared counters).  Slices are
// staged d-major, 4-column groups exchanged by their d / 4 in the slice so that
// neither the transposing stores nor the reads conflict.  A sum runs over d in
// order, as one FMA chain.
// kRows: rows a tile holds; kE: d per staged slice of pool(K); kLong: N_k > 1024 (a
// kernel of its own: the selections of long rows would lengthen the code that a
// small call has to fetch, 11.5 -> 12.6 us at 100 tokens)
template <int kRows, int kE, bool kLong>
__global__ void __launch_bounds__(kSelThreads) score_select_kernel(const float* __restrict__ pooled, int H, int d,
                                                                   int nq, int nk, int R, int k_rho,
                                                                   int32_t* __restrict__ row_ptr,
                                                                   int32_t* __restrict__ col_idx,
                                                                   uint32_t* __restrict__ bits) {
  extern __shared__ __align__(16) float smem[];
  constexpr int kTr = kRows / 2, kTc = 4;  // a thread's rows and columns: 2 row groups x 64 column groups
  const int tid = threadIdx.x;
  float* pq = smem;                      // [d][kRows]
  float* kt = pq + kRows * d;            // [kE][kSelCols]
  float* sc = kt + kE * kSelCols;     // [R][nk]
  const int h = blockIdx.x;
  const int i0 = blockIdx.y * R;
  const int rows = min(R, nq - i0);
  const int rg = tid & 1, cg = tid >> 1;
  const float* PQ = pooled + ((int64_t)h * nq + i0) * d;
  const float* PK = pooled + (int64_t)H * nq * d + ((int64_t)h * nk) * d;
  for (int t = tid; t < kRows * d; t += kSelThreads) {
    const int r = t / d, e = t % d;
    pq[e * kRows + r] = r < rows ? PQ[t] : 0.f;
  }
  for (int j0 = 0; j0 < nk; j0 += kSelCols) {
    float2 acc[kTr / 2][kTc];
#pragma unroll
    for (int r = 0; r < kTr / 2; ++r)
#pragma unroll
      for (int x = 0; x < kTc; ++x) acc[r][x] = make_float2(0.f, 0.f);
    constexpr int kLoads = kSelCols * (kE / 4) / kSelThreads;  // 16-byte loads of a slice per thread
    float4 next[kLoads];
    auto fetch = [&](int e0) {
#pragma unroll
      for (int x = 0; x < kLoads; ++x) {
        const int t = x * kSelThreads + tid, j = t / (kE / 4), a = t % (kE / 4);
        next[x] = j0 + j < nk ? *reinterpret_cast<const float4*>(PK + (int64_t)(j0 + j) * d + e0 + 4 * a)
                              : make_float4(0.f, 0.f, 0.f, 0.f);
      }
    };
    fetch(0);
    for (int e0 = 0; e0 < d; e0 += kE) {
      __syncthreads();  // the slice (and, at first, pq) is free / written
#pragma unroll
      for (int x = 0; x < kLoads; ++x) {
        const int t = x * kSelThreads + tid, j = t / (kE / 4), a = t % (kE / 4);
        float* dst = kt + 4 * a * kSelCols + (j ^ (a << 2));
        dst[0] = next[x].x;
        dst[kSelCols] = next[x].y;
        dst[2 * kSelCols] = next[x].z;
        dst[3 * kSelCols] = next[x].w;
      }
      __syncthreads();
      if (e0 + kE < d) fetch(e0 + kE);  // in flight during this slice's products
#pragma unroll 8
      for (int e = 0; e < kE; ++e) {
        const float4 kv = *reinterpret_cast<const float4*>(kt + e * kSelCols + ((cg ^ (e >> 2)) << 2));
        const float kx[kTc] = {kv.x, kv.y, kv.z, kv.w};
        float2 p[kTr / 2];
        const float* prow = pq + (e0 + e) * kRows + rg * kTr;
#pragma unroll
        for (int r = 0; r < kTr / 2; ++r) p[r] = *reinterpret_cast<const float2*>(prow + 2 * r);
#pragma unroll
        for (int x = 0; x < kTc; ++x)
#pragma unroll
          for (int r = 0; r < kTr / 2; ++r) acc[r][x] = ffma2(p[r], make_float2(kx[x], kx[x]), acc[r][x]);
      }
    }
#pragma unroll
    for (int x = 0; x < kTc; ++x) {
      const int j = j0 + cg * kTc + x;
      if (j >= nk) continue;
#pragma unroll
      for (int r = 0; r < kTr / 2; ++r) {
        const int r0 = rg * kTr + 2 * r;
        if (r0 < rows) sc[r0 * nk + j] = acc[r][x].x;
        if (r0 + 1 < rows) sc[(r0 + 1) * nk + j] = acc[r][x].y;
      }
    }
  }
  __syncthreads();
  static_assert(kE * kSelCols >= kSelThreads / 32 * 256, "256 counts a warp must fit over the last slice");
  const int lane = tid & 31, w = tid >> 5, W = (nk + 31) / 32;
  const uint32_t lt_mask = (1u << lane) - 1u;
  for (int r = w; r < rows; r += kSelThreads / 32) {
    const float* srow = sc + r * nk;
    uint32_t thr = 0;
    int equal = 0;
    if constexpr (kLong) {
      if (W <= 48) {
        select_row<48>(srow, nk, k_rho, lane, thr, equal);
      } else if (W <= 64) {
        select_row<64>(srow, nk, k_rho, lane, thr, equal);
      } else {
        select_row_radix(srow, nk, k_rho, lane, reinterpret_cast<uint32_t*>(kt) + w * 256, thr, equal);
      }
    } else if (W <= 8) {
      select_row<8>(srow, nk, k_rho, lane, thr, equal);
    } else if (W <= 16) {
      select_row<16>(srow, nk, k_rho, lane, thr, equal);
    } else if (W <= 24) {
      select_row<24>(srow, nk, k_rho, lane, thr, equal);
    } else {
      select_row<32>(srow, nk, k_rho, lane, thr, equal);
    }
    // all keys above thr, and the first `equal` ones at it
    const int row = h * nq + i0 + r;
    int32_t* out = col_idx + (int64_t)row * k_rho;
    uint32_t* brow = bits + (int64_t)row * W;
    int n_sel = 0, n_eq = 0;
    for (int x = 0; x < W; ++x) {
      const int j = 32 * x + lane;
      const bool valid = j < nk;
      const uint32_t u = valid ? order_key(srow[j]) : 0u;
      const uint32_t eqb = __ballot_sync(0xffffffffu, valid && u == thr);
      const bool sel = valid && (u > thr || (u == thr && n_eq + __popc(eqb & lt_mask) < equal));
      const uint32_t selb = __ballot_sync(0xffffffffu, sel);
      if (sel) out[n_sel + __popc(selb & lt_mask)] = j;
      if (lane == 0) brow[x] = selb;
      n_sel += __popc(selb);
      n_eq += __popc(eqb);
    }
    if (lane == 0) {
      row_ptr[row] = row * k_rho;
      if (row == H * nq - 1) row_ptr[row + 1] = (row + 1) * k_rho;
    }
  }
}

// grid (H, ceil(nk / 32)): the lists of 32 key blocks of one head from the bit
// mask [H, nq, W].  Every row holds k_rho entries, so a head's entries start at
// h * nq * k_rho, and what lies before these 32 columns is found here: no pass
// over all counts, no second launch (count, scan and fill took 67 us at the 2048
// canvas, this launch about 20).  Up to kTransWords words to the left it is a
// population count over them; further right, where those words would be read
// again and again (the cube of the number of blocks), a binary search in each
// row's list (666 key blocks: the lists take 62.6 us counted, 65.2 searched; 2,048:
// 751 and 637; 6,656: 2,719 and 2,525).  A warp owns a run of 32-row groups;
// ballots turn 32 rows x 32 columns round, lane c then holding column c's rows.
constexpr int kTransThreads = 256;
constexpr int kTransWords = 32;  // words to the left that are counted
__global__ void __launch_bounds__(kTransThreads) transpose_kernel(const uint32_t* __restrict__ bits,
                                                                  const int32_t* __restrict__ col_idx, int H, int nq,
                                                                  int nk, int k_rho, int32_t* __restrict__ col_ptr,
                                                                  int32_t* __restrict__ row_idx) {
  constexpr int kWarps = kTransThreads / 32;
  __shared__ int32_t s_before[kWarps], s_count[kWarps][32];
  const int W = (nk + 31) / 32, wc = blockIdx.y, h = blockIdx.x;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const uint32_t* hb = bits + (int64_t)h * nq * W;
  int before = 0;
  if (wc <= kTransWords) {
    for (int i = threadIdx.x; i < nq; i += kTransThreads)
      for (int x = 0; x < wc; ++x) before += __popc(hb[(int64_t)i * W + x]);
  } else {
    for (int i = threadIdx.x; i < nq; i += kTransThreads) {
      const int32_t* list = col_idx + ((int64_t)h * nq + i) * k_rho;
      int lo = 0, hi = k_rho;  // entries below column 32 wc
      while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (list[mid] < 32 * wc) lo = mid + 1;
        else hi = mid;
      }
      before += lo;
    }
  }
  before = __reduce_add_sync(0xffffffffu, before);
  const int groups = (nq + 31) / 32, per = (groups + kWarps - 1) / kWarps;
  const int g0 = min(groups, w * per), g1 = min(groups, g0 + per);
  auto column = [&](int g) -> uint32_t {  // rows 32 g .. 32 g + 31 of column 32 wc + lane
    const int i = 32 * g + lane;
    const uint32_t word = i < nq ? hb[(int64_t)i * W + wc] : 0u;
    uint32_t mine = 0;
#pragma unroll
    for (int c = 0; c < 32; ++c) {
      const uint32_t b = __ballot_sync(0xffffffffu, (word >> c) & 1u);
      if (lane == c) mine = b;
    }
    return mine;
  };
  int count = 0;
  for (int g = g0; g < g1; ++g) count += __popc(column(g));
  s_count[w][lane] = count;
  if (lane == 0) s_before[w] = before;
  __syncthreads();
  int start = h * nq * k_rho, total = 0, ahead = 0;
  for (int x = 0; x < kWarps; ++x) {
    start += s_before[x];
    total += s_count[x][lane];
    if (x < w) ahead += s_count[x][lane];
  }
  int incl = total;  // prefix over the 32 columns
  for (int o = 1; o < 32; o <<= 1) {
    const int v = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += v;
  }
  start += incl - total;
  const int j = 32 * wc + lane;
  if (w == 0 && j < nk) {
    col_ptr[h * nk + j] = start;
    if (h == H - 1 && j == nk - 1) col_ptr[H * nk] = start + total;
  }
  int32_t* out = row_idx + start + ahead;
  for (int g = g0; g < g1; ++g) {
    uint32_t m = column(g);
    while (m) {
      *out++ = 32 * g + __ffs(m) - 1;
      m &= m - 1;
    }
  }
}

// Line l = (h, a): a row i of [H][nq][nk], or a column j for the transpose; one
// warp per line.  Rows and columns are functions of their own so that a line's
// loads can run ahead of its stores (one function over either side's pointers, and
// the scan's counts read one by one: 47.8 us for the rows' lists of the 2048
// canvas against 33.3, 80.4 against 66.4 with the transpose).
template <bool kCols>
UT_DEV uint8_t bitmap_at(const uint8_t* __restrict__ bm, int h, int nq, int nk, int a, int b) {
  return kCols ? bm[((int64_t)h * nq + b) * nk + a] : bm[((int64_t)h * nq + a) * nk + b];
}

template <bool kCols>
UT_DEV void count_line(const uint8_t* __restrict__ bm, int H, int nq, int nk, int32_t* __restrict__ counts) {
  const int n_lines = kCols ? nk : nq, len = kCols ? nq : nk;
  const int line = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (line >= H * n_lines) return;
  const int h = line / n_lines, a = line % n_lines;
  const int lane = threadIdx.x & 31;
  int c = 0;
  for (int b = lane; b < len; b += 32) c += bitmap_at<kCols>(bm, h, nq, nk, a, b) != 0;
  for (int o = 16; o; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
  if (lane == 0) counts[line] = c;
}

// blockIdx.y: 0 the rows, 1 the columns
__global__ void bitmap_count_kernel(const uint8_t* __restrict__ bm, int H, int nq, int nk,
                                    int32_t* __restrict__ row_ptr, int32_t* __restrict__ col_ptr) {
  if (blockIdx.y == 0) count_line<false>(bm, H, nq, nk, row_ptr);
  else count_line<true>(bm, H, nq, nk, col_ptr);
}

// Exclusive scan in place of the counts ptr[0..n) into ptr[0..n], one CTA a side.
__global__ void __launch_bounds__(1024) scan_kernel(int n_rows, int n_cols, int32_t* row_ptr, int32_t* col_ptr) {
  __shared__ int64_t warp_tot[32];
  const int n = blockIdx.x ? n_cols : n_rows;
  int32_t* ptr = blockIdx.x ? col_ptr : row_ptr;
  const int tid = threadIdx.x;
  const int per = (n + 1023) / 1024;
  const int a = min(n, tid * per), b = min(n, a + per);
  constexpr int kAhead = 8;  // counts loaded before any is replaced by its prefix
  int64_t local = 0;
#pragma unroll kAhead
  for (int t = a; t < b; ++t) local += ptr[t];
  int64_t incl = local;
  const int lane = tid & 31, w = tid >> 5;
  for (int o = 1; o < 32; o <<= 1) {
    int64_t v = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += v;
  }
  if (lane == 31) warp_tot[w] = incl;
  __syncthreads();
  int64_t wpre = 0;
  for (int i = 0; i < w; ++i) wpre += warp_tot[i];
  int64_t run = wpre + incl - local;
  for (int t = a; t < b; t += kAhead) {
    int c[kAhead];
#pragma unroll
    for (int x = 0; x < kAhead; ++x) c[x] = t + x < b ? ptr[t + x] : 0;
#pragma unroll
    for (int x = 0; x < kAhead; ++x) {
      if (t + x < b) ptr[t + x] = (int32_t)run;
      run += c[x];
    }
  }
  if (tid == 1023) ptr[n] = (int32_t)(wpre + incl);
}

template <bool kCols>
UT_DEV void fill_line(const uint8_t* __restrict__ bm, int H, int nq, int nk, const int32_t* __restrict__ ptr,
                      int32_t* __restrict__ out, int64_t cap, int32_t* status) {
  const int n_lines = kCols ? nk : nq, len = kCols ? nq : nk;
  const int line = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (line >= H * n_lines) return;
  const int h = line / n_lines, a = line % n_lines;
  const int lane = threadIdx.x & 31;
  const uint32_t lt_mask = (1u << lane) - 1u;
  int64_t pos = ptr[line];
  bool overflow = false;
  for (int b0 = 0; b0 < len; b0 += 32) {
    const int b = b0 + lane;
    const bool on = b < len && bitmap_at<kCols>(bm, h, nq, nk, a, b) != 0;
    const uint32_t bal = __ballot_sync(0xffffffffu, on);
    if (on) {
      int64_t p = pos + __popc(bal & lt_mask);
      if (p < cap) out[p] = b;
      else overflow = true;
    }
    pos += __popc(bal);
  }
  if (__any_sync(0xffffffffu, overflow) && lane == 0) set_status(status, UT_ERR_CAPACITY);
}

__global__ void bitmap_fill_kernel(const uint8_t* __restrict__ bm, int H, int nq, int nk,
                                   const int32_t* __restrict__ row_ptr, int32_t* __restrict__ col_idx,
                                   const int32_t* __restrict__ col_ptr, int32_t* __restrict__ row_idx, int64_t cap,
                                   int32_t* status) {
  if (blockIdx.y == 0) fill_line<false>(bm, H, nq, nk, row_ptr, col_idx, cap, status);
  else fill_line<true>(bm, H, nq, nk, col_ptr, row_idx, cap, status);
}

// ----------------------------------------------------------------- launchers
template <int kRows, int kE, bool kLong>
static cudaError_t launch_score_select(const float* pooled, int H, int d, int nq, int nk, int R, int k_rho,
                                       int32_t* row_ptr, int32_t* col_idx, uint32_t* bits, cudaStream_t stream) {
  const size_t smem = ((size_t)kRows * d + (size_t)kE * kSelCols + (size_t)R * nk) * sizeof(float);
  cudaError_t e =
      cudaFuncSetAttribute(score_select_kernel<kRows, kE, kLong>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  score_select_kernel<kRows, kE, kLong><<<dim3(H, (nq + R - 1) / R), kSelThreads, smem, stream>>>(
      pooled, H, d, nq, nk, R, k_rho, row_ptr, col_idx, bits);
  return cudaGetLastError();
}

// More than the kernels use, and kept: a workspace of the size that was asked for
// before is still enough, and one that was refused still is.  Top-K holds the
// pooled rows and the bit mask, 4 ceil(nk / 32) bytes a row, which fits the nk
// bytes a row counted here (for nk < 4 with the counts after them); the bitmap
// mode counts into the pointer arrays and uses none.
size_t block_mask_ws(const MaskProblem& p, int mode) {
  const size_t H = p.H, nq = p.nq, nk = p.nk, d = p.d;
  size_t counts = (H * (nq > nk ? nq : nk) + 1) * sizeof(int32_t);
  if (mode == UT_MASK_BITMAP) return counts;
  size_t pooled = H * (nq + nk) * d * sizeof(float);
  size_t bitmap = H * nq * nk;
  return pooled + ((bitmap + 255) / 256) * 256 + counts;
}

cudaError_t launch_block_mask_topk(const MaskProblem& p, const void* q, const void* k, int k_rho, int32_t* row_ptr,
                                   int32_t* col_idx, int32_t* col_ptr_t, int32_t* row_idx_t, void* ws,
                                   cudaStream_t stream) {
  const int H = p.H, nq = p.nq, nk = p.nk, d = p.d;
  float* pooled = static_cast<float*>(ws);
  uint32_t* bits = reinterpret_cast<uint32_t*>(pooled + (size_t)H * (nq + nk) * d);
  const int elems = p.dtype == UT_BF16 ? 8 : 4;
  dim3 pg(nq > nk ? nq : nk, 2, (H * d / elems + kPoolThreads - 1) / kPoolThreads);
  if (p.dtype == UT_BF16)
    block_pool_kernel<__nv_bfloat16><<<pg, kPoolThreads, 0, stream>>>(
        static_cast<const __nv_bfloat16*>(q), static_cast<const __nv_bfloat16*>(k), p.N, H, d, p.row_stride, p.block,
        nq, p.block_k, nk, pooled);
  else
    block_pool_kernel<float><<<pg, kPoolThreads, 0, stream>>>(static_cast<const float*>(q),
                                                              static_cast<const float*>(k), p.N, H, d, p.row_stride,
                                                              p.block, nq, p.block_k, nk, pooled);
  // query blocks per CTA: as many as keep their scores within 64 KB (three CTAs
  // per SM overlap one's selection with another's products), at least one; the
  // narrower tiles do not compute rows that a CTA does not hold, and the short
  // slice leaves the longest rows their room
  int R = (64 * 1024) / (nk * 4);
  R = R < 1 ? 1 : (R > kSelRows ? kSelRows : R);
  const bool roomy = ((size_t)4 * d + 16 * kSelCols + (size_t)R * nk) * sizeof(float) <= 232448;  // 227 KB a block
  auto launch = nk <= 1024 ? launch_score_select<16, 16, false>
                : R > 8    ? launch_score_select<16, 16, true>
                : R > 4    ? launch_score_select<8, 16, true>
                : roomy    ? launch_score_select<4, 16, true>
                           : launch_score_select<4, 4, true>;
  const cudaError_t e = launch(pooled, H, d, nq, nk, R, k_rho, row_ptr, col_idx, bits, stream);
  if (e != cudaSuccess) return e;
  if (col_ptr_t && row_idx_t)
    transpose_kernel<<<dim3(H, (nk + 31) / 32), kTransThreads, 0, stream>>>(bits, col_idx, H, nq, nk, k_rho,
                                                                          col_ptr_t, row_idx_t);
  return cudaGetLastError();
}

cudaError_t launch_block_mask_bitmap(const MaskProblem& p, const uint8_t* bitmap, int32_t* row_ptr, int32_t* col_idx,
                                     int32_t* col_ptr_t, int32_t* row_idx_t, int64_t col_cap, int32_t* status,
                                     cudaStream_t stream) {
  const bool with_cols = col_ptr_t && row_idx_t;
  const int lines = p.H * (with_cols && p.nk > p.nq ? p.nk : p.nq);
  const dim3 grid((lines + 7) / 8, with_cols ? 2 : 1);
  if (lines == 0) return cudaSuccess;
  bitmap_count_kernel<<<grid, 256, 0, stream>>>(bitmap, p.H, p.nq, p.nk, row_ptr, col_ptr_t);
  scan_kernel<<<with_cols ? 2 : 1, 1024, 0, stream>>>(p.H * p.nq, p.H * p.nk, row_ptr, col_ptr_t);
  bitmap_fill_kernel<<<grid, 256, 0, stream>>>(bitmap, p.H, p.nq, p.nk, row_ptr, col_idx, col_ptr_t, row_idx_t, col_cap,
                                              status);
  return cudaGetLastError();
}

}  // namespace ut
