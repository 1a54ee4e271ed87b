// Block-sparse attention on the CUDA cores in fp32 arithmetic (Sec. 3.3): the
// path for fp32 inputs, whose tolerance rules out tf32 tensor cores.
//
//   attn_bwd_pre_kernel  D_r = dO_r . O_r.
//   attn_*_f32_kernel    a cluster of two CTAs per 32 own rows of a head, walking
//                        the rows of the other side that its block lists:
//     kFwd   own Q, other K, V: online softmax; O, LSE.
//     kDq    own Q, dO, other K, V: dQ_r = scale * sum_k P_rk (dO_r . V_k - D_r) K_k.
//     kDkv   own K, V, other Q, dO over the transposed lists (query blocks that
//            listed the key block): dV_k = sum_r P_rk dO_r,
//            dK_k = scale * sum_r dS_rk Q_r.
//
// What bounds it: fp32 FMAs (152 SMs x 128 a cycle), fed from shared memory.  A
// thread that owns a whole row reads one shared value per FMA and leaves one
// warp per SM at these sizes; here a 32 x (4096/D) tile of scores is spread over
// 128 threads in 4 x 4 (D = 128: 4 x 2) register tiles, so that eight 16-byte
// shared loads feed 64 FMAs, two to an instruction (even and odd d summed
// apart), and the tile goes through shared memory to the second product.  The
// two groups of 128 threads in each of the cluster's CTAs take chunks of the list
// in turn (few own tiles exist at these sizes and some lists are far longer than
// the others, so the list is what is left to split) and add their sums at the
// end, across the CTAs through distributed shared memory; each group copies its next chunk with cp.async while
// it works on the present one.  The row maximum is updated once per chunk, not
// per key.
// Measured: forward and backward of 2,002 tokens, 2 heads, D = 64, 32-row blocks
// 8,746 -> 243 us with one CTA per tile (45 forward, 193 backward), 201 with two
// (47, 150); the whole path over 195 tokens 1,414 -> 233 -> 168 us, the last with
// less host work.  Errors against 64 bits 7.2e-7 -> 4.0e-7 (fewer rescalings,
// shorter chains).
#include <math.h>

#include "common.cuh"
#include "kernels.h"

namespace ut {

constexpr int kOwn = 32;          // own rows per CTA
constexpr int kGroups = 2;        // thread groups of a CTA
constexpr int kParts = 2;         // CTAs of a cluster: kGroups * kParts groups share the list
constexpr int kGroupThreads = 128;
constexpr int kF32Threads = kGroups * kGroupThreads;

enum F32Mode { kFwd = 0, kDq = 1, kDkv = 2 };

struct F32Args {
  const float *q, *k, *v, *o, *dout, *lse;
  float* dsum;               // D, [H, N]
  const int32_t *ptr, *idx;  // lists of the own side's blocks
  float *out0, *out1;        // kFwd: O, LSE; kDq: dQ, -; kDkv: dV, dK
  int64_t N, rs;
  int H, b, nb;              // own blocks of b rows, nb per head
  float scale;
};

template <int D, int MODE>
struct F32Smem {
  static constexpr int KC = 4096 / D;  // rows of the other side per chunk: 64 or 32
  static constexpr int LD = D + 4;     // padded row: 16-byte reads of 8 rows meet 32 different banks
  static constexpr int LP = KC + 4;
  float a1[kOwn * LD];
  float a2[MODE == kFwd ? 4 : kOwn * LD];
  struct Stage {
    float b1[KC * LD], b2[KC * LD];
    float lse[KC], dsum[KC];
  };
  struct Group {
    Stage st[2];
    float p[kOwn * LP];
    float ds[MODE == kDkv ? kOwn * LP : 4];
  } g[kGroups];
};

UT_DEV void cp_async16(float* dst, const float* src, bool ok) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_u32(dst)), "l"(src), "r"(ok ? 16 : 0)
               : "memory");
}
UT_DEV void cp_async4(float* dst, const float* src, bool ok) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(smem_u32(dst)), "l"(src), "r"(ok ? 4 : 0)
               : "memory");
}
UT_DEV void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
UT_DEV void cp_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}
// Address of the same shared variable in CTA `rank` of the cluster, a store
// there, and the cluster's barrier (release / acquire).
UT_DEV uint32_t cluster_addr(const void* p, uint32_t rank) {
  uint32_t a;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(smem_u32(p)), "r"(rank));
  return a;
}
UT_DEV void st_cluster(uint32_t addr, float v) {
  asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(addr), "f"(v) : "memory");
}
UT_DEV void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
UT_DEV void group_sync(int g) { asm volatile("bar.sync %0, %1;" ::"r"(g + 1), "n"(kGroupThreads) : "memory"); }

// rows r0 .. r0 + valid - 1 of head h into dst[0 .. rows) (padded rows), zeros
// beyond; `threads` threads, this one number t.  kVec: 16-byte aligned source
// rows (row strides always are; a base may be aligned to 4 bytes only).
template <int D, bool kVec>
UT_DEV void copy_rows(float* dst, const float* src, int64_t r0, int valid, int rows, int64_t off, int64_t rs, int t,
                      int threads) {
  constexpr int LD = D + 4;
  if constexpr (kVec) {
    for (int x = t; x < rows * (D / 4); x += threads) {
      const int r = x / (D / 4), e = (x % (D / 4)) * 4;
      const bool ok = r < valid;
      cp_async16(dst + r * LD + e, src + (ok ? (r0 + r) * rs + off + e : 0), ok);
    }
  } else {
    for (int x = t; x < rows * D; x += threads) {
      const int r = x / D, e = x % D;
      const bool ok = r < valid;
      cp_async4(dst + r * LD + e, src + (ok ? (r0 + r) * rs + off + e : 0), ok);
    }
  }
}

// acc[y][x] = A[rg * 4 + y] . B[c + 16 x] over D
template <int D, int NX>
UT_DEV void dots(const float* A, const float* B, int rg, int c, float (&acc)[4][NX]) {
  constexpr int LD = D + 4;
  float2 s[4][NX];
#pragma unroll
  for (int y = 0; y < 4; ++y)
#pragma unroll
    for (int x = 0; x < NX; ++x) s[y][x] = make_float2(0.f, 0.f);
#pragma unroll 4
  for (int e = 0; e < D; e += 4) {
    float4 av[4], bv[NX];
#pragma unroll
    for (int y = 0; y < 4; ++y) av[y] = *reinterpret_cast<const float4*>(A + (rg * 4 + y) * LD + e);
#pragma unroll
    for (int x = 0; x < NX; ++x) bv[x] = *reinterpret_cast<const float4*>(B + (c + 16 * x) * LD + e);
#pragma unroll
    for (int y = 0; y < 4; ++y)
#pragma unroll
      for (int x = 0; x < NX; ++x) {
        s[y][x] = ffma2(make_float2(av[y].x, av[y].y), make_float2(bv[x].x, bv[x].y), s[y][x]);
        s[y][x] = ffma2(make_float2(av[y].z, av[y].w), make_float2(bv[x].z, bv[x].w), s[y][x]);
      }
  }
#pragma unroll
  for (int y = 0; y < 4; ++y)
#pragma unroll
    for (int x = 0; x < NX; ++x) acc[y][x] = s[y][x].x + s[y][x].y;
}

// acc[y][.] += sum_k P[rg * 4 + y][k] B[k][this thread's D/16 columns: c * 4 .. and, for D = 128, 64 + c * 4 ..]
template <int D>
UT_DEV void accumulate(const float* P, const float* B, int rg, int c, float2 (&acc)[4][D / 32]) {
  constexpr int KC = 4096 / D, LD = D + 4, LP = KC + 4;
#pragma unroll 2
  for (int k = 0; k < KC; k += 4) {
    float4 pv[4];
#pragma unroll
    for (int y = 0; y < 4; ++y) pv[y] = *reinterpret_cast<const float4*>(P + (rg * 4 + y) * LP + k);
#pragma unroll
    for (int kk = 0; kk < 4; ++kk) {
      float4 bv[D / 64];
#pragma unroll
      for (int x = 0; x < D / 64; ++x) bv[x] = *reinterpret_cast<const float4*>(B + (k + kk) * LD + 64 * x + c * 4);
#pragma unroll
      for (int y = 0; y < 4; ++y) {
        const float p = kk == 0 ? pv[y].x : (kk == 1 ? pv[y].y : (kk == 2 ? pv[y].z : pv[y].w));
        const float2 pp = make_float2(p, p);
#pragma unroll
        for (int x = 0; x < D / 64; ++x) {
          acc[y][2 * x] = ffma2(pp, make_float2(bv[x].x, bv[x].y), acc[y][2 * x]);
          acc[y][2 * x + 1] = ffma2(pp, make_float2(bv[x].z, bv[x].w), acc[y][2 * x + 1]);
        }
      }
    }
  }
}

// this thread's columns of row y, times f[y], to global rows (own row rg * 4 + y)
template <int D, bool kVec>
UT_DEV void store_rows(float* out, int64_t r0, int valid, int64_t off, int64_t rs, int rg, int c,
                       const float2 (&acc)[4][D / 32], const float (&f)[4]) {
#pragma unroll
  for (int y = 0; y < 4; ++y) {
    const int r = rg * 4 + y;
    if (r >= valid) continue;
    float* row = out + (r0 + r) * rs + off;
#pragma unroll
    for (int x = 0; x < D / 64; ++x) {
      const float4 v = make_float4(acc[y][2 * x].x * f[y], acc[y][2 * x].y * f[y], acc[y][2 * x + 1].x * f[y],
                                   acc[y][2 * x + 1].y * f[y]);
      float* p = row + 64 * x + c * 4;
      if (kVec) {
        *reinterpret_cast<float4*>(p) = v;
      } else {
        p[0] = v.x;
        p[1] = v.y;
        p[2] = v.z;
        p[3] = v.w;
      }
    }
  }
}

template <int D, int MODE, bool kVec>
UT_DEV void f32_tile(const F32Args& a, F32Smem<D, MODE>& sm, int part) {
  using S = F32Smem<D, MODE>;
  constexpr int KC = S::KC, NX = KC / 16, LP = S::LP, NC = D / 32, kSubs = KC / 32;
  const int g = threadIdx.x / kGroupThreads, t = threadIdx.x % kGroupThreads;
  const int gg = part * kGroups + g;  // this group among all that share the list
  constexpr int kAll = kGroups * kParts;
  const int rg = t / 16, c = t % 16;  // rows rg * 4 .. + 3; columns c + 16 x of the scores, c * 4 .. of the outputs
  const int h = blockIdx.y;
  const int64_t r0 = (int64_t)blockIdx.x * kOwn, off = (int64_t)h * D;
  const int valid = (int)min((int64_t)kOwn, a.N - r0);
  const float* own1 = MODE == kDkv ? a.k : a.q;
  const float* own2 = MODE == kDkv ? a.v : a.dout;
  const float* oth1 = MODE == kDkv ? a.q : a.k;
  const float* oth2 = MODE == kDkv ? a.dout : a.v;
  const int line = h * a.nb + (int)(r0 / a.b);
  const int p0 = a.ptr[line], per = a.b / 32;  // 32-row pieces of a block
  const int pieces = (a.ptr[line + 1] - p0) * per, chunks = (pieces + kSubs - 1) / kSubs;
  auto piece = [&](int s, int64_t& row, int& n) {  // piece s of the list: first row, rows that exist
    row = 0;
    n = 0;
    if (s < pieces) {
      row = (int64_t)a.idx[p0 + s / per] * a.b + (s % per) * 32;
      n = (int)max((int64_t)0, min((int64_t)32, a.N - row));
    }
  };
  auto load = [&](int ch, int stage) {
    auto& st = sm.g[g].st[stage];
#pragma unroll
    for (int u = 0; u < kSubs; ++u) {
      int64_t row;
      int n;
      piece(ch * kSubs + u, row, n);
      copy_rows<D, kVec>(st.b1 + u * 32 * S::LD, oth1, row, n, 32, off, a.rs, t, kGroupThreads);
      copy_rows<D, kVec>(st.b2 + u * 32 * S::LD, oth2, row, n, 32, off, a.rs, t, kGroupThreads);
      if (MODE == kDkv && t < 64) {
        const float* src = t < 32 ? a.lse : a.dsum;
        float* dst = (t < 32 ? st.lse : st.dsum) + u * 32 + (t & 31);
        const bool ok = (t & 31) < n;
        cp_async4(dst, src + (ok ? (int64_t)h * a.N + row + (t & 31) : 0), ok);
      }
    }
  };
  copy_rows<D, kVec>(sm.a1, own1, r0, valid, kOwn, off, a.rs, threadIdx.x, kF32Threads);
  if (MODE != kFwd) copy_rows<D, kVec>(sm.a2, own2, r0, valid, kOwn, off, a.rs, threadIdx.x, kF32Threads);
  cp_commit();
  if (gg < chunks) load(gg, 0);
  cp_commit();
  cp_wait<1>();
  __syncthreads();
  float2 acc[4][NC], acc2[MODE == kDkv ? 4 : 1][NC];
#pragma unroll
  for (int y = 0; y < 4; ++y)
#pragma unroll
    for (int x = 0; x < NC; ++x) {
      acc[y][x] = make_float2(0.f, 0.f);
      if (MODE == kDkv) acc2[y][x] = make_float2(0.f, 0.f);
    }
  float m[4], l[4], lse_r[4], d_r[4];
#pragma unroll
  for (int y = 0; y < 4; ++y) {
    m[y] = -INFINITY;
    l[y] = 0.f;
    const int r = rg * 4 + y;
    lse_r[y] = MODE == kDq && r < valid ? a.lse[(int64_t)h * a.N + r0 + r] : 0.f;
    d_r[y] = MODE == kDq && r < valid ? a.dsum[(int64_t)h * a.N + r0 + r] : 0.f;
  }
  int stage = 0;
  for (int ch = gg; ch < chunks; ch += kAll, stage ^= 1) {
    if (ch + kAll < chunks) load(ch + kAll, stage ^ 1);
    cp_commit();
    cp_wait<1>();
    group_sync(g);
    auto& st = sm.g[g].st[stage];
    float* P = sm.g[g].p;
    bool exists[NX];  // columns beyond the list or beyond N
#pragma unroll
    for (int x = 0; x < NX; ++x) {
      int64_t row;
      int n;
      piece(ch * kSubs + (c + 16 * x) / 32, row, n);
      exists[x] = ((c + 16 * x) & 31) < n;
    }
    float s[4][NX];
    dots<D, NX>(sm.a1, st.b1, rg, c, s);
    if constexpr (MODE == kFwd) {
#pragma unroll
      for (int y = 0; y < 4; ++y) {
        float mx = -INFINITY;
#pragma unroll
        for (int x = 0; x < NX; ++x) {
          s[y][x] = exists[x] ? s[y][x] * a.scale : -INFINITY;
          mx = fmaxf(mx, s[y][x]);
        }
#pragma unroll
        for (int w = 8; w; w >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, w));
        const float mn = fmaxf(m[y], mx);
        const float ref = mn == -INFINITY ? 0.f : mn;  // nothing seen yet: exp(-inf - 0) = 0
        const float alpha = expf(m[y] - ref);
        m[y] = mn;
        float sum = 0.f;
#pragma unroll
        for (int x = 0; x < NX; ++x) {
          const float p = expf(s[y][x] - ref);
          sum += p;
          P[(rg * 4 + y) * LP + c + 16 * x] = p;
        }
        l[y] = l[y] * alpha + sum;  // this thread's columns only; added up at the end
#pragma unroll
        for (int x = 0; x < NC; ++x) {
          acc[y][x].x *= alpha;
          acc[y][x].y *= alpha;
        }
      }
    } else {
      float dp[4][NX];
      dots<D, NX>(sm.a2, st.b2, rg, c, dp);
#pragma unroll
      for (int x = 0; x < NX; ++x) {
        const float ls = MODE == kDkv ? st.lse[c + 16 * x] : 0.f, dd = MODE == kDkv ? st.dsum[c + 16 * x] : 0.f;
#pragma unroll
        for (int y = 0; y < 4; ++y) {
          const float p = exists[x] ? expf(s[y][x] * a.scale - (MODE == kDq ? lse_r[y] : ls)) : 0.f;
          const float ds = p * (dp[y][x] - (MODE == kDq ? d_r[y] : dd)) * a.scale;
          if (MODE == kDq) {
            P[(rg * 4 + y) * LP + c + 16 * x] = exists[x] ? ds : 0.f;
          } else {
            P[(rg * 4 + y) * LP + c + 16 * x] = p;
            sm.g[g].ds[(rg * 4 + y) * LP + c + 16 * x] = exists[x] ? ds : 0.f;
          }
        }
      }
    }
    group_sync(g);
    accumulate<D>(P, MODE == kDq ? st.b1 : st.b2, rg, c, acc);
    if constexpr (MODE == kDkv) accumulate<D>(sm.g[g].ds, st.b1, rg, c, acc2);
    group_sync(g);  // this stage and the tile are free for the chunk after the next
  }
  // the groups' sums: the second group's through the first one's stages, then
  // the second CTA's through the second group's stages of the first CTA (no copy
  // is in flight in either)
  cp_wait<0>();
  constexpr int kVals = 4 * NC * 2 * (MODE == kDkv ? 2 : 1) + 8;
  static_assert(kVals * kGroupThreads * sizeof(float) <= sizeof(typename S::Stage) * 2, "merge area");
  static_assert(kGroups == 2 && kParts == 2, "each merge adds one to the other");
  if constexpr (MODE == kFwd) {
#pragma unroll
    for (int y = 0; y < 4; ++y)
#pragma unroll
      for (int w = 8; w; w >>= 1) l[y] += __shfl_xor_sync(0xffffffffu, l[y], w);
  }
  auto give = [&](auto put) {  // put(n, value)
    int n = 0;
#pragma unroll
    for (int y = 0; y < 4; ++y)
#pragma unroll
      for (int x = 0; x < NC; ++x) {
        put(n++, acc[y][x].x);
        put(n++, acc[y][x].y);
        if (MODE == kDkv) {
          put(n++, acc2[y][x].x);
          put(n++, acc2[y][x].y);
        }
      }
#pragma unroll
    for (int y = 0; y < 4; ++y) {
      put(n++, m[y]);
      put(n++, l[y]);
    }
  };
  auto add = [&](const float* ex) {
    float f0[4], f1[4];
#pragma unroll
    for (int y = 0; y < 4; ++y) {
      f0[y] = f1[y] = 1.f;
      if (MODE == kFwd) {
        const float mo = ex[(4 * NC * 2 + 2 * y) * kGroupThreads], lo = ex[(4 * NC * 2 + 2 * y + 1) * kGroupThreads];
        const float mn = fmaxf(m[y], mo), ref = mn == -INFINITY ? 0.f : mn;
        f0[y] = expf(m[y] - ref);
        f1[y] = expf(mo - ref);
        l[y] = l[y] * f0[y] + lo * f1[y];
        m[y] = mn;
      }
    }
    int n = 0;
#pragma unroll
    for (int y = 0; y < 4; ++y)
#pragma unroll
      for (int x = 0; x < NC; ++x) {
        acc[y][x].x = acc[y][x].x * f0[y] + ex[n++ * kGroupThreads] * f1[y];
        acc[y][x].y = acc[y][x].y * f0[y] + ex[n++ * kGroupThreads] * f1[y];
        if (MODE == kDkv) {
          acc2[y][x].x += ex[n++ * kGroupThreads];
          acc2[y][x].y += ex[n++ * kGroupThreads];
        }
      }
  };
  float* ex0 = reinterpret_cast<float*>(&sm.g[0].st[0]) + t;
  float* ex1 = reinterpret_cast<float*>(&sm.g[1].st[0]) + t;
  __syncthreads();
  if (g == 1) give([&](int n, float v) { ex0[n * kGroupThreads] = v; });
  __syncthreads();
  if (g == 0) add(ex0);
  cluster_sync();  // the first CTA's second group is done with its stages
  if (part == 1 && g == 0) {
    const uint32_t to = cluster_addr(ex1, 0);
    give([&](int n, float v) { st_cluster(to + n * kGroupThreads * (uint32_t)sizeof(float), v); });
  }
  cluster_sync();
  if (part != 0 || g != 0) return;
  add(ex1);
  float f[4];
#pragma unroll
  // a row that lists nothing gets O = 0; one whose scores are all -inf has no
  // softmax (0 / 0)
  for (int y = 0; y < 4; ++y) f[y] = MODE == kFwd ? (l[y] > 0.f ? 1.f / l[y] : (pieces > 0 ? NAN : 0.f)) : 1.f;
  store_rows<D, kVec>(a.out0, r0, valid, off, a.rs, rg, c, acc, f);
  if constexpr (MODE == kDkv) store_rows<D, kVec>(a.out1, r0, valid, off, a.rs, rg, c, acc2, f);
  if (MODE == kFwd && c == 0) {
#pragma unroll
    for (int y = 0; y < 4; ++y)
      if (rg * 4 + y < valid)
        a.out1[(int64_t)h * a.N + r0 + rg * 4 + y] = l[y] > 0.f ? m[y] + logf(l[y]) : -INFINITY;
  }
}

// grid (own tiles, H, kParts): a cluster spans z
template <int D>
__global__ void __cluster_dims__(1, 1, kParts) __launch_bounds__(kF32Threads, 1)
    attn_fwd_f32_kernel(const F32Args a) {
  extern __shared__ __align__(16) uint8_t smem_raw[];
  f32_tile<D, kFwd, true>(a, *reinterpret_cast<F32Smem<D, kFwd>*>(smem_raw), blockIdx.z);
}

// grid (own tiles, H, 2 kParts): the first kParts of z the query tiles (dQ), the
// others the key tiles (dK, dV)
template <int D, bool kVec>
__global__ void __cluster_dims__(1, 1, kParts) __launch_bounds__(kF32Threads, 1)
    attn_bwd_f32_kernel(const F32Args dq, const F32Args dkv) {
  extern __shared__ __align__(16) uint8_t smem_raw[];
  const int part = blockIdx.z % kParts;
  if (blockIdx.z < kParts) f32_tile<D, kDq, kVec>(dq, *reinterpret_cast<F32Smem<D, kDq>*>(smem_raw), part);
  else f32_tile<D, kDkv, kVec>(dkv, *reinterpret_cast<F32Smem<D, kDkv>*>(smem_raw), part);
}

// D_r = dO_r . O_r: 16 lanes per (row, head)
__global__ void __launch_bounds__(256) attn_bwd_pre_kernel(const float* __restrict__ o, const float* __restrict__ dout,
                                                           int64_t N, int H, int d, int64_t rs,
                                                           float* __restrict__ dsum) {
  const int64_t x = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / 16;
  const int lane = threadIdx.x & 15;
  const bool ok = x < N * H;
  const int64_t r = ok ? x / H : 0, off = r * rs + (ok ? x % H : 0) * d;
  float s = 0.f;
  if (ok)
    for (int e = lane; e < d; e += 16) s = fmaf(o[off + e], dout[off + e], s);
  for (int w = 8; w; w >>= 1) s += __shfl_xor_sync(0xffffffffu, s, w);
  if (ok && lane == 0) dsum[(x % H) * N + r] = s;
}

// ----------------------------------------------------------------- launchers
static bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

template <int D>
static cudaError_t fwd_impl(const AttnProblem& p, const F32Args& a, cudaStream_t s) {
  constexpr size_t smem = sizeof(F32Smem<D, kFwd>);
  cudaError_t e = cudaFuncSetAttribute(attn_fwd_f32_kernel<D>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  attn_fwd_f32_kernel<D><<<dim3((unsigned)((p.N + kOwn - 1) / kOwn), p.H, kParts), kF32Threads, smem, s>>>(a);
  return cudaGetLastError();
}

static F32Args args_of(const AttnProblem& p, const void* q, const void* k, const void* v) {
  F32Args a{};
  a.q = static_cast<const float*>(q);
  a.k = static_cast<const float*>(k);
  a.v = static_cast<const float*>(v);
  a.N = p.N;
  a.rs = p.row_stride;
  a.H = p.H;
  a.b = p.block;
  a.nb = p.nq;
  a.scale = p.scale;
  return a;
}

cudaError_t launch_attn_fwd_simt(const AttnProblem& p, const void* q, const void* k, const void* v,
                                 const int32_t* row_ptr, const int32_t* col_idx, void* o, float* lse,
                                 cudaStream_t stream) {
  if (p.nq == 0) return cudaSuccess;
  F32Args a = args_of(p, q, k, v);
  a.ptr = row_ptr;
  a.idx = col_idx;
  a.out0 = static_cast<float*>(o);
  a.out1 = lse;
  return p.d == 64 ? fwd_impl<64>(p, a, stream) : fwd_impl<128>(p, a, stream);
}

size_t attn_bwd_simt_ws(const AttnProblem& p) { return (size_t)p.H * p.N * sizeof(float); }

template <int D, bool kVec>
static cudaError_t bwd_impl(const AttnProblem& p, const F32Args& dq, const F32Args& dkv, cudaStream_t s) {
  constexpr size_t s1 = sizeof(F32Smem<D, kDq>), s2 = sizeof(F32Smem<D, kDkv>), smem = s1 > s2 ? s1 : s2;
  static_assert(smem <= 232448, "fp32 backward shared layout exceeds the per-block limit");
  cudaError_t e =
      cudaFuncSetAttribute(attn_bwd_f32_kernel<D, kVec>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  attn_bwd_f32_kernel<D, kVec>
      <<<dim3((unsigned)((p.N + kOwn - 1) / kOwn), p.H, 2 * kParts), kF32Threads, smem, s>>>(dq, dkv);
  return cudaGetLastError();
}

cudaError_t launch_attn_bwd_simt(const AttnProblem& p, const void* q, const void* k, const void* v, const void* o,
                                 const float* lse, const void* dout, const int32_t* row_ptr, const int32_t* col_idx,
                                 const int32_t* col_ptr_t, const int32_t* row_idx_t, void* dq, void* dk, void* dv,
                                 void* ws, cudaStream_t stream) {
  if (p.nq == 0) return cudaSuccess;
  F32Args a = args_of(p, q, k, v);
  a.o = static_cast<const float*>(o);
  a.dout = static_cast<const float*>(dout);
  a.lse = lse;
  a.dsum = static_cast<float*>(ws);
  const int64_t threads = p.N * p.H * 16;
  attn_bwd_pre_kernel<<<(unsigned)((threads + 255) / 256), 256, 0, stream>>>(a.o, a.dout, p.N, p.H, p.d, p.row_stride,
                                                                             a.dsum);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  F32Args x = a, y = a;
  x.ptr = row_ptr;
  x.idx = col_idx;
  x.out0 = static_cast<float*>(dq);
  y.ptr = col_ptr_t;
  y.idx = row_idx_t;
  y.out0 = static_cast<float*>(dv);
  y.out1 = static_cast<float*>(dk);
  const bool vec = aligned16(q) && aligned16(k) && aligned16(v) && aligned16(dout) && aligned16(dq) && aligned16(dk) &&
                   aligned16(dv);
  if (p.d == 64) return vec ? bwd_impl<64, true>(p, x, y, stream) : bwd_impl<64, false>(p, x, y, stream);
  return vec ? bwd_impl<128, true>(p, x, y, stream) : bwd_impl<128, false>(p, x, y, stream);
}

}  // namespace ut
