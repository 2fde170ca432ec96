// Grouped fp32 products of a tensor with a narrow factor (1..64 columns), any sizes, strides and ranks: the
// projections V_m = A_m^T U_m, the expansions P_m = A_m V_m (Algorithm 1), the core products and the first
// contraction of the linear backward wherever no shape-specialised kernel applies.  One launch runs several
// products (the modes of a layer), a CTA finds its product in a table.
//
//   C[m][j] = sum_k A(m, k) B[k][j]      m: 32 rows per CTA, j < n <= BN, k in chunks of 128
//     m-major A (a projection of a strided mode, the expansion of the last mode): A(m, k) = X[o sxo + k ld + m]
//     k-major A (a projection of the last mode, the expansion of a strided mode): A(m, k) = X[(k / kin) sxo + m ld + k % kin]
//
// What bounds it: the factor is so narrow that a product is a stream over X; with 32 x n outputs per CTA there are
// few CTAs and a long contraction, so the eight warps of a CTA split every chunk of 128 along k (16 each, all 32
// rows and all columns in registers) and meet once, at the end, in warp order.  fp32 tensors with 16-byte rows
// arrive by cp.async two or three chunks ahead; bf16 and ragged tensors pass through registers one chunk ahead.
#include <cuda_bf16.h>

#include <algorithm>
#include <cstring>

#include "asi_internal.h"

namespace asi {

namespace {

constexpr int kGT = 256, kGW = 8, kGM = 32, kGK = 128;
constexpr int kPK = kGK + 4;             // pitch of a k-major tile: rows four banks apart

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void cp16(float* dst, const void* src, bool on) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_u32(dst)), "l"(src), "r"(on ? 16 : 0) : "memory");
}
__device__ __forceinline__ void cp4(float* dst, const void* src, bool on) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(smem_u32(dst)), "l"(src), "r"(on ? 4 : 0) : "memory");
}
__device__ __forceinline__ float as_f(float v) { return v; }
__device__ __forceinline__ float as_f(__nv_bfloat16 v) { return __bfloat162float(v); }

// What passes through registers between global and shared memory: four 8-byte groups of bf16 or 16 single values
template <typename TX, bool VEC> struct Regs { TX v[16]; };
template <> struct Regs<__nv_bfloat16, true> { uint2 v[4]; };

__device__ __forceinline__ int cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return (int)r;
}
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ float ld_cluster(const float* own, int rank) {
  uint32_t a;
  float v;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;"
               : "=r"(a)
               : "r"(static_cast<uint32_t>(__cvta_generic_to_shared(own))), "r"(rank));
  asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(a) : "memory");
  return v;
}

template <typename TX, bool KM, bool VEC, int BN>
struct GemmTile {
  static constexpr bool kAsync = VEC && sizeof(TX) == 4;
  static constexpr int kTileA = KM ? kGM * kPK : kGK * kGM;      // floats
  static constexpr int kTileB = kGK * BN;

  // A chunk [k0, k0 + 128) x rows [m0, m0 + 32): position of element / vector t of this thread
  static __device__ __forceinline__ void issue_async(float* As, const TX* X, const GemmArg& p, int m0, int k0, int kend) {
    const int tid = threadIdx.x;
    if constexpr (KM) {
      const int v = tid & 31, k = k0 + 4 * v;
      const bool kon = k < kend;
      const int o = (kon && p.kin < p.K) ? k / p.kin : 0;
      const TX* src = X + (kon ? (int64_t)o * p.sxo + (k - o * p.kin) : 0);
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        const int m = (tid >> 5) + 8 * t;
        const bool on = kon && m0 + m < p.M;
        cp16(As + m * kPK + 4 * v, src + (on ? (int64_t)(m0 + m) * p.ld : 0), on);
      }
    } else {
      const int v = tid & 7, m = m0 + 4 * v;
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        const int k = (tid >> 3) + 32 * t;
        const bool on = k0 + k < kend && m < p.M;
        cp16(As + k * kGM + 4 * v, X + (on ? (int64_t)(k0 + k) * p.ld + m : 0), on);
      }
    }
  }
  static __device__ __forceinline__ void load_regs(Regs<TX, VEC>& rg, const TX* X, const GemmArg& p, int m0, int k0, int kend) {
    const int tid = threadIdx.x;
    if constexpr (VEC) {
      static_assert(sizeof(TX) == 2, "fp32 vectors go through cp.async");
      if constexpr (KM) {
        const int k = k0 + 4 * (tid & 31);
        const bool kon = k < kend;
        const int o = (kon && p.kin < p.K) ? k / p.kin : 0;
        const TX* src = X + (kon ? (int64_t)o * p.sxo + (k - o * p.kin) : 0);
#pragma unroll
        for (int t = 0; t < 4; ++t) {
          const int m = m0 + (tid >> 5) + 8 * t;
          rg.v[t] = __ldg(reinterpret_cast<const uint2*>(src + ((kon && m < p.M) ? (int64_t)m * p.ld : 0)));
        }
      } else {
        const int m = m0 + 4 * (tid & 7);
#pragma unroll
        for (int t = 0; t < 4; ++t) {
          const int k = k0 + (tid >> 3) + 32 * t;
          rg.v[t] = __ldg(reinterpret_cast<const uint2*>(X + ((k < kend && m < p.M) ? (int64_t)k * p.ld + m : 0)));
        }
      }
    } else if constexpr (KM) {
      const int k = k0 + (tid & 127);
      const bool kon = k < kend;
      const int o = (kon && p.kin < p.K) ? k / p.kin : 0;
      const TX* src = X + (kon ? (int64_t)o * p.sxo + (k - o * p.kin) : 0);
#pragma unroll
      for (int t = 0; t < 16; ++t) {
        const int m = m0 + (tid >> 7) + 2 * t;
        rg.v[t] = src[(kon && m < p.M) ? (int64_t)m * p.ld : 0];
      }
    } else {
      const int m = m0 + (tid & 31);
#pragma unroll
      for (int t = 0; t < 16; ++t) {
        const int k = k0 + (tid >> 5) + 8 * t;
        rg.v[t] = X[(k < kend && m < p.M) ? (int64_t)k * p.ld + m : 0];
      }
    }
  }
  static __device__ __forceinline__ void store_regs(const Regs<TX, VEC>& rg, float* As, const GemmArg& p, int m0, int k0, int kend) {
    const int tid = threadIdx.x;
    if constexpr (VEC) {
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        int m, k;
        float* dst;
        if constexpr (KM) { m = (tid >> 5) + 8 * t; k = 4 * (tid & 31); dst = As + m * kPK + k; }
        else { m = 4 * (tid & 7); k = (tid >> 3) + 32 * t; dst = As + k * kGM + m; }
        const bool on = m0 + m < p.M && k0 + k < kend;
        float4 f = make_float4(0.f, 0.f, 0.f, 0.f);
        if (on)
          f = make_float4(__uint_as_float(rg.v[t].x << 16), __uint_as_float(rg.v[t].x & 0xffff0000u),
                          __uint_as_float(rg.v[t].y << 16), __uint_as_float(rg.v[t].y & 0xffff0000u));
        *reinterpret_cast<float4*>(dst) = f;
      }
    } else {
#pragma unroll
      for (int t = 0; t < 16; ++t) {
        int m, k;
        if constexpr (KM) { m = (tid >> 7) + 2 * t; k = tid & 127; }
        else { m = tid & 31; k = (tid >> 5) + 8 * t; }
        As[KM ? m * kPK + k : k * kGM + m] = (m0 + m < p.M && k0 + k < kend) ? as_f(rg.v[t]) : 0.f;
      }
    }
  }
  static __device__ __forceinline__ void issue_b(float* Bs, const float* B, const GemmArg& p, int k0, int kend) {
    const int tid = threadIdx.x;
    if (p.bvec) {
      constexpr int VPR = BN / 4;
#pragma unroll
      for (int t = 0; t < (kGK * VPR + kGT - 1) / kGT; ++t) {
        const int e = tid + t * kGT, k = e / VPR, v = e - k * VPR;
        if (kGK * VPR % kGT && e >= kGK * VPR) break;
        const bool on = k0 + k < kend && 4 * v < p.n;
        cp16(Bs + k * BN + 4 * v, B + (on ? (int64_t)(k0 + k) * p.ldb + 4 * v : 0), on);
      }
    } else {
#pragma unroll 4
      for (int t = 0; t < kGK * BN / kGT; ++t) {
        const int e = tid + t * kGT, k = e / BN, j = e - k * BN;
        const bool on = k0 + k < kend && j < p.n;
        cp4(Bs + e, B + (on ? (int64_t)(k0 + k) * p.ldb + j : 0), on);
      }
    }
  }

  // WIDE: p is one tile of one split, its first k is p.k0
  template <bool CL, bool WIDE>
  static __device__ void run(const GemmArg& p, int cta, int nst, float* smem) {
    constexpr int TN = BN / 4;                         // columns per lane
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, lm = lane & 7, ln = lane >> 3;
    const bool shared = CL && p.ksp > 1;
    const int rank = shared ? cluster_rank() : 0;
    if (shared) cta /= p.ksp;
    const int mt = cta % p.tiles_m, rest = cta / p.tiles_m, o = rest % p.O, split = rest / p.O;
    const int m0 = mt * kGM;
    int kbeg = WIDE ? p.k0 : split * p.kps, kend = WIDE ? p.K : min(p.K, kbeg + p.kps);
    int nit = kend > kbeg ? (kend - kbeg + kGK - 1) / kGK : 0;
    if (shared) {                                      // this CTA's chunks of the tile it shares
      const int per = (nit + p.ksp - 1) / p.ksp;
      kbeg += rank * per * kGK;
      kend = min(kend, kbeg + per * kGK);
      nit = max(0, min(per, nit - rank * per));
    }
    const TX* X = reinterpret_cast<const TX*>(p.X) + (KM ? 0 : (int64_t)o * p.sxo);
    const float* B = p.B;
    float* stage = smem;
    constexpr int kStage = kTileA + kTileB;
    float acc[4][TN];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < TN; ++j) acc[i][j] = 0.f;
    Regs<TX, VEC> rg;
    for (int s = 0; s < nst - 1; ++s) {
      if (s < nit) {
        if constexpr (kAsync) issue_async(stage + s * kStage, X, p, m0, kbeg + s * kGK, kend);
        issue_b(stage + s * kStage + kTileA, B, p, kbeg + s * kGK, kend);
      }
      asm volatile("cp.async.commit_group;" ::: "memory");
    }
    if constexpr (!kAsync) {
      if (nit > 0) {
        load_regs(rg, X, p, m0, kbeg, kend);
        store_regs(rg, stage, p, m0, kbeg, kend);
      }
    }
    int st = 0;
#pragma unroll 1
    for (int it = 0; it < nit; ++it) {
      if (nst == 2) asm volatile("cp.async.wait_group 0;" ::: "memory");
      else asm volatile("cp.async.wait_group 1;" ::: "memory");
      __syncthreads();
      {
        int sf = st + nst - 1;
        if (sf >= nst) sf -= nst;
        if (it + nst - 1 < nit) {
          const int k0 = kbeg + (it + nst - 1) * kGK;
          if constexpr (kAsync) issue_async(stage + sf * kStage, X, p, m0, k0, kend);
          issue_b(stage + sf * kStage + kTileA, B, p, k0, kend);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
      }
      const int k1 = kbeg + (it + 1) * kGK;
      if constexpr (!kAsync) {
        if (it + 1 < nit) load_regs(rg, X, p, m0, k1, kend);
      }
      const float* As = stage + st * kStage;
      const float* Bs = As + kTileA + warp * 16 * BN;
      if (kbeg + it * kGK + warp * 16 < kend) {
#pragma unroll 1
        for (int k4 = 0; k4 < 16; k4 += 4) {           // not unrolled: the loop runs a few dozen times per CTA, and
                                                       // straight-line code stalled on instruction fetch
          float a[4][4];                               // [k][row] (m-major) or [row][k] (k-major)
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const float4 v = KM ? *reinterpret_cast<const float4*>(As + (lm + 8 * i) * kPK + warp * 16 + k4)
                                : *reinterpret_cast<const float4*>(As + (warp * 16 + k4 + i) * kGM + 4 * lm);
            a[i][0] = v.x; a[i][1] = v.y; a[i][2] = v.z; a[i][3] = v.w;
          }
#pragma unroll
          for (int kk = 0; kk < 4; ++kk) {
            const float* b = Bs + (k4 + kk) * BN;
            if constexpr (BN == 8) {
              const float2 v = *reinterpret_cast<const float2*>(b + 2 * ln);
#pragma unroll
              for (int i = 0; i < 4; ++i) {
                const float x = KM ? a[i][kk] : a[kk][i];
                acc[i][0] = fmaf(x, v.x, acc[i][0]);
                acc[i][1] = fmaf(x, v.y, acc[i][1]);
              }
            } else {
#pragma unroll
              for (int q = 0; q < TN / 4; ++q) {
                const float4 v = *reinterpret_cast<const float4*>(b + 4 * ln + 16 * q);
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                  const float x = KM ? a[i][kk] : a[kk][i];
                  acc[i][4 * q] = fmaf(x, v.x, acc[i][4 * q]);
                  acc[i][4 * q + 1] = fmaf(x, v.y, acc[i][4 * q + 1]);
                  acc[i][4 * q + 2] = fmaf(x, v.z, acc[i][4 * q + 2]);
                  acc[i][4 * q + 3] = fmaf(x, v.w, acc[i][4 * q + 3]);
                }
              }
            }
          }
        }
      }
      st = (st + 1 == nst) ? 0 : st + 1;
      if constexpr (!kAsync) {
        if (it + 1 < nit) store_regs(rg, stage + st * kStage, p, m0, k1, kend);
      }
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();
    pdl_launch_dependents();
    // the warps' shares meet in warp order
    float* red = smem;                                 // [8][32][BN]
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      float* dst = red + (warp * kGM + (KM ? lm + 8 * i : 4 * lm + i)) * BN;
      if constexpr (BN == 8) {
        *reinterpret_cast<float2*>(dst + 2 * ln) = make_float2(acc[i][0], acc[i][1]);
      } else {
#pragma unroll
        for (int q = 0; q < TN / 4; ++q)
          *reinterpret_cast<float4*>(dst + 4 * ln + 16 * q) =
              make_float4(acc[i][4 * q], acc[i][4 * q + 1], acc[i][4 * q + 2], acc[i][4 * q + 3]);
      }
    }
    __syncthreads();
    float* Y = p.Y + (int64_t)split * p.ysplit + (int64_t)o * p.so;
    if (shared) {
      // the CTA's sum in place, then CTA `rank` adds its share of the tile over the cluster in rank order; it tells its
      // peers that it is done with theirs before it stores
      for (int e = tid; e < kGM * BN; e += kGT) {
        float v = red[e];
#pragma unroll
        for (int w = 1; w < kGW; ++w) v += red[w * kGM * BN + e];
        red[e] = v;
      }
      cluster_arrive();
      cluster_wait();
      const int per = kGM * BN / p.ksp;                // 32 values or more
      constexpr int kItems = kGM * BN / 2 / kGT > 0 ? kGM * BN / 2 / kGT : 1;
      float sum[kItems];
#pragma unroll
      for (int u = 0; u < kItems; ++u) {
        const int e = tid + u * kGT;
        const float* src = red + rank * per + (e < per ? e : 0);
        float v[8];
#pragma unroll
        for (int t = 0; t < 8; ++t) v[t] = ld_cluster(src, t < p.ksp ? t : 0);
        sum[u] = v[0];
#pragma unroll
        for (int t = 1; t < 8; ++t) sum[u] += t < p.ksp ? v[t] : 0.f;
      }
      cluster_arrive();
#pragma unroll
      for (int u = 0; u < kItems; ++u) {
        const int e = tid + u * kGT, m = (rank * per + e) / BN, j = (rank * per + e) % BN;
        if (e < per && m0 + m < p.M && j < p.n) Y[(int64_t)j * p.sj + (int64_t)(m0 + m) * p.si] = sum[u];
      }
      cluster_wait();
      return;
    }
    if (BN >= 16 && p.sj == 1 && p.yvec) {              // rows of C are contiguous: four columns at a time
#pragma unroll 1
      for (int e = tid; e < kGM * BN / 4; e += kGT) {
        const int m = e / (BN / 4), j = 4 * (e - m * (BN / 4));
        float4 v = *reinterpret_cast<const float4*>(red + m * BN + j);
#pragma unroll
        for (int w = 1; w < kGW; ++w) {
          const float4 t = *reinterpret_cast<const float4*>(red + (w * kGM + m) * BN + j);
          v.x += t.x; v.y += t.y; v.z += t.z; v.w += t.w;
        }
        if (m0 + m < p.M && j < p.n) *reinterpret_cast<float4*>(Y + (int64_t)(m0 + m) * p.si + j) = v;
      }
      return;
    }
#pragma unroll 1
    for (int t = 0; t < kGM * BN / kGT; ++t) {
      const int e = tid + t * kGT;
      int m, j;
      if (p.si == 1) { j = e / kGM; m = e - j * kGM; } else { m = e / BN; j = e - m * BN; }
      float v = red[m * BN + j];
#pragma unroll
      for (int w = 1; w < kGW; ++w) v += red[(w * kGM + m) * BN + j];
      if (m0 + m < p.M && j < p.n) Y[(int64_t)j * p.sj + (int64_t)(m0 + m) * p.si] = v;
    }
  }
};

template <bool CL, bool WIDE, typename TX, bool KM, bool VEC>
__device__ __forceinline__ void gemm_dispatch(const GemmArg& p, int cta, int nst, float* smem) {
  if (p.n <= 8) GemmTile<TX, KM, VEC, 8>::template run<CL, WIDE>(p, cta, nst, smem);
  else if (p.n <= 16) GemmTile<TX, KM, VEC, 16>::template run<CL, WIDE>(p, cta, nst, smem);
  else if (p.n <= 32) GemmTile<TX, KM, VEC, 32>::template run<CL, WIDE>(p, cta, nst, smem);
  else GemmTile<TX, KM, VEC, 64>::template run<CL, WIDE>(p, cta, nst, smem);
}

int bn_of(int n) { return n <= 8 ? 8 : (n <= 16 ? 16 : (n <= 32 ? 32 : 64)); }

}  // namespace

// CL: a launch in clusters (kept apart: with the shares' code in one kernel every other launch was 1 to 2 % slower)
template <typename TX, bool CL>
__global__ void __launch_bounds__(kGT, 2) k_gemm_group(const __grid_constant__ GemmArgs g) {
  extern __shared__ __align__(16) float gemm_smem[];
  int q = 0;
  while (q + 1 < g.np && (int)blockIdx.x >= g.p[q + 1].first) ++q;
  const GemmArg& p = g.p[q];
  const int cta = (int)blockIdx.x - p.first;
  pdl_wait();
  if (CL && cta >= p.n_cta) return;                          // padding of the last cluster of a product without shared tiles
  if (blockIdx.x == 0 && g.clear) g.clear[threadIdx.x] = 0;   // status block of the workspace (256 ints)
  if (p.km) {
    if (p.vec) gemm_dispatch<CL, false, TX, true, true>(p, cta, g.nst, gemm_smem);
    else gemm_dispatch<CL, false, TX, true, false>(p, cta, g.nst, gemm_smem);
  } else {
    if (p.vec) gemm_dispatch<CL, false, TX, false, true>(p, cta, g.nst, gemm_smem);
    else gemm_dispatch<CL, false, TX, false, false>(p, cta, g.nst, gemm_smem);
  }
}

// One product whose sizes 32 bits do not count (a batch mode has C H W columns): every CTA rebases the product to its own
// tile and span in 64 bits and runs it as a narrow one.  Kept apart from k_gemm_group, which it would cost 2 to 3 % (the
// cold start of a 64 x 128 x 28 x 28 layer takes 79.0 us, with 64-bit spans in the one kernel it took 80.5).
template <typename TX>
__global__ void __launch_bounds__(kGT, 2) k_gemm_wide(const __grid_constant__ GemmProb p, const int64_t first, const int nst,
                                                      int* const clear) {
  extern __shared__ __align__(16) float gemm_smem[];
  __shared__ GemmArg w;
  pdl_wait();
  if (blockIdx.x == 0 && clear) clear[threadIdx.x] = 0;
  if (threadIdx.x == 0) w = gemm_tile_arg(p, first + blockIdx.x, (int)sizeof(TX));
  __syncthreads();
  if (p.km) {
    if (p.vec) gemm_dispatch<false, true, TX, true, true>(w, 0, nst, gemm_smem);
    else gemm_dispatch<false, true, TX, true, false>(w, 0, nst, gemm_smem);
  } else {
    if (p.vec) gemm_dispatch<false, true, TX, false, true>(w, 0, nst, gemm_smem);
    else gemm_dispatch<false, true, TX, false, false>(w, 0, nst, gemm_smem);
  }
}

// CTAs the projection of a mode launches, and column splits of an expansion: enough for two CTAs per SM, at least
// two chunks of 128 each, so that a partial of P is worth its reduction
int gemm_expand_splits(int64_t a, int64_t Q) {
  const int64_t tiles = (a + kGM - 1) / kGM;
  int64_t ns = std::max<int64_t>(1, 296 / tiles);
  ns = std::min<int64_t>(ns, std::max<int64_t>(1, Q / (2 * kGK)));
  return (int)std::max<int64_t>(std::min<int64_t>(ns, 296), (Q + kGemmMaxSpan - 129) / (kGemmMaxSpan - 128));
}

GemmProb gemm_project(const void* X, const float* B, float* Y, int64_t O, int64_t a, int64_t I, int n, int64_t so, int64_t sj,
                      int64_t si, bool bf16) {
  GemmProb p;
  std::memset(&p, 0, sizeof(p));
  p.X = X; p.B = B; p.Y = Y; p.n = n; p.ldb = n;
  p.km = I == 1;
  p.nsplit = 1;
  p.K = p.kps = p.kin = a;
  p.sj = sj;
  if (I == 1) {
    p.M = O; p.O = 1; p.ld = a; p.si = so;
  } else {
    p.M = I; p.O = O; p.ld = I; p.sxo = a * I; p.so = so; p.si = si;
  }
  const int64_t al = I == 1 ? a : I;
  p.vec = al % 4 == 0 && (reinterpret_cast<uintptr_t>(X) & (bf16 ? 7u : 15u)) == 0;
  p.bvec = n % 4 == 0 && (reinterpret_cast<uintptr_t>(B) & 15u) == 0;
  p.yvec = p.sj == 1 && n % 4 == 0 && p.si % 4 == 0 && p.so % 4 == 0 && p.ysplit % 4 == 0 &&
           (reinterpret_cast<uintptr_t>(p.Y) & 15u) == 0;
  return p;
}

GemmProb gemm_expand(const void* X, const float* V, float* Pp, int64_t O, int64_t a, int64_t I, int n, int nsplit, int64_t kps,
                     bool bf16) {
  GemmProb p;
  std::memset(&p, 0, sizeof(p));
  p.X = X; p.B = V; p.Y = Pp; p.n = n; p.ldb = n;
  p.km = I != 1;
  p.M = a; p.O = 1; p.K = O * I;
  p.nsplit = nsplit; p.kps = kps;
  p.ysplit = a * n; p.si = n; p.sj = 1;
  if (I == 1) { p.ld = a; p.kin = p.K; }
  else { p.ld = I; p.kin = I; p.sxo = a * I; }
  const int64_t al = I == 1 ? a : I;
  p.vec = al % 4 == 0 && (reinterpret_cast<uintptr_t>(X) & (bf16 ? 7u : 15u)) == 0;
  p.bvec = n % 4 == 0 && (reinterpret_cast<uintptr_t>(V) & 15u) == 0;
  p.yvec = p.sj == 1 && n % 4 == 0 && p.si % 4 == 0 && p.so % 4 == 0 && p.ysplit % 4 == 0 &&
           (reinterpret_cast<uintptr_t>(p.Y) & 15u) == 0;
  return p;
}

// adds a product; more than 64 columns go as several products over the same X
void gemm_add(GemmGroup* g, const GemmProb& p) {
  for (int j = 0; j < p.n; j += 64) {
    GemmProb q = p;
    q.n = std::min(64, p.n - j);
    q.B = p.B + j;
    q.Y = p.Y + (int64_t)j * p.sj;
    g->p[g->np++] = q;
  }
}

// 32 bits count every index of the product, up to the end of the last chunk of the last split
bool gemm_narrow(const GemmProb& p) {
  constexpr int64_t most = (1ll << 31) - 2 * kGM * kGK;
  return p.M < most && p.K < most && p.kps < most && p.K + p.kps < most &&
         (p.M + kGM - 1) / kGM * p.O < (1ll << 26) / p.nsplit;    // eight products, eight CTAs a tile
}

// a tile and a split of a wide product (t counts the row tiles, then the outer indices, then the splits) as a product of
// its own
__host__ __device__ GemmArg gemm_tile_arg(const GemmProb& p, int64_t t, int xbytes) {
  const int64_t tiles_m = (p.M + kGM - 1) / kGM, m0 = t % tiles_m * kGM, o = t / tiles_m % p.O, split = t / tiles_m / p.O;
  const int64_t k = split * p.kps, left = p.K - k, len = left < 0 ? 0 : (left < p.kps ? left : p.kps);
  GemmArg w;
  int64_t x = m0 * (p.km ? p.ld : 1) + o * p.sxo + (p.km ? k : k * p.ld);
  w.k0 = 0;
  w.sxo = p.sxo; w.ld = p.ld; w.ysplit = 0; w.so = 0; w.sj = p.sj; w.si = p.si;
  w.kin = (int)len;                                  // one slab, unless the span reaches into a second one
  if (p.km && p.kin < p.K && len > 0) {
    const int64_t slab = k / p.kin, in = k - slab * p.kin;
    x = m0 * p.ld + slab * p.sxo + in;
    if (p.kin < kGemmMaxSpan) {                      // k counted from the start of the slab
      w.k0 = (int)in;
      w.kin = (int)p.kin;
    } else if (p.kin - in < len) {                   // slabs longer than a span: the one end it holds comes to lie at 2^29
      w.k0 = (int)(kGemmMaxSpan - (p.kin - in));
      w.kin = (int)kGemmMaxSpan;
      w.sxo = p.sxo - p.kin + kGemmMaxSpan;
    }
    x -= w.k0;
  }
  w.X = static_cast<const char*>(p.X) + (len > 0 ? x * xbytes : 0);
  w.B = p.B + (len > 0 ? (k - w.k0) * p.ldb : 0);
  w.Y = p.Y + split * p.ysplit + o * p.so + m0 * p.si;
  w.ldb = p.ldb;
  w.M = (int)(p.M - m0 < kGM ? p.M - m0 : kGM);
  w.K = w.k0 + (int)len;
  w.O = w.nsplit = w.tiles_m = w.ksp = w.n_cta = 1;
  w.n = p.n;
  w.kps = w.K;
  w.first = 0;
  w.km = p.km; w.vec = p.vec; w.bvec = p.bvec; w.yvec = p.yvec;
  return w;
}

static cudaError_t launch_narrow(GemmArgs& g, bool bf16, cudaStream_t st) {
  // the longest contractions first: their CTAs would otherwise start last and run alone
  std::sort(g.p, g.p + g.np, [](const GemmArg& a, const GemmArg& b) {
    return (int64_t)std::min(a.K, a.kps) * bn_of(a.n) > (int64_t)std::min(b.K, b.kps) * bn_of(b.n);
  });
  // a product of few tiles and a long contraction shares each tile between the CTAs of a cluster, as far as an
  // SM still gets one CTA: 128 x 1280 by 16 columns on 4 CTAs took 12.9 us, ten chunks in turn, and takes 5.9 on 32 (99
  // tiles of six chunks: 12.8 us as they are, 15.0 in pairs).  Up to three chunks the barriers cost what the split saves
  int cs = 1;
  for (int q = 0; q < g.np; ++q) {
    const int64_t tiles = (int64_t)g.p[q].tiles_m * g.p[q].O * g.p[q].nsplit;
    const int chunks = (std::min(g.p[q].K, g.p[q].kps) + kGK - 1) / kGK;
    while (cs < 8 && tiles * 2 * cs <= 148 && chunks >= 4 && 2 * cs <= chunks) cs *= 2;
  }
  int first = 0, bn = 8;
  for (int q = 0; q < g.np; ++q) {
    GemmArg& p = g.p[q];
    const int64_t tiles = (int64_t)p.tiles_m * p.O * p.nsplit;
    const int chunks = (std::min(p.K, p.kps) + kGK - 1) / kGK;
    p.ksp = (cs > 1 && tiles * cs <= 148 && chunks >= 4 && cs <= chunks) ? cs : 1;
    p.first = first;
    p.n_cta = (int)tiles * p.ksp;
    first += (p.n_cta + cs - 1) / cs * cs;
    bn = std::max(bn, bn_of(p.n));
  }
  g.nst = bn == 64 ? 2 : 3;
  const size_t stage = (size_t)(kGM * kPK + kGK * bn) * 4;
  const size_t smem = std::max<size_t>(stage * g.nst, (size_t)kGW * kGM * bn * 4);
  auto kernel = cs > 1 ? (bf16 ? k_gemm_group<__nv_bfloat16, true> : k_gemm_group<float, true>)
                       : (bf16 ? k_gemm_group<__nv_bfloat16, false> : k_gemm_group<float, false>);
  cudaError_t e = opt_in_smem(reinterpret_cast<const void*>(kernel), smem);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)first);
  cfg.blockDim = dim3(kGT);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[2];
  int na = 0;
  if (cs > 1) {
    at[na].id = cudaLaunchAttributeClusterDimension;
    at[na].val.clusterDim.x = (unsigned)cs;
    at[na].val.clusterDim.y = 1;
    at[na].val.clusterDim.z = 1;
    ++na;
  }
  at[na].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[na].val.programmaticStreamSerializationAllowed = 1;
  ++na;
  cfg.attrs = at;
  cfg.numAttrs = na;
  return cudaLaunchKernelEx(&cfg, kernel, g);
}

template <typename TX>
static cudaError_t launch_wide(const GemmProb& p, int* clear, cudaStream_t st) {
  if (p.kps > (p.nsplit > 1 || p.kin < p.K ? kGemmMaxSpan : INT32_MAX - kGK)) return cudaErrorInvalidValue;
  const int64_t ctas = (p.M + kGM - 1) / kGM * p.O * p.nsplit;
  const int bn = bn_of(p.n), nst = bn == 64 ? 2 : 3;
  const size_t stage = (size_t)(kGM * kPK + kGK * bn) * 4;
  const size_t smem = std::max<size_t>(stage * nst, (size_t)kGW * kGM * bn * 4);
  cudaError_t e = opt_in_smem(reinterpret_cast<const void*>(k_gemm_wide<TX>), smem);
  for (int64_t t = 0; t < ctas && e == cudaSuccess; t += kGemmMaxGrid) {       // more tiles than a grid holds: in parts
    e = launch_pdl(k_gemm_wide<TX>, dim3((unsigned)std::min(ctas - t, kGemmMaxGrid)), dim3(kGT), smem, st, p, t, nst,
                         clear);
    clear = nullptr;
  }
  return e;
}

cudaError_t launch_gemm_group(const GemmGroup& group, bool bf16, cudaStream_t st) {
  GemmArgs g;
  g.np = 0;
  g.clear = group.clear;
  double bytes = 0.0;
  for (int q = 0; q < group.np; ++q) {
    const GemmProb& p = group.p[q];
    bytes += (double)p.M * p.O * p.K * (bf16 ? 2 : 4);
    if (!gemm_narrow(p)) continue;
    GemmArg& a = g.p[g.np++];
    a.X = p.X; a.B = p.B; a.Y = p.Y;
    a.sxo = p.sxo; a.ld = p.ld; a.ysplit = p.ysplit; a.so = p.so; a.sj = p.sj; a.si = p.si;
    a.ldb = p.ldb; a.kin = (int)p.kin;
    a.M = (int)p.M; a.K = (int)p.K; a.O = (int)p.O; a.n = p.n;
    a.nsplit = p.nsplit; a.kps = (int)p.kps;
    a.tiles_m = (a.M + kGM - 1) / kGM;
    a.k0 = 0;
    a.km = p.km; a.vec = p.vec; a.bvec = p.bvec; a.yvec = p.yvec;
  }
  ProfScope prof(ASI_K_MODEPROD, st, bytes);
  const bool any = g.np > 0;
  if (any) {
    const cudaError_t e = launch_narrow(g, bf16, st);
    if (e != cudaSuccess) return e;
  }
  int* clear = any ? nullptr : group.clear;          // the first launch clears
  for (int q = 0; q < group.np; ++q) {
    const GemmProb& p = group.p[q];
    if (gemm_narrow(p)) continue;
    const cudaError_t e = bf16 ? launch_wide<__nv_bfloat16>(p, clear, st) : launch_wide<float>(p, clear, st);
    if (e != cudaSuccess) return e;
    clear = nullptr;
  }
  return cudaSuccess;
}

}  // namespace asi
