// Small dense kernels of the token (linear-layer) path.
//
//   k_core_tok  : the core products after the first one (T = A x_3 U_3^T) in one launch.
//   k_lin_mid   : the middle of the linear backward (Sec. 3.1 footnote, derived steps L1-L2): the batch-mode
//                 contraction of dY x_2 U_2^T and Z4[o][k] = sum_{l1,l2} Z(l1, l2, o) core[l1][l2][k].
//   k_lin_tail  : dW[o][d] = sum_k Z4[o][k] U[d][k] in 64 x 128 tiles, 8 x 4 per thread, written once, coalesced.
#include <cuda_bf16.h>

#include <algorithm>

#include "asi_internal.h"

namespace asi {

namespace {
constexpr int kLtO = 64, kLtD = 128;
}  // namespace

// ---------------------------------------------------------------------------------------------
// k_core_tok: core[i][j][l] = sum_b sum_n U1[b][i] U2[n][j] T[b][n][l] for T = A x_3 U_3^T of a token layer
// ([B][N][r3]; U1 == null: B = 1 with coefficient one, the two-mode layer).  CTA (l-block of 4, i) takes every n:
// thread n forms W[n][l..l+3] = sum_b U1[b][i] T[b][n][l..] with 16 loads of T in flight, 256 values of n at a time;
// thread (j, l, n-group) then adds U2[n][j] W[n][l], the groups meet in order.  T is small (a few hundred KB, in L2)
// and read r1 times; what counts is the number of round trips, so no partial leaves the CTA and every load of a
// chunk -- T, U1, U2 -- is issued before the first is used (8 x 32 x 64 core from 32 x 197 tokens: 17 -> 6 us).
// ---------------------------------------------------------------------------------------------
__device__ __forceinline__ void cp_async4(float* dst, const float* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(static_cast<uint32_t>(__cvta_generic_to_shared(dst))), "l"(src)
               : "memory");
}
__device__ __forceinline__ void cp_async16(float* dst, const float* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(static_cast<uint32_t>(__cvta_generic_to_shared(dst))), "l"(src)
               : "memory");
}
__device__ __forceinline__ void cp_async_all() {
  asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 0;" ::: "memory");
}
// n contiguous floats to shared memory, 16 bytes at a time where both sides allow it
__device__ __forceinline__ void stage_flat(float* dst, const float* src, int n) {
  if ((reinterpret_cast<uintptr_t>(src) & 15u) == 0) {
    const int n4 = n >> 2;
    for (int e = threadIdx.x; e < n4; e += blockDim.x) cp_async16(dst + 4 * e, src + 4 * e);
    for (int e = 4 * n4 + threadIdx.x; e < n; e += blockDim.x) cp_async4(dst + e, src + e);
  } else {
    for (int e = threadIdx.x; e < n; e += blockDim.x) cp_async4(dst + e, src + e);
  }
}

constexpr int kU1Max = 1024;             // batch sizes whose column(s) of U1 fit shared memory beside the rest
constexpr int kCtL = 4, kCtN = 256, kCtB = 16;
template <bool VEC>
__global__ void __launch_bounds__(256) k_core_tok(const __grid_constant__ CoreTokArgs p) {
  extern __shared__ __align__(16) float ct_smem[];
  float* Ws = ct_smem;                                // [kCtN][4]
  float* U2s = Ws + kCtN * kCtL;                      // [kCtN][r2]
  float* red = U2s + kCtN * p.r2;                     // [256]
  float* U1s = red + 256;                             // [B]: column i
  const int tid = threadIdx.x, r2 = p.r2, r3 = p.r3;
  const int l0 = blockIdx.x * kCtL, i = blockIdx.y;
  const int n_out = r2 * kCtL;                        // (j, l), l fastest
  const int G = n_out <= 256 ? 256 / n_out : 1;
  const int oidx = tid % n_out, g = tid / n_out;
  float acc0 = 0.f, acc1 = 0.f;                       // outputs tid and tid + 256 (r2 <= 128)
  pdl_wait();
  const bool u1_staged = p.B <= kU1Max;
  for (int b = tid; b < p.B && u1_staged; b += 256) {
    if (p.U1) cp_async4(U1s + b, p.U1 + (int64_t)b * p.r1 + i);
    else U1s[b] = 1.f;
  }
  const int64_t sb = (int64_t)p.N * r3;
  for (int n0 = 0; n0 < p.N; n0 += kCtN) {
    const int nn = (p.N - n0 < kCtN) ? p.N - n0 : kCtN;
    stage_flat(U2s, p.U2 + (int64_t)n0 * r2, nn * r2);
    const int n = tid < nn ? tid : nn - 1;
    const float* src = p.T + (int64_t)(n0 + n) * r3 + l0;
    float w[4] = {0.f, 0.f, 0.f, 0.f};
    for (int b0 = 0; b0 < p.B; b0 += kCtB) {
      float x[kCtB][4];
#pragma unroll
      for (int q = 0; q < kCtB; ++q) {
        const float* s = src + (b0 + q < p.B ? b0 + q : p.B - 1) * sb;
        if constexpr (VEC) {
          const float4 v = __ldg(reinterpret_cast<const float4*>(s));
          x[q][0] = v.x; x[q][1] = v.y; x[q][2] = v.z; x[q][3] = v.w;
        } else {
#pragma unroll
          for (int c = 0; c < 4; ++c) x[q][c] = __ldg(s + (l0 + c < r3 ? c : 0));
        }
      }
      if (b0 == 0) {
        cp_async_all();
        __syncthreads();                              // U1 and U2 of this chunk (all threads: the loop is uniform)
      }
#pragma unroll
      for (int q = 0; q < kCtB; ++q) {
        float u = 0.f;
        if (b0 + q < p.B) u = u1_staged ? U1s[b0 + q] : __ldg(p.U1 + (int64_t)(b0 + q) * p.r1 + i);   // B > 1 has a U1
#pragma unroll
        for (int c = 0; c < 4; ++c) w[c] = fmaf(u, x[q][c], w[c]);
      }
    }
    if (tid < nn) *reinterpret_cast<float4*>(Ws + tid * kCtL) = make_float4(w[0], w[1], w[2], w[3]);
    __syncthreads();
    const int l = oidx % kCtL, j = oidx / kCtL;
    if (n_out <= 256) {
      if (g < G) {
#pragma unroll 8
        for (int k = g; k < nn; k += G) acc0 = fmaf(Ws[k * kCtL + l], U2s[k * r2 + j], acc0);
      }
    } else {
#pragma unroll 4
      for (int k = 0; k < nn; ++k) {
        acc0 = fmaf(Ws[k * kCtL + l], U2s[k * r2 + j], acc0);
        if (tid + 256 < n_out) acc1 = fmaf(Ws[k * kCtL + l], U2s[k * r2 + j + 64], acc1);
      }
    }
    __syncthreads();
  }
  const int l = oidx % kCtL, j = oidx / kCtL;
  if (n_out <= 256) {
    if (g < G) red[g * n_out + oidx] = acc0;
    __syncthreads();
    if (tid < n_out) {
      float v = red[tid];
      for (int q = 1; q < G; ++q) v += red[q * n_out + tid];
      if (l0 + l < r3) p.core[((int64_t)i * r2 + j) * r3 + l0 + l] = v;
    }
  } else if (l0 + l < r3) {
    p.core[((int64_t)i * r2 + j) * r3 + l0 + l] = acc0;
    if (tid + 256 < n_out) p.core[((int64_t)i * r2 + j + 64) * r3 + l0 + l] = acc1;
  }
}

cudaError_t launch_core_tok(const CoreTokArgs& p, cudaStream_t st) {
  ProfScope prof(ASI_K_MODEPROD, st, 4.0 * ((double)p.B * p.N * p.r3 + (double)p.r1 * p.r2 * p.r3));
  const size_t smem = 4 * ((size_t)kCtN * kCtL + (size_t)kCtN * p.r2 + 256 + kU1Max);
  const bool vec = p.r3 % 4 == 0 && (reinterpret_cast<uintptr_t>(p.T) & 15u) == 0;
  auto kernel = vec ? k_core_tok<true> : k_core_tok<false>;
  cudaError_t e = opt_in_smem(reinterpret_cast<const void*>(kernel), smem);
  if (e != cudaSuccess) return e;
  return launch_pdl(kernel, dim3((unsigned)((p.r3 + kCtL - 1) / kCtL), (unsigned)p.r1), dim3(256), smem, st, p);
}

// ---------------------------------------------------------------------------------------------
// k_lin_mid: Z4[o][k] = sum_{i,j} (sum_b U1[b][i] Y1[b][o][j]) core[i][j][k], the middle of the linear backward
// after Y1 = dY x_2 U_2^T ([B][Dout][r2]; U1 == null: the two-mode layer, B = 1 and i has one value).  CTA = 8
// output rows: phase 1 contracts the batch in registers (thread = four neighbouring (o, j) entries, a share of b; the
// shares meet in shared memory as Z[lead][o]), phase 2 contracts the leading indices (thread = one k, all 8 rows,
// a share of the leads: each value of the core feeds eight multiply-adds).  The leading index i goes in chunks whose
// block of the core fits 64 KB of shared memory; that block, U1 and the first eight rows of Y1 per thread travel
// together (8 x 32 x 64 core, 3072 rows: 53 -> 12 us against loads issued where they are used).
// ---------------------------------------------------------------------------------------------
constexpr int kLmO = 8, kLmI = 8, kLmCore = 16384;
__host__ __device__ inline int lin_mid_chunk(int r1, int r2, int r3) {
  int c = kLmCore / (r2 * r3);
  if (c > kLmI) c = kLmI;
  if (c > r1) c = r1;
  return c < 1 ? 1 : c;
}
template <int CW>
__global__ void __launch_bounds__(256, 2) k_lin_mid(const __grid_constant__ LinMidArgs p) {
  extern __shared__ __align__(16) float lm_smem[];
  const int tid = threadIdx.x, r2 = p.r2, r3 = p.r3;
  const int o0 = blockIdx.x * kLmO;
  const int ic = lin_mid_chunk(p.r1, r2, r3);
  const int n4 = kLmO * r2 / CW;                      // items of one sample: CW neighbouring entries of (o, j)
  const int BG = n4 <= 256 ? 256 / n4 : 1;
  const int n_red = (r3 <= 256 ? 256 / r3 : 1) * r3 * kLmO, n_part = BG * ic * r2 * kLmO;
  float* cs = lm_smem;                                // [ic r2][r3]
  float* Z = cs + (((size_t)ic * r2 * r3 + 3) & ~(size_t)3);   // [ic r2][8]
  float* part = Z + ic * r2 * kLmO;                   // [BG][ic][r2][8]; at the end the shares of Z4 [G][r3][8]
  float* U1s = part + (n_part > n_red ? n_part : n_red);       // [B][8]
  const int G = r3 <= 256 ? 256 / r3 : 1;
  const int k = tid % r3, kg = tid / r3;              // r3 <= 128
  float z4[kLmO];
#pragma unroll
  for (int q = 0; q < kLmO; ++q) z4[q] = 0.f;
  pdl_wait();
  for (int i0 = 0; i0 < p.r1; i0 += ic) {
    const int ni = (p.r1 - i0 < ic) ? p.r1 - i0 : ic;
    stage_flat(cs, p.core + (int64_t)i0 * r2 * r3, ni * r2 * r3);
    for (int e = tid; e < p.B * kLmI && p.B <= kU1Max; e += 256) {
      const int b = e / kLmI, i = e % kLmI;
      if (p.U1 && i < ni) cp_async4(U1s + e, p.U1 + (int64_t)b * p.r1 + i0 + i);
      else U1s[e] = (!p.U1 && i == 0) ? 1.f : 0.f;
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
    const int64_t sb = (int64_t)p.Dout * r2;
    const int avail = (p.Dout - o0 < kLmO ? p.Dout - o0 : kLmO) * r2;   // valid entries of a sample
    bool waited = false;
    for (int it = tid % n4, bg = tid / n4, pass = 0; pass < (n4 + 255) / 256; ++pass, it += 256) {
      float acc[kLmI][CW];
#pragma unroll
      for (int i = 0; i < kLmI; ++i)
#pragma unroll
        for (int q = 0; q < CW; ++q) acc[i][q] = 0.f;
      const bool on = bg < BG && it < n4 && it * CW < avail;
      const float* src = p.Y1 + (int64_t)o0 * r2 + (on ? it * CW : 0);
      for (int b0 = bg < BG ? bg : 0, first = 1; first || b0 < p.B; b0 += 8 * BG, first = 0) {
        float x[8][CW];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          const int b = b0 + u * BG < p.B ? b0 + u * BG : p.B - 1;
          if constexpr (CW == 4) {
            const float4 v = __ldg(reinterpret_cast<const float4*>(src + b * sb));
            x[u][0] = v.x; x[u][1] = v.y; x[u][2] = v.z; x[u][3] = v.w;
          } else {
            x[u][0] = __ldg(src + b * sb);
          }
        }
        if (!waited) {                                // uniform: every thread's first batch
          asm volatile("cp.async.wait_group 0;" ::: "memory");
          __syncthreads();
          waited = true;
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          const int b = b0 + u * BG;
          if (b < p.B) {
            float c[8];
            if (p.B <= kU1Max) {
              const float4 c0 = *reinterpret_cast<const float4*>(U1s + b * kLmI), c1 = *reinterpret_cast<const float4*>(U1s + b * kLmI + 4);
              c[0] = c0.x; c[1] = c0.y; c[2] = c0.z; c[3] = c0.w; c[4] = c1.x; c[5] = c1.y; c[6] = c1.z; c[7] = c1.w;
            } else {
#pragma unroll
              for (int i = 0; i < kLmI; ++i) c[i] = i < ni ? __ldg(p.U1 + (int64_t)b * p.r1 + i0 + i) : 0.f;
            }
#pragma unroll
            for (int i = 0; i < kLmI; ++i)
#pragma unroll
              for (int q = 0; q < CW; ++q) acc[i][q] = fmaf(c[i], x[u][q], acc[i][q]);
          }
        }
      }
      if (bg < BG && it < n4) {
        const int o = it * CW / r2, j = it * CW - o * r2;     // CW divides r2
#pragma unroll
        for (int i = 0; i < kLmI; ++i)
          if (i < ni)
#pragma unroll
            for (int q = 0; q < CW; ++q) part[((bg * ic + i) * r2 + j + q) * kLmO + o] = on ? acc[i][q] : 0.f;
      }
    }
    __syncthreads();
    const int nl = ni * r2;                           // leads of this chunk
    for (int e = tid; e < nl * kLmO; e += 256) {
      float v = part[e];
      for (int q = 1; q < BG; ++q) v += part[q * ic * r2 * kLmO + e];
      Z[e] = v;
    }
    __syncthreads();
    if (kg < G) {
#pragma unroll 4
      for (int l = kg; l < nl; l += G) {
        const float c = cs[l * r3 + k];
        const float4 a = *reinterpret_cast<const float4*>(Z + l * kLmO), b = *reinterpret_cast<const float4*>(Z + l * kLmO + 4);
        z4[0] = fmaf(c, a.x, z4[0]); z4[1] = fmaf(c, a.y, z4[1]);
        z4[2] = fmaf(c, a.z, z4[2]); z4[3] = fmaf(c, a.w, z4[3]);
        z4[4] = fmaf(c, b.x, z4[4]); z4[5] = fmaf(c, b.y, z4[5]);
        z4[6] = fmaf(c, b.z, z4[6]); z4[7] = fmaf(c, b.w, z4[7]);
      }
    }
    __syncthreads();
  }
  pdl_launch_dependents();
  float* red = part;
  if (kg < G) {
    *reinterpret_cast<float4*>(red + (kg * r3 + k) * kLmO) = make_float4(z4[0], z4[1], z4[2], z4[3]);
    *reinterpret_cast<float4*>(red + (kg * r3 + k) * kLmO + 4) = make_float4(z4[4], z4[5], z4[6], z4[7]);
  }
  __syncthreads();
  for (int e = tid; e < r3 * kLmO; e += 256) {        // e = (o, k), k fastest: coalesced rows of Z4
    const int o = e / r3, kk = e - o * r3;
    float v = red[kk * kLmO + o];
    for (int q = 1; q < G; ++q) v += red[(q * r3 + kk) * kLmO + o];
    if (o0 + o < p.Dout) p.Z4[(int64_t)(o0 + o) * r3 + kk] = v;
  }
}

cudaError_t launch_lin_mid(const LinMidArgs& p, cudaStream_t st) {
  ProfScope prof(ASI_K_MODEPROD, st, 4.0 * ((double)p.B * p.Dout * p.r2 + (double)p.Dout * p.r3));
  const bool vec = p.r2 % 4 == 0 && (reinterpret_cast<uintptr_t>(p.Y1) & 15u) == 0;
  const int n4 = kLmO * p.r2 / (vec ? 4 : 1), ic = lin_mid_chunk(p.r1, p.r2, p.r3);
  const int BG = n4 <= 256 ? 256 / n4 : 1, G = p.r3 <= 256 ? 256 / p.r3 : 1;
  const size_t n_part = (size_t)BG * ic * p.r2 * kLmO, n_red = (size_t)G * p.r3 * kLmO;
  const size_t smem = 4 * ((((size_t)ic * p.r2 * p.r3 + 3) & ~(size_t)3) + (size_t)ic * p.r2 * kLmO +
                           std::max(n_part, n_red) + (size_t)std::min(p.B, kU1Max) * kLmI);
  auto kernel = vec ? k_lin_mid<4> : k_lin_mid<1>;
  cudaError_t e = opt_in_smem(reinterpret_cast<const void*>(kernel), smem);
  if (e != cudaSuccess) return e;
  return launch_pdl(kernel, dim3((unsigned)((p.Dout + kLmO - 1) / kLmO)), dim3(256), smem, st, p);
}

// ---------------------------------------------------------------------------------------------
// k_lin_tail: dW[o][d] = sum_k Z4[o][k] U[d][k]: 64 x 128 tile per CTA, 8 x 4 per thread.
// Rows of Z4 and of U sit in shared memory with a pitch of 4 * (odd number) floats and zeros up to it, so the
// k loop reads four k at a time with 16-byte loads (the 8 Z4 rows of a warp are broadcasts; the 32 lanes' U
// rows fall in distinct banks): 12 loads per 64 packed multiply-adds (fma.rn.f32x2: the even and the odd k of a sum).  Both
// tiles travel by asynchronous copies, all at once (through registers they were six round trips):
// 197 x 32 tokens, 3072 x 768 weights, rank 64 29 -> 20 us beside another layer, 768 x 768 rank 32 7.9 -> 5.9.
// A short sum leaves little but the stores and wants CTAs: up to rank 12 plain multiply-adds, whose sums take half the
// registers, three CTAs an SM (whole weight gradient of 128 tokens, 4096 x 4096 weights: rank 3 30.8 -> 25.9 us, rank 8 34.3 -> 28.8, rank 12
// 37.4 -> 32.6; 67 MB of it take 10).
template <bool PACKED>
__global__ void __launch_bounds__(256, PACKED ? 2 : 3) k_lin_tail(const __grid_constant__ LinTailArgs p, int PR) {
  extern __shared__ __align__(16) float lt_smem[];
  const int r = p.r;
  float* Z4s = lt_smem;                              // [64][PR]
  float* Us = Z4s + kLtO * PR;                       // [128][PR]
  const int tid = threadIdx.x, lane = tid & 31;
  const int o0 = blockIdx.x * kLtO, d0 = blockIdx.y * kLtD;
  const int no = (p.Dout - o0 < kLtO) ? p.Dout - o0 : kLtO;
  const int nd = (p.Din - d0 < kLtD) ? p.Din - d0 : kLtD;
  pdl_wait();
  // entries of a row in turn: [rows][per] with per = r / 4 units or r values, zeros behind them
  auto stage = [&](float* dst, const float* src, int valid) {
    if (r % 4 == 0 && p.vec) {
      const int per = r / 4;
      for (int e = tid; e < valid * per; e += 256) {
        const int row = e / per, v = e - row * per;
        cp_async16(dst + row * PR + 4 * v, src + (int64_t)row * r + 4 * v);
      }
    } else {
      for (int e = tid; e < valid * r; e += 256) {
        const int row = e / r, v = e - row * r;
        cp_async4(dst + row * PR + v, src + (int64_t)row * r + v);
      }
    }
    const int pad = (r + 3) / 4 * 4 - r;             // what the loop reads beyond the row; sums of rows >= valid are not stored
    for (int e = tid; e < valid * pad; e += 256) {
      const int row = e / pad;
      dst[row * PR + r + e - row * pad] = 0.f;
    }
  };
  stage(Us, p.U + (int64_t)d0 * r, nd);
  stage(Z4s, p.Z4 + (int64_t)o0 * r, no);
  cp_async_all();
  __syncthreads();
  // dW[o0 + o][d0 + d] for o = 8 to .. 8 to + 7, d = lane + 32 i
  const int to = tid >> 5;
  float out[8][4];
  const float* zrow = Z4s + 8 * to * PR;
  const float* urow = Us + lane * PR;
  if constexpr (PACKED) {
    unsigned long long acc[8][4];
#pragma unroll
    for (int x = 0; x < 8; ++x)
#pragma unroll
      for (int y = 0; y < 4; ++y) acc[x][y] = 0ull;
    for (int k = 0; k < r; k += 4) {
      ulonglong2 uu[4];
#pragma unroll
      for (int y = 0; y < 4; ++y) uu[y] = *reinterpret_cast<const ulonglong2*>(urow + 32 * y * PR + k);
#pragma unroll
      for (int x = 0; x < 8; ++x) {
        const ulonglong2 zz = *reinterpret_cast<const ulonglong2*>(zrow + x * PR + k);
#pragma unroll
        for (int y = 0; y < 4; ++y) {
          asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc[x][y]) : "l"(zz.x), "l"(uu[y].x));
          asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc[x][y]) : "l"(zz.y), "l"(uu[y].y));
        }
      }
    }
#pragma unroll
    for (int x = 0; x < 8; ++x)
#pragma unroll
      for (int y = 0; y < 4; ++y) {
        float lo, hi;
        asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(acc[x][y]));
        out[x][y] = lo + hi;
      }
  } else {
#pragma unroll
    for (int x = 0; x < 8; ++x)
#pragma unroll
      for (int y = 0; y < 4; ++y) out[x][y] = 0.f;
    for (int k = 0; k < r; k += 4) {
      float4 uu[4];
#pragma unroll
      for (int y = 0; y < 4; ++y) uu[y] = *reinterpret_cast<const float4*>(urow + 32 * y * PR + k);
#pragma unroll
      for (int x = 0; x < 8; ++x) {
        const float4 zz = *reinterpret_cast<const float4*>(zrow + x * PR + k);
#pragma unroll
        for (int y = 0; y < 4; ++y)
          out[x][y] = fmaf(zz.w, uu[y].w, fmaf(zz.z, uu[y].z, fmaf(zz.y, uu[y].y, fmaf(zz.x, uu[y].x, out[x][y]))));
      }
    }
  }
#pragma unroll
  for (int x = 0; x < 8; ++x) {
    const int o = o0 + 8 * to + x;
    if (o >= p.Dout) continue;
#pragma unroll
    for (int y = 0; y < 4; ++y) {
      const int d = d0 + lane + 32 * y;
      if (d < p.Din) p.dW[(int64_t)o * p.Din + d] = out[x][y];
    }
  }
}

cudaError_t launch_lin_tail(const LinTailArgs& p0, cudaStream_t st) {
  LinTailArgs p = p0;
  p.vec = ((reinterpret_cast<uintptr_t>(p.U) | reinterpret_cast<uintptr_t>(p.Z4)) & 15u) == 0;
  int PR = (p.r + 3) / 4 * 4;                     // pitch: 4 * (odd number) floats
  if ((PR / 4) % 2 == 0) PR += 4;
  ProfScope prof(ASI_K_MODEPROD, st, 4.0 * ((double)p.Dout * p.Din + (double)p.Dout * p.r));
  const size_t smem = 4 * (size_t)(kLtO + kLtD) * PR;
  dim3 grid((unsigned)((p.Dout + kLtO - 1) / kLtO), (unsigned)((p.Din + kLtD - 1) / kLtD));
  const auto kernel = p.r > 12 ? k_lin_tail<true> : k_lin_tail<false>;
  cudaError_t e = opt_in_smem(reinterpret_cast<const void*>(kernel), smem);
  if (e != cudaSuccess) return e;
  return launch_pdl(kernel, grid, dim3(256), smem, st, p, PR);
}

}  // namespace asi
