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
// ([B][N][r3]; U1 == null: B = 1 with coefficient one, the two-mode layer).  CTA (l-block of 8, i) takes every n:
// W[n][l] = sum_b U1[b][i] T[b][n][l] goes to shared memory a chunk of n at a time, thread (j, l, n-group) adds
// U2[n][j] W[n][l], the groups meet in order.  T is small (a few hundred KB, in L2) and read r1 times; what counts
// is the length of the chain of loads, so every thread has eight of them in flight and no partial leaves the CTA.
// ---------------------------------------------------------------------------------------------
constexpr int kCtL = 8, kCtN = 256;
template <bool VEC>
__global__ void __launch_bounds__(256) k_core_tok(const __grid_constant__ CoreTokArgs p) {
  extern __shared__ __align__(16) float ct_smem[];
  pdl_launch_dependents();
  float* Ws = ct_smem;                                // [kCtN][8]
  float* U2s = Ws + kCtN * kCtL;                      // [kCtN][r2]
  float* red = U2s + kCtN * p.r2;                     // [256][2]
  const int tid = threadIdx.x, r2 = p.r2, r3 = p.r3;
  const int l0 = blockIdx.x * kCtL, i = blockIdx.y;
  const int n_out = r2 * kCtL;                        // (j, l), l fastest
  const int G = n_out <= 256 ? 256 / n_out : 1;
  const int oidx = n_out <= 256 ? tid % n_out : tid, g = n_out <= 256 ? tid / n_out : 0;
  constexpr int kPer = 4;                             // outputs of a thread when n_out > 256 (r2 <= 128)
  float acc[kPer] = {0.f, 0.f, 0.f, 0.f};
  pdl_wait();
  for (int n0 = 0; n0 < p.N; n0 += kCtN) {
    const int nn = (p.N - n0 < kCtN) ? p.N - n0 : kCtN;
    for (int e = tid; e < nn * r2; e += 256) U2s[e] = __ldg(p.U2 + (int64_t)n0 * r2 + e);
    constexpr int CW = VEC ? 4 : 1, PER = kCtL / CW;  // columns per item
    for (int e = tid; e < nn * PER; e += 256) {
      const int n = e / PER, c = (e - n * PER) * CW;
      float w[CW];
#pragma unroll
      for (int q = 0; q < CW; ++q) w[q] = 0.f;
      if (l0 + c < r3) {
        const float* src = p.T + (int64_t)(n0 + n) * r3 + l0 + c;
        const int64_t sb = (int64_t)p.N * r3;
        for (int b0 = 0; b0 < p.B; b0 += 8) {
          float u[8];
          float4 x4[8];
          float x1[8];
#pragma unroll
          for (int q = 0; q < 8; ++q) {
            const int b = b0 + q < p.B ? b0 + q : p.B - 1;
            u[q] = (b0 + q < p.B) ? (p.U1 ? __ldg(p.U1 + (int64_t)b * p.r1 + i) : 1.f) : 0.f;
            if constexpr (VEC) x4[q] = __ldg(reinterpret_cast<const float4*>(src + b * sb));
            else x1[q] = __ldg(src + b * sb);
          }
#pragma unroll
          for (int q = 0; q < 8; ++q) {
            if constexpr (VEC) {
              w[0] = fmaf(u[q], x4[q].x, w[0]); w[1] = fmaf(u[q], x4[q].y, w[1]);
              w[2] = fmaf(u[q], x4[q].z, w[2]); w[3] = fmaf(u[q], x4[q].w, w[3]);
            } else {
              w[0] = fmaf(u[q], x1[q], w[0]);
            }
          }
        }
      }
#pragma unroll
      for (int q = 0; q < CW; ++q) Ws[n * kCtL + c + q] = w[q];
    }
    __syncthreads();
    if (n_out <= 256) {
      if (g < G) {
        const int l = oidx % kCtL, j = oidx / kCtL;
#pragma unroll 4
        for (int n = g; n < nn; n += G) acc[0] = fmaf(Ws[n * kCtL + l], U2s[n * r2 + j], acc[0]);
      }
    } else {
#pragma unroll
      for (int t = 0; t < kPer; ++t) {
        const int o = tid + t * 256, l = o % kCtL, j = o / kCtL;
        if (o < n_out)
          for (int n = 0; n < nn; ++n) acc[t] = fmaf(Ws[n * kCtL + l], U2s[n * r2 + j], acc[t]);
      }
    }
    __syncthreads();
  }
  if (n_out <= 256) {
    if (g < G) red[g * n_out + oidx] = acc[0];
    __syncthreads();
    if (tid < n_out) {
      float v = red[tid];
      for (int q = 1; q < G; ++q) v += red[q * n_out + tid];
      const int l = tid % kCtL, j = tid / kCtL;
      if (l0 + l < r3) p.core[((int64_t)i * r2 + j) * r3 + l0 + l] = v;
    }
  } else {
#pragma unroll
    for (int t = 0; t < kPer; ++t) {
      const int o = tid + t * 256, l = o % kCtL, j = o / kCtL;
      if (o < n_out && l0 + l < r3) p.core[((int64_t)i * r2 + j) * r3 + l0 + l] = acc[t];
    }
  }
}

cudaError_t launch_core_tok(const CoreTokArgs& p, cudaStream_t st) {
  ProfScope prof(ASI_K_MODEPROD, st, 4.0 * ((double)p.B * p.N * p.r3 + (double)p.r1 * p.r2 * p.r3));
  const size_t smem = 4 * ((size_t)kCtN * kCtL + (size_t)kCtN * p.r2 + 256);
  const bool vec = p.r3 % 4 == 0 && (reinterpret_cast<uintptr_t>(p.T) & 15u) == 0;
  auto kernel = vec ? k_core_tok<true> : k_core_tok<false>;
  cudaError_t e = opt_in_smem(reinterpret_cast<const void*>(kernel), smem);
  if (e != cudaSuccess) return e;
  return launch_pdl(kernel, dim3((unsigned)((p.r3 + kCtL - 1) / kCtL), (unsigned)p.r1), dim3(256), smem, st, p);
}

// ---------------------------------------------------------------------------------------------
// k_lin_mid: Z4[o][k] = sum_{i,j} (sum_b U1[b][i] Y1[b][o][j]) core[i][j][k], the middle of the linear backward
// after Y1 = dY x_2 U_2^T ([B][Dout][r2]; U1 == null: the two-mode layer, B = 1 and i has one value).  CTA = 8
// output rows: phase 1 contracts the batch in registers (thread = one row's four neighbouring j, a share of b; the
// shares meet in shared memory as Z[lead][o]), phase 2 contracts the leading indices (thread = one k, all 8 rows,
// a share of the leads: each value of the core feeds eight multiply-adds).  i goes in chunks of 8.
// ---------------------------------------------------------------------------------------------
constexpr int kLmO = 8, kLmI = 8;
template <int CW>
__global__ void __launch_bounds__(256) k_lin_mid(const __grid_constant__ LinMidArgs p) {
  extern __shared__ __align__(16) float lm_smem[];
  pdl_launch_dependents();
  const int tid = threadIdx.x, r2 = p.r2, r3 = p.r3;
  const int o0 = blockIdx.x * kLmO;
  const int n4 = kLmO * r2 / CW;                      // (o, j-group) items
  const int BG = n4 <= 256 ? 256 / n4 : 1;
  float* part = lm_smem;                              // [BG][kLmI][r2][8]
  float* Z = part + (size_t)BG * kLmI * r2 * kLmO;    // [kLmI r2][8]
  float* red = Z + kLmI * r2 * kLmO;                  // [G][r3][8]
  const int G = r3 <= 256 ? 256 / r3 : 1;
  const int k = tid % r3, kg = tid / r3;              // r3 <= 128
  float z4[kLmO];
#pragma unroll
  for (int q = 0; q < kLmO; ++q) z4[q] = 0.f;
  pdl_wait();
  for (int i0 = 0; i0 < p.r1; i0 += kLmI) {
    const int ni = (p.r1 - i0 < kLmI) ? p.r1 - i0 : kLmI;
    for (int e = tid; e < n4 * BG; e += 256) {
      const int it = e % n4, bg = e / n4;
      const int o = it * CW / r2, j = it * CW - o * r2;
      float acc[kLmI][CW];
#pragma unroll
      for (int i = 0; i < kLmI; ++i)
#pragma unroll
        for (int q = 0; q < CW; ++q) acc[i][q] = 0.f;
      if (o0 + o < p.Dout) {
        const float* src = p.Y1 + (int64_t)(o0 + o) * r2 + j;
        const int64_t sb = (int64_t)p.Dout * r2;
        for (int b0 = bg; b0 < p.B; b0 += 4 * BG) {
          float x[4][CW];
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int b = b0 + u * BG < p.B ? b0 + u * BG : b0;
            if constexpr (CW == 4) {
              const float4 v = __ldg(reinterpret_cast<const float4*>(src + b * sb));
              x[u][0] = v.x; x[u][1] = v.y; x[u][2] = v.z; x[u][3] = v.w;
            } else {
              x[u][0] = __ldg(src + b * sb);
            }
          }
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int b = b0 + u * BG;
            if (b >= p.B) break;
#pragma unroll
            for (int i = 0; i < kLmI; ++i) {
              const float c = p.U1 ? (i < ni ? __ldg(p.U1 + (int64_t)b * p.r1 + i0 + i) : 0.f) : (i == 0 ? 1.f : 0.f);
#pragma unroll
              for (int q = 0; q < CW; ++q) acc[i][q] = fmaf(c, x[u][q], acc[i][q]);
            }
          }
        }
      }
#pragma unroll
      for (int i = 0; i < kLmI; ++i)
#pragma unroll
        for (int q = 0; q < CW; ++q) part[((bg * kLmI + i) * r2 + j + q) * kLmO + o] = acc[i][q];
    }
    __syncthreads();
    const int nl = ni * r2;                           // leads of this chunk
    for (int e = tid; e < nl * kLmO; e += 256) {
      float v = part[e];
      for (int q = 1; q < BG; ++q) v += part[q * kLmI * r2 * kLmO + e];
      Z[e] = v;
    }
    __syncthreads();
    if (kg < G) {
      const float* cr = p.core + (int64_t)i0 * r2 * r3 + k;
#pragma unroll 1
      for (int l0 = kg; l0 < nl; l0 += 8 * G) {
        float c[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) c[u] = __ldg(cr + (int64_t)(l0 + u * G < nl ? l0 + u * G : l0) * r3);
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          const int l = l0 + u * G;
          if (l >= nl) break;
          const float4 a = *reinterpret_cast<const float4*>(Z + l * kLmO), b = *reinterpret_cast<const float4*>(Z + l * kLmO + 4);
          z4[0] = fmaf(c[u], a.x, z4[0]); z4[1] = fmaf(c[u], a.y, z4[1]);
          z4[2] = fmaf(c[u], a.z, z4[2]); z4[3] = fmaf(c[u], a.w, z4[3]);
          z4[4] = fmaf(c[u], b.x, z4[4]); z4[5] = fmaf(c[u], b.y, z4[5]);
          z4[6] = fmaf(c[u], b.z, z4[6]); z4[7] = fmaf(c[u], b.w, z4[7]);
        }
      }
    }
    __syncthreads();
  }
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
  const int n4 = kLmO * p.r2 / (vec ? 4 : 1);
  const int BG = n4 <= 256 ? 256 / n4 : 1, G = p.r3 <= 256 ? 256 / p.r3 : 1;
  const size_t smem = 4 * ((size_t)(BG + 1) * kLmI * p.r2 * kLmO + (size_t)G * p.r3 * kLmO);
  auto kernel = vec ? k_lin_mid<4> : k_lin_mid<1>;
  cudaError_t e = opt_in_smem(reinterpret_cast<const void*>(kernel), smem);
  if (e != cudaSuccess) return e;
  return launch_pdl(kernel, dim3((unsigned)((p.Dout + kLmO - 1) / kLmO)), dim3(256), smem, st, p);
}

// ---------------------------------------------------------------------------------------------
// k_lin_tail: dW[o][d] = sum_k Z4[o][k] U[d][k]: 64 x 128 tile per CTA, 8 x 4 per thread.
// Rows of Z4 and of U sit in shared memory with a pitch of 4 * (odd number) floats and zeros up to it, so the
// k loop reads four k at a time with 16-byte loads (the 8 Z4 rows of a warp are broadcasts; the 32 lanes' U
// rows fall in distinct banks): 12 loads per 128 multiply-adds.
__global__ void __launch_bounds__(256) k_lin_tail(const __grid_constant__ LinTailArgs p, int PR) {
  extern __shared__ __align__(16) float lt_smem[];
  pdl_launch_dependents();
  const int r = p.r;
  float* Z4s = lt_smem;                              // [64][PR]
  float* Us = Z4s + kLtO * PR;                       // [128][PR]
  const int tid = threadIdx.x, lane = tid & 31;
  const int o0 = blockIdx.x * kLtO, d0 = blockIdx.y * kLtD;
  const int no = (p.Dout - o0 < kLtO) ? p.Dout - o0 : kLtO;
  const int nd = (p.Din - d0 < kLtD) ? p.Din - d0 : kLtD;
  pdl_wait();
  // rows of a few vectors each: the lane index splits into (row, vector) by shifts
  const bool vec = p.r % 4 == 0 && p.vec;
  const int per = vec ? PR / 4 : PR;
  int lg = 2;
  while ((1 << lg) < per) ++lg;
  const int v0 = tid & ((1 << lg) - 1), step = 256 >> lg;
  auto stage = [&](float* dst, const float* src, int rows, int valid) {
#pragma unroll 4
    for (int row = tid >> lg; row < rows; row += step)
      if (vec) {
        if (v0 < per) {
          const bool on = row < valid && 4 * v0 < r;
          const float4 x = __ldcg(reinterpret_cast<const float4*>(src + (on ? (int64_t)row * r + 4 * v0 : 0)));
          *reinterpret_cast<float4*>(dst + row * PR + 4 * v0) = on ? x : make_float4(0.f, 0.f, 0.f, 0.f);
        }
      } else if (v0 < per) {
        const bool on = row < valid && v0 < r;
        const float x = __ldcg(src + (on ? (int64_t)row * r + v0 : 0));
        dst[row * PR + v0] = on ? x : 0.f;
      }
  };
  stage(Us, p.U + (int64_t)d0 * r, kLtD, nd);
  stage(Z4s, p.Z4 + (int64_t)o0 * r, kLtO, no);
  __syncthreads();
  // dW[o0 + o][d0 + d] for o = 8 to .. 8 to + 7, d = lane + 32 i
  const int to = tid >> 5;
  float out[8][4];
#pragma unroll
  for (int x = 0; x < 8; ++x)
#pragma unroll
    for (int y = 0; y < 4; ++y) out[x][y] = 0.f;
  const float* zrow = Z4s + 8 * to * PR;
  const float* urow = Us + lane * PR;
  for (int k = 0; k < PR; k += 4) {
    float4 zz[8], uu[4];
#pragma unroll
    for (int x = 0; x < 8; ++x) zz[x] = *reinterpret_cast<const float4*>(zrow + x * PR + k);
#pragma unroll
    for (int y = 0; y < 4; ++y) uu[y] = *reinterpret_cast<const float4*>(urow + 32 * y * PR + k);
#pragma unroll
    for (int x = 0; x < 8; ++x)
#pragma unroll
      for (int y = 0; y < 4; ++y) {
        out[x][y] = fmaf(zz[x].x, uu[y].x, out[x][y]);
        out[x][y] = fmaf(zz[x].y, uu[y].y, out[x][y]);
        out[x][y] = fmaf(zz[x].z, uu[y].z, out[x][y]);
        out[x][y] = fmaf(zz[x].w, uu[y].w, out[x][y]);
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
  cudaError_t e = opt_in_smem(reinterpret_cast<const void*>(k_lin_tail), smem);
  if (e != cudaSuccess) return e;
  return launch_pdl(k_lin_tail, grid, dim3(256), smem, st, p, PR);
}

}  // namespace asi
