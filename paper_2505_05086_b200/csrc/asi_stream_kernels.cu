// Modes of at most 128 entries with ranks up to 8, streamed by warps that wait for nobody.
//
//   k_wfiber : both products of one mode with strided fibers, V = A_m^T U and P = A_m V (Algorithm 1), or the mode
//              product Y = X x_m U^T alone
//   k_wplane : both products of the two spatial modes of a conv activation, maps of at most 64 x 64, square or not
//
// Every warp owns a ring of two tiles in shared memory that it fills itself (cp.async) and empties itself, so there
// is no barrier of the CTA between the first tile and the last: a warp that waits for memory does not hold up the
// arithmetic of the others, and one CTA with as many warps as the SM's shared memory holds keeps 80 to 110 KB of
// loads in flight.  Rows of a tile are padded to an odd number of quads: four neighbouring values of a row by row
// owners, and pairs of neighbouring columns by column owners, are both read without bank conflicts, and the
// alignment of the tensor's rows does not matter to anything but the width of the copies.  All arithmetic is
// fma.rn.f32x2: column owners keep a pair of columns per register pair (factor rows duplicated in shared memory), row
// owners the even and the odd columns of their sums (factor rows transposed).
#include <cuda_bf16.h>

#include <algorithm>

#include "asi_internal.h"

namespace asi {

namespace {

typedef unsigned long long f2;
__device__ __forceinline__ f2 pack2(float lo, float hi) {
  f2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ float2 unpack2(f2 v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}
__device__ __forceinline__ void ffma2(f2& d, f2 a, f2 b) { asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(a), "l"(b)); }

// Two and four neighbouring values of a staged row as packed fp32
__device__ __forceinline__ f2 ld_pair(const float* s) { return *reinterpret_cast<const f2*>(s); }
__device__ __forceinline__ f2 ld_pair(const __nv_bfloat16* s) {
  const uint32_t v = *reinterpret_cast<const uint32_t*>(s);
  return pack2(__uint_as_float(v << 16), __uint_as_float(v & 0xffff0000u));
}
__device__ __forceinline__ void ld_quad(const float* s, f2& a, f2& b) {
  const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(s);
  a = v.x; b = v.y;
}
__device__ __forceinline__ void ld_quad(const __nv_bfloat16* s, f2& a, f2& b) {
  const uint2 v = *reinterpret_cast<const uint2*>(s);
  a = pack2(__uint_as_float(v.x << 16), __uint_as_float(v.x & 0xffff0000u));
  b = pack2(__uint_as_float(v.y << 16), __uint_as_float(v.y & 0xffff0000u));
}

__device__ __forceinline__ unsigned s_addr(const void* p) { return static_cast<unsigned>(__cvta_generic_to_shared(p)); }
// four values at an address aligned to four; on = false fills with zeros (the source is not read)
__device__ __forceinline__ void cp_quad(float* dst, const float* src, bool on) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(s_addr(dst)), "l"(src), "r"(on ? 16 : 0) : "memory");
}
__device__ __forceinline__ void cp_quad(__nv_bfloat16* dst, const __nv_bfloat16* src, bool on) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(s_addr(dst)), "l"(src), "r"(on ? 8 : 0) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_wait1() { asm volatile("cp.async.wait_group 1;" ::: "memory"); }
// one value: asynchronous for fp32; a two-byte element has no asynchronous copy and goes through a register
__device__ __forceinline__ void cp_one(float* dst, const float* src, bool on) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(s_addr(dst)), "l"(src), "r"(on ? 4 : 0) : "memory");
}

// a pair of columns against one factor row: v[c][j / 2] += (x_c, x_c) (u_j, u_{j+1}).  A uniform 16-byte read of shared
// memory costs two cycles whatever it holds, so the factor row is read once and the column values are doubled
template <int R>
__device__ __forceinline__ void fma_cols(f2 (&v)[2][R / 2], f2 x, const float* __restrict__ u) {
  const float2 xs = unpack2(x);
  const f2 x0 = pack2(xs.x, xs.x), x1 = pack2(xs.y, xs.y);
#pragma unroll
  for (int j = 0; j < R / 2; j += 2) {
    const ulonglong2 w = *reinterpret_cast<const ulonglong2*>(u + 2 * j);
    ffma2(v[0][j], x0, w.x);
    ffma2(v[1][j], x1, w.x);
    ffma2(v[0][j + 1], x0, w.y);
    ffma2(v[1][j + 1], x1, w.y);
  }
}
// the lanes that share a pair of columns: neighbours s, 2 s, .. below 32
template <int R>
__device__ __forceinline__ void sum_cols(f2 (&v)[2][R / 2], int from, int to) {
  for (int s = from; s < to; s *= 2)
#pragma unroll
    for (int c = 0; c < 2; ++c)
#pragma unroll
      for (int j = 0; j < R / 2; ++j) {
        const float2 w = unpack2(v[c][j]);
        v[c][j] = pack2(w.x + __shfl_xor_sync(0xffffffffu, w.x, s), w.y + __shfl_xor_sync(0xffffffffu, w.y, s));
      }
}
// column j of the pair
template <int R>
__device__ __forceinline__ float2 col_pair(const f2 (&v)[2][R / 2], int j) {
  const float2 a = unpack2(v[0][j >> 1]), b = unpack2(v[1][j >> 1]);
  return (j & 1) ? make_float2(a.y, b.y) : make_float2(a.x, b.x);
}

constexpr int kWMaxWarps = 16;
constexpr size_t kWSmemBudget = 224 * 1024;

// ---------------------------------------------------------------------------------------------
// k_wfiber.  Tile = all a rows of TC neighbouring columns of one slab X[o].  RK = rows per lane (32 RK >= a).
//   columns  lane (kq, cp) owns columns 2 cp, 2 cp + 1 and every KQ-th row: V pair[j] += X(k, pair) U[k][j]; the KQ
//            lanes of a pair meet by shuffles
//   rows     lane owns rows lane + 32 i: P[k][j] += sum_q X(k, q) V[q][j], in registers across the warp's tiles
// ---------------------------------------------------------------------------------------------
template <typename TX>
__host__ __device__ constexpr int wf_cols(int RK) {
  return 2048 * (sizeof(TX) == 2 ? 2 : 1) / (32 * RK) > 64 ? 64 : 2048 * (sizeof(TX) == 2 ? 2 : 1) / (32 * RK);
}

template <int R, int RK, bool VEC, typename TX>
__global__ void __launch_bounds__(32 * kWMaxWarps, 1) k_wfiber(const __grid_constant__ Fiber2Args p) {
  constexpr int TC = wf_cols<TX>(RK), PT = TC + 4, NP = TC / 2, KQ = 32 / NP, UP = 12;
  constexpr int KB = 8, KS = KQ == 4 ? 2 : KQ;       // rows per step of the column pass, between a lane's rows
  extern __shared__ __align__(16) unsigned char ws_smem[];
  if (!p.project_only || p.first) pass_begin(p.clear, p.first);   // a product alone: its successor starts when it ends (see k_fiber2)
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = blockDim.x >> 5;
  const int a = p.a, r = p.r, a8 = (a + 7) & ~7;
  float* Ud = reinterpret_cast<float*>(ws_smem);     // [a8][UP]: rows >= a and columns >= r zero; rows 1, 4 and 5 apart are bank-disjoint
  float* Vt = Ud + a8 * UP + warp * (R * TC);        // [R][TC]
  TX* T = reinterpret_cast<TX*>(Ud + a8 * UP + nw * (R * TC)) + (size_t)warp * (2 * a8 * PT);   // [2][a8][PT]
  if (p.project_only) pdl_wait();                    // its factor comes from the kernel before
  for (int e = tid; e < a8 * R; e += blockDim.x) {
    const int k = e / R, j = e % R;
    const float u = (k < a && j < r) ? p.U[(int64_t)k * p.ldu + j] : 0.f;
    Ud[k * UP + j] = u;
  }
  for (int e = lane; e < (a8 - a) * PT; e += 32) {   // rows a .. a8 - 1 of both tiles are never written again
    T[a * PT + e] = TX(0.f);
    T[(a8 + a) * PT + e] = TX(0.f);
  }
  __syncthreads();
  const TX* __restrict__ X = static_cast<const TX*>(p.X);
  const int nti = (int)((p.I + TC - 1) / TC);
  const int total = (int)p.n_tiles, stride = (int)gridDim.x * nw;
  const int d_o = stride / nti, d_i = stride - d_o * nti;
  int t_ld = warp * (int)gridDim.x + (int)blockIdx.x;
  int o_ld = t_ld / nti, i_ld = t_ld - o_ld * nti;
  const int64_t slab = (int64_t)a * p.I;
  auto stage = [&](TX* dst) {
    if (t_ld < total) {
      const int64_t i0 = (int64_t)i_ld * TC;
      const TX* src = X + o_ld * slab + i0;
      const int nv = p.I - i0 < TC ? (int)(p.I - i0) : TC;
      if constexpr (VEC) {
        constexpr int QR = TC / 4, NR = 32 / QR;     // quads per row, rows per instruction
        const int k0 = lane / QR, c = 4 * (lane % QR);
        const bool on = c < nv;
        const TX* s = src + k0 * p.I + (on ? c : 0);
        TX* d = dst + k0 * PT + c;
#pragma unroll 4
        for (int k = k0; k < a; k += NR) {
          cp_quad(d, s, on);
          s += NR * p.I;
          d += NR * PT;
        }
      } else {
        constexpr int NR = TC < 32 ? 32 / TC : 1, NC = TC > 32 ? TC / 32 : 1;
        const int k0 = TC < 32 ? lane / TC : 0, c = TC < 32 ? lane % TC : lane;
#pragma unroll
        for (int h = 0; h < NC; ++h) {
          const int cc = c + 32 * h;
          const bool on = cc < nv;
          const TX* s = src + k0 * p.I + (on ? cc : 0);
          TX* d = dst + k0 * PT + cc;
          if constexpr (sizeof(TX) == 4) {
#pragma unroll 8
            for (int k = k0; k < a; k += NR) {
              cp_one(d, s, on);
              s += NR * p.I;
              d += NR * PT;
            }
          } else {
#pragma unroll 1
            for (int k = k0; k < a; k += 16 * NR) {
              TX v[16];
#pragma unroll
              for (int u = 0; u < 16; ++u) v[u] = s[(k + u * NR < a ? u * NR : 0) * p.I];
#pragma unroll
              for (int u = 0; u < 16; ++u)
                if (k + u * NR < a) d[u * NR * PT] = on ? v[u] : TX(0.f);
              s += 16 * NR * p.I;
              d += 16 * NR * PT;
            }
          }
        }
      }
    }
    cp_commit();
    t_ld += stride;
    o_ld += d_o;
    i_ld += d_i;
    if (i_ld >= nti) { i_ld -= nti; ++o_ld; }
  };
  const int kq = lane / NP, cp = lane % NP;
  // rows of the pair's lanes: neighbours differ by four rows where four lanes share a pair (bank-disjoint reads)
  const int kfirst = KQ == 4 ? (kq & 1) * 4 + (kq >> 1) : kq;
  f2 acc[RK][R];
#pragma unroll
  for (int i = 0; i < RK; ++i)
#pragma unroll
    for (int j = 0; j < R; ++j) acc[i][j] = 0ull;
  int t = t_ld, o_c = o_ld, i_c = i_ld, buf = 0;
  stage(T);
  for (; t < total; t += stride) {
    const TX* Tc = T + buf * (a8 * PT);
    buf ^= 1;
    const int o_n = o_ld, i_n = i_ld;
    stage(T + buf * (a8 * PT));
    cp_wait1();
    __syncwarp();
    f2 v[2][R / 2];
#pragma unroll
    for (int j = 0; j < R / 2; ++j) v[0][j] = v[1][j] = 0ull;
    {
      const TX* xs = Tc + kfirst * PT + 2 * cp;
      const float* us = Ud + kfirst * UP;
#pragma unroll 1
      for (int k = 0; k < a8; k += KB) {
#pragma unroll
        for (int s = 0; s < KB / KQ; ++s) fma_cols<R>(v, ld_pair(xs + KS * s * PT), us + KS * s * UP);
        xs += KB * PT;
        us += KB * UP;
      }
    }
    sum_cols<R>(v, NP, 32);
    if (p.project_only) {
      const int64_t i = (int64_t)i_c * TC + 2 * cp;
      float* dst = p.Y + (int64_t)o_c * p.y_so + i;
#pragma unroll
      for (int j = 0; j < R; ++j)
        if (j < r && j % KQ == kq) {
          const float2 w = col_pair<R>(v, j);
          if constexpr (VEC) {
            if (i < p.I) *reinterpret_cast<float2*>(dst + j * p.y_sj) = w;
          } else {
            if (i < p.I) dst[j * p.y_sj] = w.x;
            if (i + 1 < p.I) dst[j * p.y_sj + 1] = w.y;
          }
        }
    } else {
#pragma unroll
      for (int j = 0; j < R; ++j)
        if (j % KQ == kq) *reinterpret_cast<float2*>(Vt + j * TC + 2 * cp) = col_pair<R>(v, j);
      __syncwarp();
      const TX* xr[RK];
#pragma unroll
      for (int i = 0; i < RK; ++i) xr[i] = Tc + (lane + 32 * i < a ? lane + 32 * i : 0) * PT;
#pragma unroll 2
      for (int q = 0; q < TC; q += 4) {
        f2 x0[RK], x1[RK];
#pragma unroll
        for (int i = 0; i < RK; ++i) ld_quad(xr[i] + q, x0[i], x1[i]);
#pragma unroll
        for (int j = 0; j < R; ++j) {
          const ulonglong2 w = *reinterpret_cast<const ulonglong2*>(Vt + j * TC + q);
#pragma unroll
          for (int i = 0; i < RK; ++i) {
            ffma2(acc[i][j], x0[i], w.x);
            ffma2(acc[i][j], x1[i], w.y);
          }
        }
      }
    }
    __syncwarp();
    o_c = o_n; i_c = i_n;
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  if (p.project_only) return;
  if (tid == 0) pdl_wait();
  __syncthreads();
  // one partial of P per CTA: the warps' sums meet in warp order
  float* red = Ud + a8 * UP;                         // [nw][R][a] over the (idle) tiles
#pragma unroll
  for (int i = 0; i < RK; ++i) {
    const int k = lane + 32 * i;
    if (k < a) {
#pragma unroll
      for (int j = 0; j < R; ++j) {
        const float2 w = unpack2(acc[i][j]);
        red[(warp * R + j) * a + k] = w.x + w.y;
      }
    }
  }
  __syncthreads();
  for (int e = tid; e < a * R; e += blockDim.x) {
    const int j = e / a, k = e - j * a;
    float s = 0.f;
#pragma unroll 4
    for (int w = 0; w < nw; ++w) s += red[w * a * R + e];
    if (j < r) p.Pp[((int64_t)blockIdx.x * a + k) * r + j] = s;
  }
}

size_t wf_warp_bytes(int a, int R, int rk, bool bf16) {
  const int tc = bf16 ? wf_cols<__nv_bfloat16>(rk) : wf_cols<float>(rk), a8 = (a + 7) & ~7;
  return (size_t)R * tc * 4 + (size_t)2 * a8 * (tc + 4) * (bf16 ? 2 : 4);
}
size_t wf_fixed_bytes(int a) { return (size_t)((a + 7) & ~7) * 12 * 4; }
int wf_rk(int a) { return a <= 32 ? 1 : (a <= 64 ? 2 : 4); }
// warps of a CTA: as many as fit, or as few of them as take the same number of tiles each on 148 CTAs
int ws_balance(size_t fit, int64_t tiles) {
  const int64_t n = std::min<int64_t>((int64_t)fit, kWMaxWarps), rounds = (tiles + 148 * n - 1) / (148 * n);
  return (int)((tiles + 148 * rounds - 1) / (148 * rounds));
}
int wf_warps(int64_t tiles, int a, int R, bool bf16) {
  return ws_balance((kWSmemBudget - wf_fixed_bytes(a)) / wf_warp_bytes(a, R, wf_rk(a), bf16), tiles);
}


// ---------------------------------------------------------------------------------------------
// k_wplane.  Tile = np whole planes X[h][w] of H x W.  Three passes over a tile:
//   rows     V4[h][j]  = sum_w X[h][w] U4[w][j]
//   columns  V3[w][j]  = sum_h X[h][w] U3[h][j]   and   P4[w][j] += sum_h X[h][w] V4[h][j]
//   rows     P3[h][j] += sum_w X[h][w] V3[w][j]
// A lane owns one pair of columns and two rows of one plane of the tile (the same ones in every tile, so that P3 and P4
// stay in registers).  Where a tile has fewer columns or rows than that, 2, 4 or 8 neighbouring lanes share them (nsc,
// nsr) and meet by shuffles; np is as large as 32 pairs of columns and 32 pairs of rows allow.  The reads of shared
// memory bound the kernel: 606 cycles a warp for two planes of 27 x 27 at ranks 5..8.
// ---------------------------------------------------------------------------------------------
template <int R, bool VEC, typename TX>
__global__ void __launch_bounds__(32 * kWMaxWarps, 1) k_wplane(const __grid_constant__ PlaneArgs p) {
  extern __shared__ __align__(16) unsigned char ws_smem[];
  pass_begin(p.clear, p.first);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = blockDim.x >> 5;
  const int H = p.H, W = p.W, np = p.np, PT = p.pitch, W2 = (W + 1) >> 1, W4 = (W + 3) >> 2, H2 = (H + 1) >> 1;
  const int nsc = p.nsc, nsr = p.nsr;
  const int v4s = H * R + 4, v3s = R * PT + 4;       // one plane's V4 and V3, padded off each other's banks
  float* U3d = reinterpret_cast<float*>(ws_smem);    // [H][R]
  float* U4t = U3d + H * R;                          // [R][PT], columns >= W zero
  float* V4d = U4t + R * PT + warp * np * (v4s + v3s);   // [np][H][R]
  float* V3t = V4d + np * v4s;                       // [np][R][PT]
  TX* T = reinterpret_cast<TX*>(U4t + R * PT + nw * np * (v4s + v3s)) + (size_t)warp * (2 * np * H * PT);
  for (int e = tid; e < H * R; e += blockDim.x) {
    const int k = e / R, j = e % R;
    const float u = j < p.r3 ? p.U3[k * p.r3 + j] : 0.f;
    U3d[e] = u;
  }
  for (int e = tid; e < R * PT; e += blockDim.x) {
    const int j = e / PT, k = e - j * PT;
    U4t[e] = (j < p.r4 && k < W) ? p.U4[k * p.r4 + j] : 0.f;
  }
  for (int e = lane; e < 2 * np * H * PT; e += 32) T[e] = TX(0.f);   // the padding stays zero
  for (int e = lane; e < np * v3s; e += 32) V3t[e] = 0.f;
  __syncthreads();
  const TX* __restrict__ X = static_cast<const TX*>(p.X);
  const int HW = H * W, n_planes = (int)p.n_planes, total = (n_planes + np - 1) / np, stride = (int)gridDim.x * nw;
  // the first value this lane copies, and the step to its next one, as (row, column)
  const int unit = VEC ? 4 : 1, wu = W / unit;
  const int l_r = lane / wu, l_c = lane - l_r * wu, s_r = 32 / wu, s_c = 32 - s_r * wu;
  auto stage = [&](TX* dst, int t) {
    if (t < total) {
      const int nrows = np * H, nvalid = (n_planes - t * np < np ? n_planes - t * np : np) * H;
      const TX* src = X + (int64_t)t * np * HW;
      if constexpr (VEC || sizeof(TX) == 4) {
        int rr = l_r, c = l_c;
        const TX* sp = src + unit * lane;
#pragma unroll 4
        for (; rr < nrows; sp += 32 * unit) {
          const bool on = rr < nvalid;
          if constexpr (VEC) cp_quad(dst + rr * PT + 4 * c, on ? sp : src, on);
          else cp_one(dst + rr * PT + c, on ? sp : src, on);
          rr += s_r;
          c += s_c;
          if (c >= wu) { c -= wu; ++rr; }
        }
      } else {
        int rr = l_r, c = l_c;
        const TX* sp = src + lane;
#pragma unroll 1
        for (int e0 = lane; e0 < np * HW; e0 += 32 * 16) {
          TX v[16];
#pragma unroll
          for (int u = 0; u < 16; ++u) v[u] = e0 + 32 * u < nvalid * W ? sp[32 * u] : TX(0.f);
#pragma unroll
          for (int u = 0; u < 16; ++u) {
            if (e0 + 32 * u < np * HW) dst[rr * PT + c] = v[u];
            rr += s_r;
            c += s_c;
            if (c >= W) { c -= W; ++rr; }
          }
          sp += 32 * 16;
        }
      }
    }
    cp_commit();
  };
  // column role: lane = ((plane, pair), share); row role: lane = ((plane, i), share), rows i and i + H2
  const int ci = lane / nsc, cs = lane - ci * nsc;
  const bool c_on = ci < np * W2;
  const int c_pl = c_on ? ci / W2 : 0, c_p = c_on ? ci - c_pl * W2 : 0;
  const int ri = lane / nsr, r_s = lane - ri * nsr;
  const bool r_on = ri < np * H2;
  const int r_pl = r_on ? ri / H2 : 0, r_i = r_on ? ri - r_pl * H2 : 0;
  const bool r_two = r_i + H2 < H;                   // an odd height leaves the last lane one row
  const int r_row0 = r_pl * H + r_i, r_row1 = r_two ? r_row0 + H2 : r_row0;
  f2 acc3[2][R], acc4[2][R / 2];
#pragma unroll
  for (int j = 0; j < R; ++j) acc3[0][j] = acc3[1][j] = acc4[j & 1][j >> 1] = 0ull;
  int t = warp * (int)gridDim.x + (int)blockIdx.x, buf = 0;
  stage(T, t);
  for (; t < total; t += stride) {
    const TX* Tc = T + buf * (np * H * PT);
    buf ^= 1;
    stage(T + buf * (np * H * PT), t + stride);
    cp_wait1();
    __syncwarp();
    {                                                // V4: rows
      f2 v[2][R];
#pragma unroll
      for (int j = 0; j < R; ++j) v[0][j] = v[1][j] = 0ull;
      const TX* x0 = Tc + r_row0 * PT;
      const TX* x1 = Tc + r_row1 * PT;
      // all lanes take the same number of steps; a share past the row reads its last quad against zeros
#pragma unroll 2
      for (int i = 0; i < W4; i += nsr) {
        const int qa = i + r_s, wa = 4 * (qa < W4 ? qa : W4 - 1);
        f2 xa, xb, ya, yb;
        ld_quad(x0 + wa, xa, xb);
        ld_quad(x1 + wa, ya, yb);
        if (qa >= W4) xa = xb = ya = yb = 0ull;
#pragma unroll
        for (int j = 0; j < R; ++j) {
          const ulonglong2 u = *reinterpret_cast<const ulonglong2*>(U4t + j * PT + wa);
          ffma2(v[0][j], xa, u.x);
          ffma2(v[0][j], xb, u.y);
          ffma2(v[1][j], ya, u.x);
          ffma2(v[1][j], yb, u.y);
        }
      }
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        float s[R];
#pragma unroll
        for (int j = 0; j < R; ++j) {
          const float2 w = unpack2(v[q][j]);
          s[j] = w.x + w.y;
        }
        for (int o = 1; o < nsr; o *= 2)
#pragma unroll
          for (int j = 0; j < R; ++j) s[j] += __shfl_xor_sync(0xffffffffu, s[j], o);
        if (r_on && r_s == 0 && (q == 0 || r_two)) {
          float* d = V4d + r_pl * v4s + (r_i + q * H2) * R;
#pragma unroll
          for (int j = 0; j < R; j += 4) *reinterpret_cast<float4*>(d + j) = make_float4(s[j], s[j + 1], s[j + 2], s[j + 3]);
        }
      }
    }
    __syncwarp();
    {                                                // V3 and P4: columns
      f2 v[2][R / 2];
#pragma unroll
      for (int j = 0; j < R / 2; ++j) v[0][j] = v[1][j] = 0ull;
      const TX* x0 = Tc + c_pl * H * PT + 2 * c_p;
      const float* v4 = V4d + c_pl * v4s;
#pragma unroll 2
      for (int i = 0; i < H; i += nsc) {
        const int h = i + cs < H ? i + cs : H - 1;
        f2 x = ld_pair(x0 + h * PT);
        if (i + cs >= H) x = 0ull;
        fma_cols<R>(v, x, U3d + h * R);
        fma_cols<R>(acc4, x, v4 + h * R);
      }
      sum_cols<R>(v, 1, nsc);
      if (c_on && cs == 0) {
        float* d = V3t + c_pl * v3s + 2 * c_p;
#pragma unroll
        for (int j = 0; j < R; ++j) *reinterpret_cast<float2*>(d + j * PT) = col_pair<R>(v, j);
      }
    }
    __syncwarp();
    {                                                // P3: rows
      const TX* x0 = Tc + r_row0 * PT;
      const TX* x1 = Tc + r_row1 * PT;
      const float* va = V3t + r_pl * v3s;
#pragma unroll 1
      for (int i = 0; i < W4; i += nsr) {
        const int qa = i + r_s, wa = 4 * (qa < W4 ? qa : W4 - 1);
        f2 xa, xb, ya, yb;
        ld_quad(x0 + wa, xa, xb);
        ld_quad(x1 + wa, ya, yb);
        if (qa >= W4) xa = xb = ya = yb = 0ull;
#pragma unroll
        for (int j = 0; j < R; ++j) {
          const ulonglong2 u = *reinterpret_cast<const ulonglong2*>(va + j * PT + wa);
          ffma2(acc3[0][j], xa, u.x);
          ffma2(acc3[0][j], xb, u.y);
          ffma2(acc3[1][j], ya, u.x);
          ffma2(acc3[1][j], yb, u.y);
        }
      }
    }
    __syncwarp();
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  if (tid == 0) pdl_wait();
  __syncthreads();
  // one partial of P3 and of P4 per CTA: warps, then planes, then shares, in index order
  float* red3 = U4t + R * PT;                        // [nw][R][2][32], over the idle tiles
  float* red4 = red3 + nw * R * 64;                  // [nw][R][2][32]
#pragma unroll
  for (int j = 0; j < R; ++j) {
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const float2 w = unpack2(acc3[q][j]);
      red3[((warp * R + j) * 2 + q) * 32 + lane] = w.x + w.y;
    }
    const float2 c = col_pair<R>(acc4, j);
    red4[(warp * R + j) * 64 + lane] = c.x;
    red4[(warp * R + j) * 64 + 32 + lane] = c.y;
  }
  __syncthreads();
  for (int e = tid; e < (H + W) * R; e += blockDim.x) {
    const bool rows = e < H * R;
    const int n = rows ? H : W, f = rows ? e : e - H * R, j = f / n, k = f - j * n;
    const int half = rows ? (k >= H2 ? 1 : 0) : (k & 1), i = rows ? k - half * H2 : k >> 1;
    const int ns = rows ? nsr : nsc, per = (rows ? H2 : W2) * ns;
    const float* src = (rows ? red3 : red4) + (j * 2 + half) * 32 + i * ns;
    float s = 0.f;
#pragma unroll 2
    for (int w = 0; w < nw; ++w)
      for (int q = 0; q < np; ++q)
        for (int o = 0; o < ns; ++o) s += src[w * R * 64 + q * per + o];
    if (rows) {
      if (j < p.r3) p.Pp3[((int64_t)blockIdx.x * H + k) * p.r3 + j] = s;
    } else {
      if (j < p.r4) p.Pp4[((int64_t)blockIdx.x * W + k) * p.r4 + j] = s;
    }
  }
}

// planes per tile, row pitch, lanes per column pair and per row
void wp_geometry(int H, int W, int* np, int* pitch, int* nsc, int* nsr) {
  const int w2 = (W + 1) / 2, h2 = (H + 1) / 2, q = (W + 3) / 4;
  *pitch = 4 * (q | 1);
  *np = std::max(1, std::min(32 / w2, 32 / h2));
  *nsc = *nsr = 1;
  while (*nsc < 8 && 2 * *nsc <= H && *np * w2 * 2 * *nsc <= 32) *nsc *= 2;
  while (*nsr < 8 && 2 * *nsr <= q && *np * h2 * 2 * *nsr <= 32) *nsr *= 2;
}
size_t wp_fixed_bytes(int H, int pitch, int R) { return (size_t)(H * R + R * pitch) * 4; }
size_t wp_warp_bytes(int H, int np, int pitch, int R, bool bf16) {
  const size_t b = (size_t)np * ((size_t)(H * R + 4 + R * pitch + 4) * 4 + (size_t)2 * H * pitch * (bf16 ? 2 : 4));
  return std::max(b, (size_t)128 * R * 4);           // the final sums of a warp
}
int wp_warps(int64_t n_planes, int H, int W, int R, bool bf16) {
  int np, pitch, nsc, nsr;
  wp_geometry(H, W, &np, &pitch, &nsc, &nsr);
  return ws_balance((kWSmemBudget - wp_fixed_bytes(H, pitch, R)) / wp_warp_bytes(H, np, pitch, R, bf16),
                    (n_planes + np - 1) / np);
}

template <int R, int RK, bool VEC, typename TX>
cudaError_t wfiber_t(const Fiber2Args& p, int grid, cudaStream_t st) {
  const bool bf16 = sizeof(TX) == 2;
  const int nw = wf_warps(p.n_tiles, p.a, R, bf16);
  const size_t smem = wf_fixed_bytes(p.a) + nw * wf_warp_bytes(p.a, R, RK, bf16);
  cudaError_t e = opt_in_smem(reinterpret_cast<const void*>(k_wfiber<R, RK, VEC, TX>), smem);
  if (e != cudaSuccess) return e;
  return launch_pdl(k_wfiber<R, RK, VEC, TX>, dim3(grid), dim3(32 * nw), smem, st, p);
}
template <int R, int RK>
cudaError_t wfiber_x(const Fiber2Args& p, int grid, bool bf16, bool vec, cudaStream_t st) {
  if (bf16) return vec ? wfiber_t<R, RK, true, __nv_bfloat16>(p, grid, st) : wfiber_t<R, RK, false, __nv_bfloat16>(p, grid, st);
  return vec ? wfiber_t<R, RK, true, float>(p, grid, st) : wfiber_t<R, RK, false, float>(p, grid, st);
}
template <int R>
cudaError_t wfiber_r(const Fiber2Args& p, int grid, bool bf16, bool vec, cudaStream_t st) {
  switch (wf_rk(p.a)) {
    case 1: return wfiber_x<R, 1>(p, grid, bf16, vec, st);
    case 2: return wfiber_x<R, 2>(p, grid, bf16, vec, st);
    default: return wfiber_x<R, 4>(p, grid, bf16, vec, st);
  }
}
template <int R, bool VEC, typename TX>
cudaError_t wplane_t(const PlaneArgs& p, int grid, cudaStream_t st) {
  const bool bf16 = sizeof(TX) == 2;
  const int nw = wp_warps(p.n_planes, p.H, p.W, R, bf16);
  const size_t smem = wp_fixed_bytes(p.H, p.pitch, R) + nw * wp_warp_bytes(p.H, p.np, p.pitch, R, bf16);
  cudaError_t e = opt_in_smem(reinterpret_cast<const void*>(k_wplane<R, VEC, TX>), smem);
  if (e != cudaSuccess) return e;
  return launch_pdl(k_wplane<R, VEC, TX>, dim3(grid), dim3(32 * nw), smem, st, p);
}
template <int R>
cudaError_t wplane_r(const PlaneArgs& p, int grid, bool bf16, bool vec, cudaStream_t st) {
  if (bf16) return vec ? wplane_t<R, true, __nv_bfloat16>(p, grid, st) : wplane_t<R, false, __nv_bfloat16>(p, grid, st);
  return vec ? wplane_t<R, true, float>(p, grid, st) : wplane_t<R, false, float>(p, grid, st);
}

}  // namespace

bool wfiber_supported(int64_t O, int64_t a, int64_t I, int r) {
  return r <= 8 && a <= 128 && I > 1 && wfiber_tiles(O, a, I, false) < (1ll << 30);
}
int64_t wfiber_tiles(int64_t O, int64_t a, int64_t I, bool bf16) {
  const int rk = wf_rk((int)a), tc = bf16 ? wf_cols<__nv_bfloat16>(rk) : wf_cols<float>(rk);
  return O * ((I + tc - 1) / tc);
}
// the same count for both types (a bf16 plan without tensor-core products has the fp32 plan's workspace)
int wfiber_grid(int64_t O, int64_t a, int64_t I, int r) {
  const int64_t tiles = wfiber_tiles(O, a, I, false), nw = wf_warps(tiles, (int)a, r <= 4 ? 4 : 8, false);
  return (int)std::min<int64_t>((tiles + nw - 1) / nw, 148);
}
cudaError_t launch_wfiber(const Fiber2Args& p0, int grid, bool bf16, cudaStream_t st) {
  Fiber2Args p = p0;
  p.n_tiles = wfiber_tiles(p.O, p.a, p.I, bf16);
  const double xbytes = (double)p.O * p.a * p.I * (bf16 ? 2 : 4);
  ProfScope prof(p.project_only ? ASI_K_MODEPROD : ASI_K_EXPAND, st, xbytes);
  const uintptr_t align = bf16 ? 7u : 15u;
  const bool vec = p.I % 4 == 0 && (reinterpret_cast<uintptr_t>(p.X) & align) == 0 &&
                   (!p.project_only || ((reinterpret_cast<uintptr_t>(p.Y) & 7u) == 0 && p.y_so % 2 == 0 && p.y_sj % 2 == 0));
  return p.r <= 4 ? wfiber_r<4>(p, grid, bf16, vec, st) : wfiber_r<8>(p, grid, bf16, vec, st);
}

bool wplane_supported(int64_t n_planes, int64_t H, int64_t W, int r3, int r4) {
  return r3 <= 8 && r4 <= 8 && H >= 1 && H <= 64 && W >= 1 && W <= 64 && n_planes < (1ll << 30);
}
int wplane_grid(int64_t n_planes, int H, int W, int r, bool bf16) {
  int np, pitch, nsc, nsr;
  wp_geometry(H, W, &np, &pitch, &nsc, &nsr);
  const int64_t nw = wp_warps(n_planes, H, W, r <= 4 ? 4 : 8, bf16), tiles = (n_planes + np - 1) / np;
  return (int)std::min<int64_t>((tiles + nw - 1) / nw, 148);
}
cudaError_t launch_wplane(const PlaneArgs& p0, int grid, bool bf16, cudaStream_t st) {
  PlaneArgs p = p0;
  wp_geometry(p.H, p.W, &p.np, &p.pitch, &p.nsc, &p.nsr);
  ProfScope prof(ASI_K_EXPAND, st, (double)p.n_planes * p.H * p.W * (bf16 ? 2 : 4));
  const bool vec = p.W % 4 == 0 && (reinterpret_cast<uintptr_t>(p.X) & (bf16 ? 7u : 15u)) == 0;
  return std::max(p.r3, p.r4) <= 4 ? wplane_r<4>(p, grid, bf16, vec, st) : wplane_r<8>(p, grid, bf16, vec, st);
}

}  // namespace asi
