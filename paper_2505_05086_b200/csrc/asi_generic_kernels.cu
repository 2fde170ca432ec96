// Shape-generic kernels of the ASI path (any number of modes, any sizes, ranks <= 64).
// They are the correctness baseline every layer shape can fall back on; shape-specialised
// kernels live in their own files.
//
//   k_fiber    : both products of a mode in one pass, ranks <= 8
//   k_qrb_*    : Orthogonalize(P) for ranks 65..128 as Cholesky-QR in fp64 (up to 64: asi_orth_kernels.cu)
//   k_conv_tail: terms 4 and 5 of C_ASI (appendix "Speedup")
#include <cuda_bf16.h>

#include <algorithm>
#include <map>
#include <mutex>
#include <type_traits>
#include <utility>

#include "asi_internal.h"

namespace asi {

ProfState g_prof = {0, nullptr, 0, 0, 0.0};

cudaError_t opt_in_smem(const void* kernel, size_t need) {
  static std::mutex lock;
  static std::map<std::pair<int, const void*>, size_t> granted;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  std::lock_guard<std::mutex> guard(lock);
  size_t& have = granted[std::make_pair(dev, kernel)];
  if (need <= have) return cudaSuccess;
  e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)need);
  if (e == cudaSuccess) have = need;
  return e;
}

__device__ __forceinline__ float ld_as_float(const float* p) { return *p; }
__device__ __forceinline__ float ld_as_float(const __nv_bfloat16* p) { return __bfloat162float(*p); }
// ---------------------------------------------------------------------------------------------
// k_fiber: P_m = A_m (A_m^T U_m) for one mode in ONE pass over the activation (Algorithm 1, both
// products of a mode).  A tile is TQ whole fibers of the mode: a rows of TQ contiguous values when the
// mode is not the last one, TQ contiguous fibers when it is.  Per tile, V[q,:] = sum_k X(k,q) U[k,:]
// stays in shared memory and P[k,:] += sum_q X(k,q) V[q,:] accumulates in registers across all tiles
// of the CTA, so V never reaches global memory and each CTA writes one partial of P.  fp32 tiles are
// double-buffered with cp.async.  Requires a <= 128, r <= R.
// ---------------------------------------------------------------------------------------------
constexpr int kFiberTQ = 64;

__device__ __forceinline__ unsigned smem_addr(const void* p) {
  return static_cast<unsigned>(__cvta_generic_to_shared(p));
}

template <int R, typename TX>
__global__ void __launch_bounds__(256) k_fiber(FiberArgs p) {
  constexpr int TQ = kFiberTQ, NT = 256, KS = NT / TQ;
  extern __shared__ __align__(16) float fsm[];
  pass_begin(p.clear, p.clear != nullptr);
  const int tid = threadIdx.x, lane = tid & 31;
  const int a = (int)p.a, r = p.r;
  const bool last = p.I == 1;                       // fibers are contiguous
  // logical X(k, q) of a staged tile sits at k*SK + q*SQ
  const int PQ = TQ + 4;                            // row pitch, 16-byte aligned rows
  const int PA = a | 1;                             // fiber pitch (odd: conflict-free fiber-per-thread reads)
  const int SK = last ? 1 : PQ, SQ = last ? PA : 1;
  const int tile_floats = last ? TQ * PA : a * PQ;
  float* Xs0 = fsm;
  float* Xs1 = fsm + ((tile_floats + 3) & ~3);
  float* Us = Xs1 + ((tile_floats + 3) & ~3);      // [a][R]
  float* Vp = Us + a * R;                           // [KS][TQ][R]
  float* Vs = Vp + KS * TQ * R;                     // [TQ][R]
  for (int idx = tid; idx < a * R; idx += NT) {
    const int k = idx / R, j = idx % R;
    Us[idx] = (j < r) ? p.U[k * r + j] : 0.f;
  }
  const TX* __restrict__ X = reinterpret_cast<const TX*>(p.X);
  const int64_t tiles_per_o = last ? 0 : (p.I + TQ - 1) / TQ;

  auto stage = [&](float* dst, int64_t t, int& n_q) {
    if (last) {
      const int64_t q0 = t * TQ;
      n_q = (int)((p.O - q0 < TQ) ? (p.O - q0) : TQ);
      const TX* src = X + q0 * a;
      for (int idx = tid; idx < n_q * a; idx += NT) {
        const int q = idx / a, k = idx - q * a;
        if constexpr (sizeof(TX) == 4) {
          asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_addr(dst + q * PA + k)), "l"(src + idx) : "memory");
        } else {
          dst[q * PA + k] = ld_as_float(src + idx);
        }
      }
    } else {
      const int64_t o = t / tiles_per_o, i0 = (t - o * tiles_per_o) * TQ;
      n_q = (int)((p.I - i0 < TQ) ? (p.I - i0) : TQ);
      const TX* src = X + o * a * p.I + i0;
      if (sizeof(TX) == 4 && p.vec4) {
        const int n4 = n_q >> 2;                    // I and TQ are multiples of 4 here
        for (int idx = tid; idx < a * n4; idx += NT) {
          const int k = idx / n4, v = idx - k * n4;
          asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_addr(dst + k * PQ + 4 * v)),
                       "l"(src + (int64_t)k * p.I + 4 * v)
                       : "memory");
        }
      } else {
        for (int idx = tid; idx < a * n_q; idx += NT) {
          const int k = idx / n_q, q = idx - k * n_q;
          if constexpr (sizeof(TX) == 4) {
            asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_addr(dst + k * PQ + q)),
                         "l"(src + (int64_t)k * p.I + q)
                         : "memory");
          } else {
            dst[k * PQ + q] = ld_as_float(src + (int64_t)k * p.I + q);
          }
        }
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };

  // thread roles: projection (q, ks), expansion (k, qs)
  const int pq = tid % TQ, pks = tid / TQ;
  int QS = 32;
  while (QS * a > NT && QS > 1) QS >>= 1;           // largest power of two with QS * a <= 256
  const int ek = tid / QS, eqs = tid % QS;
  float acc2[R];
#pragma unroll
  for (int j = 0; j < R; ++j) acc2[j] = 0.f;

  int n_cur = 0, n_next = 0;
  int64_t t = blockIdx.x;
  if (t < p.n_tiles) stage(Xs0, t, n_cur);
  int buf = 0;
  for (; t < p.n_tiles; t += gridDim.x) {
    float* Xc = buf ? Xs1 : Xs0;
    float* Xn = buf ? Xs0 : Xs1;
    const int64_t tn = t + gridDim.x;
    if (tn < p.n_tiles) {
      stage(Xn, tn, n_next);
      asm volatile("cp.async.wait_group 1;" ::: "memory");
    } else {
      asm volatile("cp.async.wait_group 0;" ::: "memory");
    }
    __syncthreads();
    // projection: V[q,:] = sum_k X(k,q) U[k,:]
    {
      float acc[R];
#pragma unroll
      for (int j = 0; j < R; ++j) acc[j] = 0.f;
      if (pq < n_cur) {
#pragma unroll 4
        for (int k = pks; k < a; k += KS) {
          const float x = Xc[k * SK + pq * SQ];
#pragma unroll
          for (int j = 0; j < R; j += 4) {
            const float4 u = *reinterpret_cast<const float4*>(Us + k * R + j);
            acc[j] = fmaf(x, u.x, acc[j]);
            acc[j + 1] = fmaf(x, u.y, acc[j + 1]);
            acc[j + 2] = fmaf(x, u.z, acc[j + 2]);
            acc[j + 3] = fmaf(x, u.w, acc[j + 3]);
          }
        }
      }
#pragma unroll
      for (int j = 0; j < R; j += 4)
        *reinterpret_cast<float4*>(Vp + (pks * TQ + pq) * R + j) = make_float4(acc[j], acc[j + 1], acc[j + 2], acc[j + 3]);
    }
    __syncthreads();
    for (int idx = tid; idx < TQ * R; idx += NT) {
      float v = 0.f;
#pragma unroll
      for (int ks = 0; ks < KS; ++ks) v += Vp[ks * TQ * R + idx];
      Vs[idx] = v;
    }
    __syncthreads();
    // expansion: P[k,:] += sum_q X(k,q) V[q,:]
    if (ek < a) {
#pragma unroll 4
      for (int q = eqs; q < n_cur; q += QS) {
        const float x = Xc[ek * SK + q * SQ];
#pragma unroll
        for (int j = 0; j < R; j += 4) {
          const float4 v = *reinterpret_cast<const float4*>(Vs + q * R + j);
          acc2[j] = fmaf(x, v.x, acc2[j]);
          acc2[j + 1] = fmaf(x, v.y, acc2[j + 1]);
          acc2[j + 2] = fmaf(x, v.z, acc2[j + 2]);
          acc2[j + 3] = fmaf(x, v.w, acc2[j + 3]);
        }
      }
    }
    __syncthreads();
    n_cur = n_next;
    buf ^= 1;
  }
  // the QS threads of a row meet by shuffles (fixed order), one partial of P per CTA
#pragma unroll
  for (int j = 0; j < R; ++j)
    for (int off = 1; off < QS; off <<= 1) acc2[j] += __shfl_xor_sync(0xffffffffu, acc2[j], off);
  (void)lane;
  if (tid == 0) pdl_wait();
  if (ek < a && eqs == 0) {
    float* dst = p.Pp + ((int64_t)blockIdx.x * a + ek) * r;
#pragma unroll
    for (int j = 0; j < R; ++j)
      if (j < r) dst[j] = acc2[j];
  }
}

size_t fiber_smem(int a) {
  const int TQ = kFiberTQ, PQ = TQ + 4, PA = a | 1;
  const size_t tile = (size_t)std::max(TQ * PA, a * PQ);
  return 4 * (2 * ((tile + 3) & ~(size_t)3) + (size_t)a * 8 + 5 * TQ * 8) + 64;
}

int64_t fiber_tiles(int64_t O, int64_t a, int64_t I) {
  (void)a;
  return I == 1 ? (O + kFiberTQ - 1) / kFiberTQ : O * ((I + kFiberTQ - 1) / kFiberTQ);
}

template <int R, typename TX>
static cudaError_t launch_fiber_t(const FiberArgs& p, int grid, cudaStream_t st) {
  const size_t smem = fiber_smem((int)p.a);
  cudaError_t e = opt_in_smem(reinterpret_cast<const void*>(k_fiber<R, TX>), smem);
  if (e != cudaSuccess) return e;
  return launch_pdl(k_fiber<R, TX>, dim3(grid), dim3(256), smem, st, p);
}

cudaError_t launch_fiber(const FiberArgs& p, int grid, bool x_bf16, cudaStream_t st) {
  ProfScope prof(ASI_K_EXPAND, st,
                 (double)p.O * p.a * p.I * (x_bf16 ? 2 : 4) + 4.0 * ((double)p.a * p.r * (grid + 1)));
  if (p.r <= 4) return x_bf16 ? launch_fiber_t<4, __nv_bfloat16>(p, grid, st) : launch_fiber_t<4, float>(p, grid, st);
  return x_bf16 ? launch_fiber_t<8, __nv_bfloat16>(p, grid, st) : launch_fiber_t<8, float>(p, grid, st);
}

// ---------------------------------------------------------------------------------------------
// Orthogonalize for ranks 65..128: the same Cholesky-QR in fp64 in plain kernels (these ranks are rare
// and the matrices small: a x r with r <= 128).  k_qrb_reduce sums the column-split partials in split
// order, k_qrb_gram forms G = P^T P (one thread per entry of the upper triangle, rows in order),
// k_qrb_chol factors G = R^T R in one CTA (shared memory), k_qrb_solve solves u R = p one row per thread.
// ---------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_qrb_reduce(QRArgs args) {
  const QRMode M = args.m[blockIdx.y];
  if (M.r <= kQRMaxRank) return;
  const int64_t n = (int64_t)M.a * M.r;
  for (int64_t e = (int64_t)blockIdx.x * 256 + threadIdx.x; e < n; e += (int64_t)gridDim.x * 256) {
    double acc = 0.0;
    for (int s0 = 0; s0 < M.nsplit; s0 += 8) {
      float t[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) t[q] = __ldcg(M.Pp + (int64_t)((s0 + q < M.nsplit) ? (s0 + q) : 0) * n + e);
#pragma unroll
      for (int q = 0; q < 8; ++q) acc += (s0 + q < M.nsplit) ? (double)t[q] : 0.0;
    }
    M.Pred[e] = acc;
  }
}

__global__ void __launch_bounds__(256) k_qrb_gram(QRArgs args) {
  const QRMode M = args.m[blockIdx.y];
  const int r = M.r;
  if (r <= kQRMaxRank) return;
  const int e = blockIdx.x * 256 + threadIdx.x;
  if (e >= r * r) return;
  const int i = e / r, j = e - i * r;
  if (j < i) return;
  double g = 0.0;
#pragma unroll 4
  for (int k = 0; k < M.a; ++k) g = fma(__ldcg(M.Pred + (int64_t)k * r + i), __ldcg(M.Pred + (int64_t)k * r + j), g);
  M.Gp[e] = g;
}

__global__ void __launch_bounds__(1024) k_qrb_chol(QRArgs args) {
  extern __shared__ double qb_G[];                 // [r][r + 1]
  __shared__ double s_d;
  const QRMode M = args.m[blockIdx.x];
  const int r = M.r, tid = threadIdx.x, P = r + 1;
  if (r <= kQRMaxRank) return;
  for (int e = tid; e < r * r; e += 1024) {
    const int i = e / r, j = e - i * r;
    qb_G[i * P + j] = (j >= i) ? M.Gp[e] : 0.0;
  }
  __syncthreads();
  if (tid == 0) {
    double t = 0.0;
    for (int i = 0; i < r; ++i) t += qb_G[i * P + i];
    s_d = 1e-12 * t;
  }
  __syncthreads();
  const double floor_d = s_d;
  for (int j = 0; j < r; ++j) {
    double d = qb_G[j * P + j];
    if (!(d > floor_d)) {
      if (tid == 0) atomicMax(args.status, (int)ASI_ERR_RANK_DEFICIENT);
      d = (floor_d > 0.0) ? floor_d : 1.0;
    }
    const double inv = rsqrt(d);
    __syncthreads();
    for (int k = j + tid; k < r; k += 1024) qb_G[j * P + k] = (k == j) ? d * inv : qb_G[j * P + k] * inv;
    __syncthreads();
    const int nrem = r - j - 1;
    for (int e = tid; e < nrem * nrem; e += 1024) {
      const int i = j + 1 + e / nrem, k = j + 1 + e % nrem;
      if (k >= i) qb_G[i * P + k] -= qb_G[j * P + i] * qb_G[j * P + k];
    }
    __syncthreads();
  }
  for (int e = tid; e < r * r; e += 1024) {
    const int i = e / r, j = e - i * r;
    M.Gp[e] = (j >= i) ? qb_G[i * P + j] : 0.0;    // R, upper triangular
  }
}

__global__ void __launch_bounds__(128) k_qrb_solve(QRArgs args) {
  extern __shared__ double qb_R[];                 // [r][r]
  const QRMode M = args.m[blockIdx.y];
  const int r = M.r;
  if (r <= kQRMaxRank) return;
  for (int e = threadIdx.x; e < r * r; e += 128) qb_R[e] = M.Gp[e];
  __syncthreads();
  const int row = blockIdx.x * 128 + threadIdx.x;
  if (row >= M.a) return;
  double u[2 * kQRMaxRank];
  const double* prow = M.Pred + (int64_t)row * r;
  for (int j = 0; j < r; ++j) {
    double s = prow[j];
    for (int i = 0; i < j; ++i) s = fma(-u[i], qb_R[i * r + j], s);
    u[j] = s / qb_R[j * r + j];
  }
  float* urow = M.Uout + (int64_t)row * r;
  for (int j = 0; j < r; ++j) urow[j] = (float)u[j];
}

cudaError_t launch_qr_big(const QRArgs& p, int nd, cudaStream_t st) {
  int amax = 1, rmax = 1;
  for (int m = 0; m < nd; ++m)
    if (p.m[m].r > kQRMaxRank) {
      amax = std::max(amax, p.m[m].a);
      rmax = std::max(rmax, p.m[m].r);
    }
  k_qrb_reduce<<<dim3(64, (unsigned)nd), 256, 0, st>>>(p);
  k_qrb_gram<<<dim3((unsigned)((rmax * rmax + 255) / 256), (unsigned)nd), 256, 0, st>>>(p);
  const size_t chol_smem = (size_t)rmax * (rmax + 1) * sizeof(double), solve_smem = (size_t)rmax * rmax * sizeof(double);
  cudaError_t e = opt_in_smem(reinterpret_cast<const void*>(k_qrb_chol), chol_smem);
  if (e == cudaSuccess) e = opt_in_smem(reinterpret_cast<const void*>(k_qrb_solve), solve_smem);
  if (e != cudaSuccess) return e;
  k_qrb_chol<<<nd, 1024, chol_smem, st>>>(p);
  k_qrb_solve<<<dim3((unsigned)((amax + 127) / 128), (unsigned)nd), 128, solve_smem, st>>>(p);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------------------------
// k_conv_tail: one CTA per output channel c'.  Thread (o, s): output o = (j, kh, kw) of Z4 and
// split s of the reduction over (i, h'); partial sums meet in shared memory in a fixed order.
// Then dW[c', :, :, :] = Z4[c'] x_2 U2 over the channels of c''s group.
// A chain of dependent reads: 1024 threads and sixteen reads in flight each (27 x 27 maps, stride 2, Cout = 90,
// ranks 5: 256 threads with one read at a time took 40 us).
// ---------------------------------------------------------------------------------------------
constexpr int kTailNT = 1024;

// splits s of the reduction over (i, h'): as many as the CTA's threads hold
__host__ __device__ static inline int conv_tail_split(int n_out, int n_items) {
  const int n = n_out <= kTailNT ? kTailNT / n_out : 1;
  return n < n_items ? n : n_items;
}

__global__ void __launch_bounds__(kTailNT) k_conv_tail(ConvTailArgs p) {
  extern __shared__ float sm[];
  pdl_wait();
  const int tid = threadIdx.x;
  const int co = blockIdx.x;
  const int kk = p.kh * p.kw;
  const int n_out = p.r2 * kk;
  const int nsplit = conv_tail_split(n_out, p.r1 * p.Ho);
  float* Z4s = sm;                       // [n_out]
  float* red = sm + n_out;               // [nsplit][n_out]
  const int n_items = p.r1 * p.Ho;
  for (int t0 = tid; t0 < n_out * nsplit; t0 += kTailNT) {
    const int s = t0 / n_out, o = t0 - s * n_out;
    const int j = o / kk, t = o - j * kk, ky = t / p.kw, kx = t - ky * p.kw;
    const int wo_lo = (p.pw - kx > 0) ? (p.pw - kx + p.sw - 1) / p.sw : 0;
    int wo_hi = (p.W - 1 + p.pw - kx >= 0) ? (p.W - 1 + p.pw - kx) / p.sw + 1 : 0;
    if (wo_hi > p.Wo) wo_hi = p.Wo;
    float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 1
    for (int it = s; it < n_items; it += nsplit) {
      const int i = it / p.Ho, ho = it - i * p.Ho;
      const int h = ho * p.sh + ky - p.ph;
      if (h < 0 || h >= p.H) continue;
      const float* z1 = p.Z1 + (((int64_t)i * p.Cout + co) * p.Ho + ho) * p.Wo;
      const float* z3 = p.Z3 + (((int64_t)i * p.r2 + j) * p.H + h) * p.W + kx - p.pw;
      // sixteen products in flight, from clamped addresses
#pragma unroll 1
      for (int wo = wo_lo; wo < wo_hi; wo += 8) {
        float x[8], y[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          const int w = wo + e < wo_hi ? wo + e : wo;
          x[e] = __ldg(z1 + w);
          y[e] = __ldg(z3 + w * p.sw);
        }
#pragma unroll
        for (int e = 0; e < 8; ++e)
          if (wo + e < wo_hi) acc[e & 3] = fmaf(x[e], y[e], acc[e & 3]);
      }
    }
    red[t0] = (acc[0] + acc[1]) + (acc[2] + acc[3]);
  }
  __syncthreads();
  for (int o = tid; o < n_out; o += kTailNT) {
    float v = 0.f;
    for (int s = 0; s < nsplit; ++s) v += red[s * n_out + o];
    Z4s[o] = v;
  }
  __syncthreads();
  const int cg = p.C / p.groups, og = p.Cout / p.groups;
  const int g = co / og;
  float* dw = p.dW + (int64_t)co * cg * kk;
  for (int idx = tid; idx < cg * kk; idx += kTailNT) {
    const int cl = idx / kk, t = idx - cl * kk;
    const float* u = p.U2 + (int64_t)(g * cg + cl) * p.r2;
    float v = 0.f;
#pragma unroll 4
    for (int j = 0; j < p.r2; ++j) v = fmaf(Z4s[j * kk + t], __ldg(u + j), v);
    dw[idx] = v;
  }
}

// ---------------------------------------------------------------------------------------------
// Terms 4 and 5 for large output maps, in two launches so the long reduction over (i, h', w') is
// spread over Cout x nsp CTAs: k_conv_z4 writes nsp partial Z4 per output channel (CTA (c', sp)
// takes the pairs (i, h') == sp (mod nsp); thread (o, g) every G-th of those), k_conv_dw sums them in
// order and expands with U2.  Loop bounds are computed per tap, so the inner loops carry no branch.
// ---------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_conv_z4(ConvTailArgs p, float* __restrict__ Z4p, int nsp) {
  extern __shared__ float sm[];
  pdl_launch_dependents();
  pdl_wait();
  const int tid = threadIdx.x;
  const int co = blockIdx.x, sp = blockIdx.y;
  const int kk = p.kh * p.kw;
  const int n_out = p.r2 * kk;
  const int G = (n_out <= 256) ? 256 / n_out : 1;
  float* red = sm;                                  // [G][n_out]
  const int n_items = p.r1 * p.Ho;
  for (int t = tid; t < n_out * G; t += 256) {
    const int o = t % n_out, g = t / n_out;
    const int j = o / kk, tt = o % kk, ky = tt / p.kw, kx = tt % p.kw;
    int wo_lo = (p.pw - kx > 0) ? (p.pw - kx + p.sw - 1) / p.sw : 0;
    int wo_hi = (p.W - 1 + p.pw - kx >= 0) ? (p.W - 1 + p.pw - kx) / p.sw + 1 : 0;
    if (wo_hi > p.Wo) wo_hi = p.Wo;
    float acc0 = 0.f, acc1 = 0.f;
    for (int it = sp + nsp * g; it < n_items; it += nsp * G) {
      const int i = it / p.Ho, ho = it - i * p.Ho;
      const int h = ho * p.sh + ky - p.ph;
      if (h < 0 || h >= p.H) continue;
      const float* z1 = p.Z1 + (((int64_t)i * p.Cout + co) * p.Ho + ho) * p.Wo;
      const float* z3 = p.Z3 + (((int64_t)i * p.r2 + j) * p.H + h) * p.W + kx - p.pw;
      int wo = wo_lo;
#pragma unroll 4
      for (; wo + 1 < wo_hi; wo += 2) {
        acc0 = fmaf(__ldg(z1 + wo), __ldg(z3 + wo * p.sw), acc0);
        acc1 = fmaf(__ldg(z1 + wo + 1), __ldg(z3 + (wo + 1) * p.sw), acc1);
      }
      if (wo < wo_hi) acc0 = fmaf(__ldg(z1 + wo), __ldg(z3 + wo * p.sw), acc0);
    }
    red[g * n_out + o] = acc0 + acc1;
  }
  __syncthreads();
  for (int o = tid; o < n_out; o += 256) {
    float v = 0.f;
    for (int g = 0; g < G; ++g) v += red[g * n_out + o];
    Z4p[((int64_t)sp * p.Cout + co) * n_out + o] = v;
  }
}

__global__ void __launch_bounds__(256) k_conv_dw(ConvTailArgs p, const float* Z4p, int nsp) {
  extern __shared__ float sm[];
  pdl_wait();
  const int tid = threadIdx.x;
  const int co = blockIdx.x;
  const int kk = p.kh * p.kw;
  const int n_out = p.r2 * kk;
  float* Z4s = sm;
  for (int o = tid; o < n_out; o += 256) {
    float v = 0.f;
    for (int s = 0; s < nsp; ++s) v += Z4p[((int64_t)s * p.Cout + co) * n_out + o];
    Z4s[o] = v;
  }
  __syncthreads();
  const int cg = p.C / p.groups, og = p.Cout / p.groups;
  const int g = co / og;
  float* dw = p.dW + (int64_t)co * cg * kk;
  for (int idx = tid; idx < cg * kk; idx += 256) {
    const int cl = idx / kk, t = idx % kk;
    const float* u = p.U2 + (int64_t)(g * cg + cl) * p.r2;
    float v = 0.f;
    for (int j = 0; j < p.r2; ++j) v = fmaf(Z4s[j * kk + t], u[j], v);
    dw[idx] = v;
  }
}

cudaError_t launch_conv_tail_split(const ConvTailArgs& p, float* Z4p, int nsp, cudaStream_t st) {
  ProfScope prof(ASI_K_CONV_TAIL, st,
                 4.0 * ((double)p.r1 * p.Cout * p.Ho * p.Wo + (double)p.r1 * p.r2 * p.H * p.W +
                        (double)p.C * p.r2 + (double)p.Cout * (p.C / p.groups) * p.kh * p.kw));
  const int n_out = p.r2 * p.kh * p.kw;
  const int G = (n_out <= 256) ? 256 / n_out : 1;
  const size_t smem = (size_t)G * n_out * sizeof(float);
  cudaError_t e = cudaSuccess;
  if (smem > 40 * 1024) {
    e = opt_in_smem(reinterpret_cast<const void*>(k_conv_z4), smem);
    if (e == cudaSuccess) e = opt_in_smem(reinterpret_cast<const void*>(k_conv_dw), smem);
    if (e != cudaSuccess) return e;
  }
  e = launch_pdl(k_conv_z4, dim3(p.Cout, nsp), dim3(256), smem, st, p, Z4p, nsp);
  if (e != cudaSuccess) return e;
  return launch_pdl(k_conv_dw, dim3(p.Cout), dim3(256), (size_t)n_out * sizeof(float), st, p, (const float*)Z4p, nsp);
}

static size_t conv_tail_smem(int r1, int r2, int Ho, int kh, int kw) {
  const size_t n_out = (size_t)r2 * kh * kw;
  return n_out * (1 + conv_tail_split((int)n_out, r1 * Ho)) * sizeof(float);
}
cudaError_t launch_conv_tail(const ConvTailArgs& p, cudaStream_t st) {
  ProfScope prof(ASI_K_CONV_TAIL, st,
                 4.0 * ((double)p.r1 * p.Cout * p.Ho * p.Wo + (double)p.r1 * p.r2 * p.H * p.W +
                        (double)p.C * p.r2 + (double)p.Cout * (p.C / p.groups) * p.kh * p.kw));
  const size_t smem = conv_tail_smem(p.r1, p.r2, p.Ho, p.kh, p.kw);
  if (smem > 40 * 1024) {
    cudaError_t e = opt_in_smem(reinterpret_cast<const void*>(k_conv_tail), smem);
    if (e != cudaSuccess) return e;
  }
  return launch_pdl(k_conv_tail, dim3(p.Cout), dim3(kTailNT), smem, st, p);
}

}  // namespace asi
