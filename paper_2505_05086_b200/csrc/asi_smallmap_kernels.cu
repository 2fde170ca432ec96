// Fused kernels for conv layers with small feature maps (H W <= 256, ranks <= 8) -- the shapes of the ResNet /
// MobileNet tails.  One compress call is three launches:
//
//   k_sm_pass1  : forms every P_m = A_m (A_m^T U_m^prev) (Algorithm 1) tile-locally, so no V_m ever reaches global
//                 memory; the activation is read once from HBM and once more from L2 (mode 1 needs whole batches,
//                 modes 2-4 whole samples);
//   k_sm_reduce : fixed-order fp64 reduction of the per-tile partials of every P_m and per-chunk
//                 shares of the Gram matrices G_m = P_m^T P_m, factored once per mode;
//   k_sm_core   : every CTA finishes Orthogonalize for the factor rows it needs (U_m = P_m R^{-1}: the Gram-Schmidt
//                 basis), then contracts its channels with U_1, U_3, U_4; the last CTAs contract the channels.
//
// and the whole compressed weight gradient is one kernel, k_sm_wgrad (terms 1-5 of C_ASI).
// Every wait on an mbarrier is bounded (about one second); on expiry the CTA records
// ASI_ERR_TIMEOUT in the status word and returns.
#include <cooperative_groups.h>
#include <cuda_bf16.h>

#include <type_traits>

#include "asi_internal.h"

namespace asi {

namespace {

// threads per CTA of the partial-reduction kernel: fused layers (whose grids have many CTAs that end at once: MobileNetV2 tail 16.6 us,
// 20.4 with 512 threads), and the layers of large maps
constexpr int kRedNT = 256, kRedNTLarge = 512;
static_assert(kSolveRows <= kRedNTLarge, "a row a thread");


// ---- bulk-copy engine (TMA, untiled form) and mbarrier ------------------------------------------
__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
               : "memory");
}
// dst and src 16-byte aligned, bytes a multiple of 16
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   smem_u32(dst)),
               "l"(src), "r"(bytes), "r"(smem_u32(bar))
               : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t* bar, uint32_t parity, uint64_t limit_ns) {
  const long long t0 = clock64();
  for (uint32_t it = 0; it < (1u << 28); ++it) {
    if (mbar_try_wait(bar, parity)) return true;
    if ((it & 255u) == 255u && clock64() - t0 > 2 * (long long)limit_ns) return false;
  }
  return false;
}
// Thread 0 waits for the staged tile with a time limit; every thread learns the outcome.  On expiry
// the status word gets ASI_ERR_TIMEOUT and thread 0 gives the copies in flight one more bounded
// wait before the CTA returns.
__device__ __forceinline__ bool cta_wait_tile(uint64_t* bar, int* s_flag, int* status, uint64_t limit_ns) {
  if (threadIdx.x == 0) {
    bool ok = mbar_wait_bounded(bar, 0, limit_ns);
    if (!ok) {
      atomicMax(status, (int)ASI_ERR_TIMEOUT);
      mbar_wait_bounded(bar, 0, limit_ns);
    }
    *s_flag = ok ? 1 : 0;
  }
  __syncthreads();
  const bool ok = *s_flag != 0;
  if (ok)
    for (int it = 0; it < 64 && !mbar_try_wait(bar, 0); ++it) {
    }
  return ok;
}

// Warp 0 stages one contiguous block in chunks of 16 KB.
__device__ __forceinline__ void stage_block(uint64_t* bar, char* dst, const char* src, uint32_t bytes, bool stall) {
  constexpr uint32_t kChunk = 16384;
  const int lane = threadIdx.x & 31;
  if ((threadIdx.x >> 5) != 0) return;
  if (lane == 0) {
    mbar_init(bar, 1);
    mbar_expect_tx(bar, bytes);
  }
  __syncwarp();
  const int nchunk = stall ? 0 : (int)((bytes + kChunk - 1) / kChunk);
  for (int i = lane; i < nchunk; i += 32) {
    const uint32_t off = (uint32_t)i * kChunk;
    const uint32_t n = (bytes - off < kChunk) ? bytes - off : kChunk;
    bulk_g2s(dst + off, src + off, n, bar);
  }
}

// Small read-only arrays a CTA keeps in shared memory (factors, the core).  fac_issue_*() start one
// 4-byte asynchronous copy (cp.async) per element -- short loops, no registers held -- and
// fac_wait() waits for this thread's copies; a __syncthreads() after it publishes them.  Whatever a
// kernel does in between overlaps the single round trip, and these small loads are ahead of its bulk
// traffic in the memory system.
__device__ __forceinline__ void cp_async4(float* dst, const float* src, int bytes /* 4, or 0 to store 0.f */) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(smem_u32(dst)), "l"(src), "r"(bytes) : "memory");
}
// dst[k*RD + j] = j < r ? src[k*r + j] : 0 for k < rows: a factor [rows x r] padded to RD columns
template <int RD, int NT>
__device__ __forceinline__ void fac_issue_padded(const float* __restrict__ src, float* dst, int rows, int r) {
#pragma unroll 1
  for (int idx = threadIdx.x; idx < rows * RD; idx += NT) {
    const int k = idx / RD, j = idx % RD;
    cp_async4(dst + idx, src + (j < r ? k * r + j : 0), j < r ? 4 : 0);
  }
}
__device__ __forceinline__ void fac_wait() {
  asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 0;" ::: "memory");
}
// two packed fp32 values (fma.rn.f32x2): one instruction, two multiply-adds
typedef unsigned long long f2;
__device__ __forceinline__ f2 pack2(float lo, float hi) {
  f2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ void ffma2(f2& d, f2 a, f2 b) { asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(a), "l"(b)); }
__device__ __forceinline__ f2 fmul2(f2 a, f2 b) {
  f2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ float2 unpack2(f2 v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}

template <int R>
__device__ __forceinline__ void fma_row(float (&acc)[R], float x, const float* __restrict__ u) {
#pragma unroll
  for (int j = 0; j < R; j += 4) {
    const float4 v = *reinterpret_cast<const float4*>(u + j);
    acc[j] = fmaf(x, v.x, acc[j]);
    acc[j + 1] = fmaf(x, v.y, acc[j + 1]);
    acc[j + 2] = fmaf(x, v.z, acc[j + 2]);
    acc[j + 3] = fmaf(x, v.w, acc[j + 3]);
  }
}

// Division of a small index (n < 2^21) by a run-time divisor through one reciprocal: the integer
// division sequence costs ~150 cycles of latency, which dominates the short index loops below.
struct FDiv {
  float inv;
  int d;
  __device__ __forceinline__ explicit FDiv(int d_) : inv(1.0f / (float)d_), d(d_) {}
  __device__ __forceinline__ int div(int n) const { return __float2int_rd(((float)n + 0.5f) * inv); }
  __device__ __forceinline__ void divmod(int n, int& q, int& r) const {
    q = div(n);
    r = n - q * d;
  }
};

// Sum of N per-lane values over the 32 lanes of a warp by recursive halving: every step each lane
// hands half of its values to its partner, so the whole reduction costs N-N/32 shuffles.  On return
// v[i], i < N/32, is the total of element scatter_base<N>(lane) + i.  The order of additions is fixed.
template <int N, int OFF>
__device__ __forceinline__ void halving_step(float* v, int lane) {
  constexpr int n = N / 2;
  const bool up = (lane & OFF) != 0;
#pragma unroll
  for (int i = 0; i < n; ++i) {
    const float send = up ? v[i] : v[i + n];
    const float keep = up ? v[i + n] : v[i];
    v[i] = keep + __shfl_xor_sync(0xffffffffu, send, OFF);
  }
}
template <int N>
__device__ __forceinline__ void warp_reduce_scatter(float (&v)[N], int lane) {
  static_assert(N % 32 == 0, "pad the accumulator count to a multiple of 32");
  halving_step<N, 16>(v, lane);
  halving_step<N / 2, 8>(v, lane);
  halving_step<N / 4, 4>(v, lane);
  halving_step<N / 8, 2>(v, lane);
  halving_step<N / 16, 1>(v, lane);
}
template <int N>
__device__ __forceinline__ int scatter_base(int lane) {
  return ((lane >> 4) & 1) * (N / 2) + ((lane >> 3) & 1) * (N / 4) + ((lane >> 2) & 1) * (N / 8) +
         ((lane >> 1) & 1) * (N / 16) + (lane & 1) * (N / 32);
}

__host__ __device__ constexpr int tri_index(int S, int k, int k2) {   // k <= k2 < S, row-major upper triangle
  return k * S - k * (k - 1) / 2 + (k2 - k);
}

// 14 x 14 Gram matrix G = A_m A_m^T of a tile [planes x 196] in 7 x 7 blocks.  With a = rows 0..6 and
// b = rows 7..13 of a fiber, warp role 0 accumulates the upper triangle of a a^T, role 1 that of
// b b^T, role 2 the block a b[0..3]^T and role 3 the block a b[4..6]^T (<= 28 accumulators each).
// A unit is a quarter of a plane (fibers == part mod 4), so the lanes of a warp hit 32 banks; this
// thread takes units u0, u0 + ustride, ...  es = step between the elements of a fiber, cs = step
// between neighbouring fibers (mode 3: 14, 1; mode 4: 1, 14).
template <int es, int cs>
__device__ __forceinline__ void gram14_accumulate(const float* __restrict__ Xs, int PJ, int nunits, int u0, int ustride,
                                                  int role, float (&acc)[32]) {
#pragma unroll
  for (int i = 0; i < 32; ++i) acc[i] = 0.f;
  for (int un = u0; un < nunits; un += ustride) {
    const float* base = Xs + (un >> 2) * PJ;
#pragma unroll 1
    for (int col = un & 3; col < 14; col += 4) {
      const float* colp = base + col * cs;
      if (role < 2) {
        const float* q = colp + role * 7 * es;
        float x[7];
#pragma unroll
        for (int k = 0; k < 7; ++k) x[k] = q[k * es];
#pragma unroll
        for (int k = 0; k < 7; ++k)
#pragma unroll
          for (int k2 = k; k2 < 7; ++k2) acc[tri_index(7, k, k2)] = fmaf(x[k], x[k2], acc[tri_index(7, k, k2)]);
      } else if (role == 2) {
        float xa[7], xb[4];
#pragma unroll
        for (int k = 0; k < 7; ++k) xa[k] = colp[k * es];
#pragma unroll
        for (int k = 0; k < 4; ++k) xb[k] = colp[(7 + k) * es];
#pragma unroll
        for (int k = 0; k < 7; ++k)
#pragma unroll
          for (int k2 = 0; k2 < 4; ++k2) acc[k * 4 + k2] = fmaf(xa[k], xb[k2], acc[k * 4 + k2]);
      } else {
        float xa[7], xb[3];
#pragma unroll
        for (int k = 0; k < 7; ++k) xa[k] = colp[k * es];
#pragma unroll
        for (int k = 0; k < 3; ++k) xb[k] = colp[(11 + k) * es];
#pragma unroll
        for (int k = 0; k < 7; ++k)
#pragma unroll
          for (int k2 = 0; k2 < 3; ++k2) acc[k * 3 + k2] = fmaf(xa[k], xb[k2], acc[k * 3 + k2]);
      }
    }
  }
}
// which role (rl) and accumulator (e) hold element o = k*14 + k2 of the symmetric 14 x 14 matrix
__device__ __forceinline__ void gram14_slot(int o, int& rl, int& e) {
  const int k = o / 14, k2 = o % 14;
  const int lo = k < k2 ? k : k2, hi = k < k2 ? k2 : k;
  if (hi < 7) { rl = 0; e = tri_index(7, lo, hi); }
  else if (lo >= 7) { rl = 1; e = tri_index(7, lo - 7, hi - 7); }
  else if (hi < 11) { rl = 2; e = lo * 4 + (hi - 7); }
  else { rl = 3; e = lo * 3 + (hi - 11); }
}

}  // namespace

// ---------------------------------------------------------------------------------------------
// k_sm_pass1: every P_m = A_m (A_m^T U_m^prev) in one launch, 256 threads per CTA.
//
// Role B (mode 1), one CTA per 128 neighbouring columns (c, h, w): lane = four columns, warp w = the samples b == w
// (mod 8).  The activation goes straight from memory to registers -- a warp reads 512 contiguous bytes per sample --
// V_1 of the columns meets in shared memory, and the expansion reads the 64 KB again (from L1 or L2).  Holding the
// tile in registers instead cost half the CTAs per SM and was slower: 102 against 79 us on the MobileNetV2 tail at 128.
//
// Role C (modes 2, 3, 4), a cluster of `cs` CTAs per sample, each with cc channels of it in shared memory (one bulk
// copy): V_2 is the sum of the CTAs' shares through distributed shared memory, P_2 of the CTA's own channels follows
// from its tile; modes 3 and 4 come from the same planes -- as Gram matrices A_m A_m^T on 7 x 7 and 14 x 14 maps
// (S + 1 multiply-adds per element against 4 r; P_m = G_m U_m^prev is formed in k_sm_reduce), on other maps as the
// two products with a lane per row and per column of a plane.
// The split of a sample over a cluster is what lets two to four CTAs share an SM: with the whole sample and the whole
// batch of a tile in shared memory (up to 204 KB) one CTA per SM waited for its own copy.
// ---------------------------------------------------------------------------------------------
constexpr int kPT = 256;             // threads per CTA of k_sm_pass1 and k_sm_core

// VW neighbouring values as they lie in memory: load() wants the address a multiple of all four, load_any() of one
template <typename TX, int VW> struct RawCol;
template <> struct RawCol<float, 4> {
  float4 v;
  __device__ __forceinline__ void load(const float* p) { v = __ldg(reinterpret_cast<const float4*>(p)); }
  __device__ __forceinline__ void load_any(const float* p) { v = make_float4(__ldg(p), __ldg(p + 1), __ldg(p + 2), __ldg(p + 3)); }
  __device__ __forceinline__ void get(float (&x)[4]) const { x[0] = v.x; x[1] = v.y; x[2] = v.z; x[3] = v.w; }
};
template <> struct RawCol<float, 1> {
  float v;
  __device__ __forceinline__ void load(const float* p) { v = __ldg(p); }
  __device__ __forceinline__ void get(float (&x)[1]) const { x[0] = v; }
};
template <> struct RawCol<__nv_bfloat16, 4> {
  uint2 v;
  __device__ __forceinline__ void load(const __nv_bfloat16* p) { v = __ldg(reinterpret_cast<const uint2*>(p)); }
  __device__ __forceinline__ void load_any(const __nv_bfloat16* p) {
    const unsigned short* q = reinterpret_cast<const unsigned short*>(p);
    v = make_uint2(__ldg(q) | (uint32_t)__ldg(q + 1) << 16, __ldg(q + 2) | (uint32_t)__ldg(q + 3) << 16);
  }
  __device__ __forceinline__ void get(float (&x)[4]) const {
    x[0] = __uint_as_float(v.x << 16); x[1] = __uint_as_float(v.x & 0xffff0000u);
    x[2] = __uint_as_float(v.y << 16); x[3] = __uint_as_float(v.y & 0xffff0000u);
  }
};
template <> struct RawCol<__nv_bfloat16, 1> {
  __nv_bfloat16 v;
  __device__ __forceinline__ void load(const __nv_bfloat16* p) { v = *p; }
  __device__ __forceinline__ void get(float (&x)[1]) const { x[0] = __bfloat162float(v); }
};

// upper triangle of G = A_m A_m^T over the planes pl0, pl0 + 128, .. of a 7 x 7 map
template <int es, int cs>
__device__ __forceinline__ void gram7_accumulate(const float* __restrict__ Xs, int nc, int pl0, float (&acc)[32]) {
#pragma unroll 1
  for (int pl = pl0; pl < nc; pl += 128) {
    const float* base = Xs + pl * 49;
#pragma unroll 1
    for (int col = 0; col < 7; ++col, base += cs) {
      float x[7];
#pragma unroll
      for (int k = 0; k < 7; ++k) x[k] = base[k * es];
#pragma unroll
      for (int k = 0; k < 7; ++k)
#pragma unroll
        for (int k2 = k; k2 < 7; ++k2) acc[tri_index(7, k, k2)] = fmaf(x[k], x[k2], acc[tri_index(7, k, k2)]);
    }
  }
}

// Y[col][:] += x[col] u[:] over a thread's VW columns with column pairs packed: acc[p][j] holds columns 2 p, 2 p + 1
template <int R>
__device__ __forceinline__ void fma_pairs(f2 (&acc)[2][R], float4 x, const f2* __restrict__ ud) {      // ud[j] = (u_j, u_j)
  const f2 x01 = pack2(x.x, x.y), x23 = pack2(x.z, x.w);
#pragma unroll
  for (int j = 0; j < R; j += 2) {
    const ulonglong2 u = *reinterpret_cast<const ulonglong2*>(ud + j);
    ffma2(acc[0][j], x01, u.x); ffma2(acc[1][j], x23, u.x);
    ffma2(acc[0][j + 1], x01, u.y); ffma2(acc[1][j + 1], x23, u.y);
  }
}

template <int R, int VW, bool ANY, typename TX>
__device__ __forceinline__ void pass1_role_b(const SmPass1Args& p, int tile, float* smem) {
  constexpr int JT = 32 * VW, BPG = 32 / R;          // columns; samples per thread and butterfly of the expansion
  constexpr int U = 8;                               // samples in flight per thread
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int B = p.B, r1 = p.r[0];
  const int64_t chw = (int64_t)p.C * p.H * p.W;
  f2* U1d = reinterpret_cast<f2*>(smem);             // [B][R]: (u, u)
  float* part = smem + 2 * B * R;                    // [8][R][JT]
  float* V1s = part + 8 * JT * R;                    // [R][JT]
  for (int idx = tid; idx < B * R; idx += kPT) {
    const int k = idx / R, j = idx % R;
    const float* src = p.U_prev + p.u_off[0] + (j < r1 ? k * r1 + j : 0);
    cp_async4(reinterpret_cast<float*>(U1d + idx), src, j < r1 ? 4 : 0);
    cp_async4(reinterpret_cast<float*>(U1d + idx) + 1, src, j < r1 ? 4 : 0);
  }
  const int64_t col = (int64_t)tile * JT + VW * lane;
  const bool con = col < chw;
  const int nb = B > warp ? (B - warp + 7) / 8 : 0;  // samples of this warp: warp, warp + 8, ..
  const TX* A = reinterpret_cast<const TX*>(p.act) + (con ? col : 0) + (nb > 0 ? (int64_t)warp * chw : 0);
  const int64_t step = 8 * chw;
  f2 acc[2][R];                                      // VW == 1: the low half of acc[0]
#pragma unroll
  for (int c = 0; c < 2; ++c)
#pragma unroll
    for (int j = 0; j < R; ++j) acc[c][j] = 0ull;
  bool waited = false;
#pragma unroll 1
  for (int t0 = 0; t0 < nb || !waited; t0 += U) {
    RawCol<TX, VW> x[U];
#pragma unroll
    for (int t = 0; t < U; ++t) {
      const TX* at = A + (int64_t)(t0 + t < nb ? t0 + t : 0) * step;
      if constexpr (ANY) x[t].load_any(at);
      else x[t].load(at);
    }
    if (!waited) {
      fac_wait();
      __syncthreads();
      waited = true;
    }
#pragma unroll
    for (int t = 0; t < U; ++t) {
      if (t0 + t < nb) {                             // warp-uniform
        float xs[VW];
        x[t].get(xs);
        const f2* ud = U1d + (warp + 8 * (t0 + t)) * R;
        if constexpr (VW == 4) {
          fma_pairs<R>(acc, make_float4(xs[0], xs[1], xs[2], xs[3]), ud);
        } else {
#pragma unroll
          for (int j = 0; j < R; ++j) ffma2(acc[0][j], pack2(xs[0], 0.f), ud[j]);
        }
      }
    }
  }
  // V_1 of the tile, [j][column]: the eight warps' shares meet in warp order
#pragma unroll
  for (int j = 0; j < R; ++j) {
    float* dst = part + (warp * R + j) * JT + VW * lane;
    if constexpr (VW == 4) *reinterpret_cast<ulonglong2*>(dst) = make_ulonglong2(acc[0][j], acc[1][j]);
    else *dst = unpack2(acc[0][j]).x;
  }
  __syncthreads();
  for (int idx = tid; idx < JT * R; idx += kPT) {
    float s = part[idx];
#pragma unroll
    for (int w = 1; w < 8; ++w) s += part[w * JT * R + idx];
    V1s[idx] = s;
  }
  __syncthreads();
  pdl_launch_dependents();
#pragma unroll
  for (int j = 0; j < R; ++j) {
    if constexpr (VW == 4) {
      const ulonglong2 s = *reinterpret_cast<const ulonglong2*>(V1s + j * JT + 4 * lane);
      acc[0][j] = con ? s.x : 0ull;
      acc[1][j] = con ? s.y : 0ull;
    } else {
      acc[0][j] = con ? pack2(V1s[j * JT + lane], 0.f) : 0ull;
    }
  }
  // P1[b,:] = sum over the tile's columns of X[b][col] V1[col,:]: BPG samples meet in one butterfly of 32 values
  float* P1 = p.Pp[0] + (int64_t)tile * B * r1;
  const int e = scatter_base<32>(lane), eb = warp + 8 * (e / R), ej = e % R;
#pragma unroll 1
  for (int t0 = 0; t0 < nb; t0 += BPG) {
    RawCol<TX, VW> x[BPG];
#pragma unroll
    for (int q = 0; q < BPG; ++q) {
      const TX* at = A + (int64_t)(t0 + q < nb ? t0 + q : nb - 1) * step;
      if constexpr (ANY) x[q].load_any(at);
      else x[q].load(at);
    }
    float val[32];
#pragma unroll
    for (int q = 0; q < BPG; ++q) {
      float xs[VW];
      x[q].get(xs);
      if constexpr (VW == 4) {
        const f2 x01 = pack2(xs[0], xs[1]), x23 = pack2(xs[2], xs[3]);
#pragma unroll
        for (int j = 0; j < R; ++j) {
          f2 s = fmul2(x01, acc[0][j]);
          ffma2(s, x23, acc[1][j]);
          const float2 h = unpack2(s);
          val[q * R + j] = h.x + h.y;
        }
      } else {
#pragma unroll
        for (int j = 0; j < R; ++j) val[q * R + j] = xs[0] * unpack2(acc[0][j]).x;
      }
    }
    warp_reduce_scatter<32>(val, lane);
    const int b = eb + 8 * t0;
    if (b < B && ej < r1) P1[b * r1 + ej] = val[0];
  }
}

// modes 3 and 4 of nc planes [H][W] in shared memory (pitch P): P_m = A_m (A_m^T U_m), lane = (plane of the warp's
// group, row or column).  Rows are read rotated by the lane so that an even width does not fold them onto a few banks.
template <int R>
__device__ __forceinline__ void planes_modes34(const float* Xs, int P, int nc, int H, int W, const float* U3s, const float* U4s,
                                               float* Vw, float* red, float* P3, float* P4, int r3, int r4) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int L = H > W ? H : W, G = 32 / L;
  const int g = lane / L, x = lane - g * L;
  float* V = Vw + warp * 32 * R;                     // [32 lanes][R] of this warp
  float a3[R], a4[R];
#pragma unroll
  for (int j = 0; j < R; ++j) a3[j] = a4[j] = 0.f;
#pragma unroll 1
  for (int p0 = warp * G; p0 < nc; p0 += 8 * G) {
    const bool on = g < G && p0 + g < nc;
    const float* Xp = Xs + (on ? p0 + g : 0) * P;
    float v[R];
#pragma unroll
    for (int j = 0; j < R; ++j) v[j] = 0.f;
    if (on && x < W) {
#pragma unroll 4
      for (int h = 0; h < H; ++h) fma_row<R>(v, Xp[h * W + x], U3s + h * R);
    }
    __syncwarp();
#pragma unroll
    for (int j = 0; j < R; j += 4) *reinterpret_cast<float4*>(V + lane * R + j) = make_float4(v[j], v[j + 1], v[j + 2], v[j + 3]);
    __syncwarp();
#pragma unroll
    for (int j = 0; j < R; ++j) v[j] = 0.f;
    if (on && x < H) {
      int w = x < W ? x : 0;
#pragma unroll 4
      for (int k = 0; k < W; ++k) {
        const float xv = Xp[x * W + w];
        fma_row<R>(a3, xv, V + (g * L + w) * R);
        fma_row<R>(v, xv, U4s + w * R);
        if (++w == W) w = 0;
      }
    }
    __syncwarp();
#pragma unroll
    for (int j = 0; j < R; j += 4) *reinterpret_cast<float4*>(V + lane * R + j) = make_float4(v[j], v[j + 1], v[j + 2], v[j + 3]);
    __syncwarp();
    if (on && x < W) {
#pragma unroll 4
      for (int h = 0; h < H; ++h) fma_row<R>(a4, Xp[h * W + x], V + (g * L + h) * R);
    }
  }
  // [8 warps][32 lanes][2 R]: the planes' shares meet in (warp, group) order
#pragma unroll
  for (int j = 0; j < R; ++j) {
    red[(warp * 32 + lane) * 2 * R + j] = a3[j];
    red[(warp * 32 + lane) * 2 * R + R + j] = a4[j];
  }
  __syncthreads();
  for (int idx = tid; idx < (H + W) * R; idx += kPT) {
    const bool m4 = idx >= H * R;
    const int e = m4 ? idx - H * R : idx, k = e / R, j = e % R;
    float s = 0.f;
    for (int w = 0; w < 8; ++w)
      for (int q = 0; q < G; ++q) s += red[(w * 32 + q * L + k) * 2 * R + (m4 ? R : 0) + j];
    if (!m4 && j < r3) P3[k * r3 + j] = s;
    if (m4 && j < r4) P4[k * r4 + j] = s;
  }
}

template <int KIND, int R, bool ANY, typename TX>
__device__ __forceinline__ void pass1_role_c(const SmPass1Args& p, int bid, float* smem) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  __shared__ __align__(8) uint64_t s_bar;
  __shared__ int s_flag;
  namespace cg = cooperative_groups;
  const int C = p.C, H = KIND ? KIND : p.H, W = KIND ? KIND : p.W, HW = H * W, P = KIND ? KIND * KIND : p.pitch, cs = p.cs;
  const bool synced = p.cl > 1;                      // CTAs of several samples may share a cluster; all take its barriers
  const int b = bid / cs, rank = bid - b * cs, rank0 = (bid % p.cl) - rank;   // rank0: the sample's first CTA in the cluster
  const int c0 = rank * p.cc, nc = (C - c0 < p.cc) ? (C > c0 ? C - c0 : 0) : p.cc;
  const int r2 = p.r[1];
  float* Xs = smem;                                  // [cc][P]
  float* U2s = smem + p.off_u2;                      // [cc][R]
  float* V2l = U2s + p.cc * R;                       // [HW][R]: this CTA's share of V_2
  float* V2s = V2l + HW * R;                         // [HW][R]
  float* Vp = V2s + HW * R;                          // [G][HW][R], G = 256 / HW
  float* U3s = Vp + (kPT / HW) * HW * R;             // KIND 0: [H][R], [W][R], [8][32][R]
  float* red = Xs;                                   // free once every thread is done with the tile
  const TX* A = reinterpret_cast<const TX*>(p.act) + ((int64_t)b * C + c0) * HW;
  const bool bulk = !ANY && std::is_same<TX, float>::value && p.bulk;
  if (bulk) {
    const char* src = reinterpret_cast<const char*>(A);
    if (P == HW) {
      stage_block(&s_bar, reinterpret_cast<char*>(Xs), src, (uint32_t)(nc * HW) * 4u, p.stall_copy != 0);
    } else if (warp == 0) {                          // one row per channel, padded pitch
      if (lane == 0) {
        mbar_init(&s_bar, 1);
        mbar_expect_tx(&s_bar, (uint32_t)(nc * HW) * 4u);
      }
      __syncwarp();
      for (int c = lane; c < nc && !p.stall_copy; c += 32) bulk_g2s(Xs + c * P, src + (int64_t)c * HW * 4, (uint32_t)HW * 4u, &s_bar);
    }
  }
  for (int idx = tid; idx < nc * R; idx += kPT) {
    const int k = idx / R, j = idx % R;
    cp_async4(U2s + idx, p.U_prev + p.u_off[1] + (j < r2 ? (c0 + k) * r2 + j : 0), j < r2 ? 4 : 0);
  }
  if (KIND == 0)
    for (int idx = tid; idx < (H + W) * R; idx += kPT) {
      const int k = idx / R, j = idx % R, m = k < H ? 2 : 3, kk = k < H ? k : k - H;
      cp_async4(U3s + idx, p.U_prev + p.u_off[m] + (j < p.r[m] ? kk * p.r[m] + j : 0), j < p.r[m] ? 4 : 0);
    }
  if (!bulk) {
    if constexpr (std::is_same<TX, float>::value) {
      const FDiv dHW(HW);
      for (int idx = tid; idx < nc * HW; idx += kPT) {
        int c, q;
        dHW.divmod(idx, c, q);
        cp_async4(Xs + c * P + q, reinterpret_cast<const float*>(A) + idx, 4);
      }
    } else if (!ANY && p.vec4) {
      const FDiv dV(HW % 4 == 0 ? HW / 4 : 1 << 20);
      for (int i0 = tid; i0 < nc * HW / 4; i0 += 4 * kPT) {
        uint2 raw[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) raw[u] = __ldg(reinterpret_cast<const uint2*>(A) + (i0 + u * kPT < nc * HW / 4 ? i0 + u * kPT : 0));
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int i = i0 + u * kPT;
          if (i >= nc * HW / 4) break;
          int c = 0, q = i;
          if (P != HW) dV.divmod(i, c, q);
          *reinterpret_cast<float4*>(Xs + c * P + 4 * q) =
              make_float4(__uint_as_float(raw[u].x << 16), __uint_as_float(raw[u].x & 0xffff0000u),
                          __uint_as_float(raw[u].y << 16), __uint_as_float(raw[u].y & 0xffff0000u));
        }
      }
    } else {
      const FDiv dHW(HW);
      for (int idx = tid; idx < nc * HW; idx += kPT) {
        int c, q;
        dHW.divmod(idx, c, q);
        Xs[c * P + q] = __bfloat162float(reinterpret_cast<const __nv_bfloat16*>(A)[idx]);
      }
    }
  }
  fac_wait();
  bool ok = true;
  if (bulk && nc > 0) ok = cta_wait_tile(&s_bar, &s_flag, p.status, p.wait_ns);
  else __syncthreads();
  // ---- this CTA's share of V_2: thread (g, hw) sums the channels c == g (mod G)
  const int G = kPT / HW;                            // HW <= 256; a constant on the Gram kinds
  {
    const FDiv dHW(HW);
    int g, hw;
    dHW.divmod(tid, g, hw);
    if (g < G && ok) {
      float acc[R];
#pragma unroll
      for (int j = 0; j < R; ++j) acc[j] = 0.f;
#pragma unroll 4
      for (int c = g; c < nc; c += G) fma_row<R>(acc, Xs[c * P + hw], U2s + c * R);
      float* dst = (G == 1 ? V2l : Vp) + (g * HW + hw) * R;
#pragma unroll
      for (int j = 0; j < R; j += 4) *reinterpret_cast<float4*>(dst + j) = make_float4(acc[j], acc[j + 1], acc[j + 2], acc[j + 3]);
    }
    if (G > 1) {
      __syncthreads();
      for (int idx = tid; idx < HW * R; idx += kPT) {
        float s = Vp[idx];
        for (int q = 1; q < G; ++q) s += Vp[q * HW * R + idx];
        V2l[idx] = s;
      }
    }
  }
  if (synced) asm volatile("barrier.cluster.arrive.release;" ::: "memory");
  else __syncthreads();
  // ---- modes 3 and 4 while the other CTAs of the cluster finish their shares
  if (KIND == 7 || KIND == 14) {
    const int wq = warp & 3;                         // warps 0-3: mode 3, warps 4-7: mode 4
    float acc[32];
#pragma unroll
    for (int i = 0; i < 32; ++i) acc[i] = 0.f;
    const int n = ok ? nc : 0;
    if (KIND == 7) {
      if (warp < 4) gram7_accumulate<7, 1>(Xs, n, wq * 32 + lane, acc);
      else gram7_accumulate<1, 7>(Xs, n, wq * 32 + lane, acc);
    } else {
      if (warp < 4) gram14_accumulate<14, 1>(Xs, P, n * 4, lane, 32, wq, acc);
      else gram14_accumulate<1, 14>(Xs, P, n * 4, lane, 32, wq, acc);
    }
    warp_reduce_scatter<32>(acc, lane);
    float* gr = Vp;                                  // [8][32] (Vp is at least that large; its sums are in V2l)
    __syncthreads();
    gr[warp * 32 + scatter_base<32>(lane)] = acc[0];
    __syncthreads();
    for (int o = tid; o < 2 * HW; o += kPT) {
      const int m = o >= HW, q = m ? o - HW : o;
      float s;
      if (KIND == 7) {
        const int k = q / 7, k2 = q % 7;
        const int e = (k <= k2) ? tri_index(7, k, k2) : tri_index(7, k2, k);
        s = ((gr[(4 * m) * 32 + e] + gr[(4 * m + 1) * 32 + e]) + gr[(4 * m + 2) * 32 + e]) + gr[(4 * m + 3) * 32 + e];
      } else {
        int rl, e;
        gram14_slot(q, rl, e);
        s = gr[(4 * m + rl) * 32 + e];
      }
      p.Pp[2 + m][(int64_t)bid * HW + q] = s;
    }
  } else {
    float* Vw = U3s + (H + W) * R;
    float* rd = Vw + 8 * 32 * R;
    planes_modes34<R>(Xs, P, ok ? nc : 0, H, W, U3s, U3s + H * R, Vw, rd, p.Pp[2] + (int64_t)bid * H * p.r[2],
                      p.Pp[3] + (int64_t)bid * W * p.r[3], p.r[2], p.r[3]);
  }
  pdl_launch_dependents();
  // ---- V_2 = the shares of the cluster, in rank order
  if (synced) asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
  if (cs > 1) {
    cg::cluster_group cluster = cg::this_cluster();
    for (int idx = tid; idx < HW * R; idx += kPT) {
      float s = cluster.map_shared_rank(V2l, rank0)[idx];
      for (int q = 1; q < cs; ++q) s += cluster.map_shared_rank(V2l, rank0 + q)[idx];
      V2s[idx] = s;
    }
  } else {
    V2s = V2l;
  }
  if (synced) asm volatile("barrier.cluster.arrive.release;" ::: "memory");   // the shares have been read
  __syncthreads();
  // ---- P_2 of the CTA's channels: thread = four channels q, q + Q, .. and a share of the positions
  const int Q = (nc + 3) >> 2;
  if (ok && nc > 0) {
    float* P2 = p.Pp[1] + ((int64_t)b * C + c0) * r2;
    const int parts = Q < kPT ? (kPT / Q < 16 ? kPT / Q : 16) : 1;
    const FDiv dQ(Q);
    const int rounds = (Q * parts + kPT - 1) / kPT;  // > 1 only when parts == 1
#pragma unroll 1
    for (int rd = 0; rd < rounds; ++rd) {
      const int it = tid + rd * kPT;
      int part, q;
      dQ.divmod(it, part, q);
      const bool on = part < parts;
      float acc[4][R];
#pragma unroll
      for (int m = 0; m < 4; ++m)
#pragma unroll
        for (int j = 0; j < R; ++j) acc[m][j] = 0.f;
      if (on) {
        const float* row[4];
#pragma unroll
        for (int m = 0; m < 4; ++m) row[m] = Xs + (q + m * Q < nc ? q + m * Q : q) * P;
        if ((HW & 3) == 0) {
#pragma unroll 1
          for (int hw = 4 * part; hw < HW; hw += 4 * parts) {
            float4 xv[4];
#pragma unroll
            for (int m = 0; m < 4; ++m) xv[m] = *reinterpret_cast<const float4*>(row[m] + hw);
#pragma unroll
            for (int m = 0; m < 4; ++m) {
              fma_row<R>(acc[m], xv[m].x, V2s + hw * R);
              fma_row<R>(acc[m], xv[m].y, V2s + (hw + 1) * R);
              fma_row<R>(acc[m], xv[m].z, V2s + (hw + 2) * R);
              fma_row<R>(acc[m], xv[m].w, V2s + (hw + 3) * R);
            }
          }
        } else {
#pragma unroll 2
          for (int hw = part; hw < HW; hw += parts) {
#pragma unroll
            for (int m = 0; m < 4; ++m) fma_row<R>(acc[m], row[m][hw], V2s + hw * R);
          }
        }
      }
      if (parts > 1) {
        __syncthreads();                             // the tile is free
        if (on) {
#pragma unroll
          for (int m = 0; m < 4; ++m)
#pragma unroll
            for (int j = 0; j < R; j += 4)
              *reinterpret_cast<float4*>(red + ((part * 4 + m) * Q + q) * R + j) = make_float4(acc[m][j], acc[m][j + 1], acc[m][j + 2], acc[m][j + 3]);
        }
        __syncthreads();
        for (int idx = tid; idx < nc * R; idx += kPT) {
          const int c = idx / R, j = idx % R;        // channel c = m Q + q
          float s = red[idx];
          for (int k = 1; k < parts; ++k) s += red[k * 4 * Q * R + idx];
          if (j < r2) P2[c * r2 + j] = s;
        }
      } else if (on) {
#pragma unroll
        for (int m = 0; m < 4; ++m)
#pragma unroll
          for (int j = 0; j < R; ++j)
            if (q + m * Q < nc && j < r2) P2[(q + m * Q) * r2 + j] = acc[m][j];
      }
    }
  }
  if (synced) asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
}

// ANY: the activation starts at any element (its columns still come in groups of four where they are whole groups, so
// that the partials do not depend on the address)
template <int KIND, int R, bool ANY, typename TX>
__device__ __forceinline__ void sm_pass1_cta(const SmPass1Args& p, const int bid) {
  extern __shared__ __align__(128) float smem[];
  const int tid = threadIdx.x;
  pdl_wait();                                        // the first kernel of a call
  if (bid == 0 && tid < 241) p.status[tid == 0 ? 0 : 15 + tid] = 0;  // status word, counters 16..255
  const int nc_ctas = (p.B * p.cs + p.cl - 1) / p.cl * p.cl;
  if (bid >= nc_ctas) {
    const int tile = bid - nc_ctas;
    if (tile >= p.n_tiles_b) return;                 // padding to whole clusters
    if (p.vec4) pass1_role_b<R, 4, ANY, TX>(p, tile, smem);
    else pass1_role_b<R, 1, false, TX>(p, tile, smem);
  } else if (bid < p.B * p.cs) {
    pass1_role_c<KIND, R, ANY, TX>(p, bid, smem);
  } else {                                           // padding: only the cluster's barriers
    for (int i = 0; i < 2; ++i) asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
  }
}

// ---------------------------------------------------------------------------------------------
// k_sm_tile1: the first pass for S x S maps, S in {7, 14, 16}, and batches that are a multiple of 8, where the tiles of
// two CTAs of 512 threads fit an SM (ResNet-18 tail: 19 against 28 us of k_sm_pass1, whose smaller CTAs repeat more
// set-up; a 16 x 16 layer of eight samples: 6.4 against 13 us).  CTAs of role B hold a tile [all B x J contiguous
// (c, h, w)] with whole mode-1/3/4 fibers (one half of the CTA iterates mode 1 while the other does modes 3 and 4);
// CTAs of role C hold one sample [all C x HW] (larger maps: a quarter of its positions) for mode 2.
// ---------------------------------------------------------------------------------------------
constexpr int kTT = 512;             // threads per CTA
constexpr int kNG = 256;             // threads of one half (warp-specialised phases)

__host__ __device__ constexpr int pitch4(int J) {      // >= J, multiple of 4, == 4 (mod 32)
  int p = (J + 3) / 4 * 4;
  while (p % 32 != 4) p += 4;
  return p;
}

__device__ __forceinline__ float to_f(float v) { return v; }
__device__ __forceinline__ float to_f(__nv_bfloat16 v) { return __bfloat162float(v); }

template <typename TX>
__device__ __forceinline__ float4 ld4(const TX* p);
template <>
__device__ __forceinline__ float4 ld4<float>(const float* p) {
  return *reinterpret_cast<const float4*>(p);
}
template <>
__device__ __forceinline__ float4 ld4<__nv_bfloat16>(const __nv_bfloat16* p) {
  const uint2 raw = *reinterpret_cast<const uint2*>(p);
  const __nv_bfloat162 lo = *reinterpret_cast<const __nv_bfloat162*>(&raw.x);
  const __nv_bfloat162 hi = *reinterpret_cast<const __nv_bfloat162*>(&raw.y);
  return make_float4(__low2float(lo), __high2float(lo), __low2float(hi), __high2float(hi));
}

// Starts the copy of `rows` fp32 rows of J values (J a multiple of 4, both sides 16-byte aligned): row i
// from src + i*src_stride to dst + i*PJ, 16 bytes per cp.async, one row per warp at a time.  (One bulk
// copy per row would leave the issuing warp busy for ~60 cycles per row: the tile of a 64-sample
// batch would arrive ~2 us later.)
__device__ __forceinline__ void stage_rows_async(float* dst, const float* __restrict__ src, int rows, int J,
                                                 int64_t src_stride, int PJ) {
  const int lane = threadIdx.x & 31, nv = J >> 2;
  for (int i = threadIdx.x >> 5; i < rows; i += kTT / 32) {
    const float* s = src + i * src_stride;
    float* d = dst + i * PJ;
    for (int v = lane; v < nv; v += 32)
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(d + 4 * v)), "l"(s + 4 * v) : "memory");
  }
}

__device__ __forceinline__ void bar_sync(int id, int nthreads) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(nthreads) : "memory");
}

// Number of interleaved sample groups project_batch uses for a tile of J columns on nthr threads.
__host__ __device__ constexpr int batch_groups(int nthr, int J) {
  const int items = J / 2;
  int nh = nthr / items;
  return nh < 1 ? 1 : (nh > 4 ? 4 : nh);
}

// out[j][0..R) = sum_b Xs[b*PJ + j] * Us[b*R + ..] for j < J: the mode-1 contraction of a staged tile
// [B x J].  Runs on `nthr` threads (t = 0..nthr-1) that synchronise on named barrier `bar`.  A thread
// owns two neighbouring columns (one 8-byte shared load per sample) and the samples b == h (mod NH);
// the NH partial sums meet in `part` ([NH][J][R]) in a fixed order.
template <int R>
__device__ __forceinline__ void project_batch(const float* __restrict__ Xs, int PJ,
                                              const float* __restrict__ Us, int B, int J,
                                              float* __restrict__ part, float* __restrict__ out, int t,
                                              int nthr, int bar) {
  const int NH = batch_groups(nthr, J);
  const int J2 = J >> 1;                             // J is even
  const FDiv dJ2(J2);
#pragma unroll 1
  for (int it = t; it < NH * J2; it += nthr) {
    int h, jp;
    dJ2.divmod(it, h, jp);
    float a0[R], a1[R];
#pragma unroll
    for (int q = 0; q < R; ++q) a0[q] = a1[q] = 0.f;
#pragma unroll 4
    for (int b = h; b < B; b += NH) {
      const float2 x = *reinterpret_cast<const float2*>(Xs + b * PJ + 2 * jp);
      fma_row<R>(a0, x.x, Us + b * R);
      fma_row<R>(a1, x.y, Us + b * R);
    }
    float* dst = (NH > 1 ? part + h * J * R : out) + 2 * jp * R;
#pragma unroll
    for (int q = 0; q < R; q += 4) {
      *reinterpret_cast<float4*>(dst + q) = make_float4(a0[q], a0[q + 1], a0[q + 2], a0[q + 3]);
      *reinterpret_cast<float4*>(dst + R + q) = make_float4(a1[q], a1[q + 1], a1[q + 2], a1[q + 3]);
    }
  }
  if (NH > 1) {
    bar_sync(bar, nthr);
#pragma unroll 1
    for (int idx = t; idx < J * R; idx += nthr) {
      float s = 0.f;
      for (int h = 0; h < NH; ++h) s += part[h * J * R + idx];
      out[idx] = s;
    }
  }
  bar_sync(bar, nthr);
}

// V[hw][:] = sum_c Xs[c*PC + hw] * Us[c][:] for a staged block Xs [C][HWC] of one sample (the mode-2
// projection of HWC positions).  Thread (g, hw) sums the channels c = g (mod G); group 0 writes V
// itself, groups 1..G-1 write Vp ([G-1][HWC][R]; may alias Us: it is written only after every thread
// has finished reading Us) and the sums meet in a fixed order.  All kTT threads call it.
template <int HWC, int PC, int R>
__device__ __forceinline__ void project_channels(const float* __restrict__ Xs, const float* Us, float* Vp,
                                                 float* V, int C) {
  constexpr int G = kTT / HWC;
  const int tid = threadIdx.x;
  float acc[R];
#pragma unroll
  for (int j = 0; j < R; ++j) acc[j] = 0.f;
  const int g = tid / HWC, hw = tid - g * HWC;
  if (g < G) {
#pragma unroll 4
    for (int c = g; c < C; c += G) fma_row<R>(acc, Xs[c * PC + hw], Us + c * R);
  }
  if (G > 1) __syncthreads();
  if (g < G) {
    float* dst = (g == 0 ? V : Vp + (g - 1) * HWC * R) + hw * R;
#pragma unroll
    for (int j = 0; j < R; j += 4)
      *reinterpret_cast<float4*>(dst + j) = make_float4(acc[j], acc[j + 1], acc[j + 2], acc[j + 3]);
  }
  __syncthreads();
  if (G > 1) {
    for (int idx = tid; idx < HWC * R; idx += kTT) {
      float s = V[idx];
#pragma unroll
      for (int gg = 0; gg < G - 1; ++gg) s += Vp[gg * HWC * R + idx];
      V[idx] = s;
    }
    __syncthreads();
  }
}

// Stages one tile [B x J] (row b at src + b*sample_stride) as fp32 rows of pitch PJ.
template <bool ANY, typename TX>
__device__ __forceinline__ void stage_tile_begin(const TX* __restrict__ src, int64_t sample_stride, float* Xs,
                                                 int B, int J, int PJ) {
  if constexpr (ANY) {                               // one value at a time
    for (int b = threadIdx.x >> 5; b < B; b += kTT / 32)
      for (int j = threadIdx.x & 31; j < J; j += 32) Xs[b * PJ + j] = to_f(src[b * sample_stride + j]);
  } else if constexpr (std::is_same<TX, float>::value) {
    stage_rows_async(Xs, src, B, J, sample_stride, PJ);
  } else {
    const int J4 = J / 4;
    for (int idx = threadIdx.x; idx < B * J4; idx += kTT) {
      const int b = idx / J4, v = idx - b * J4;
      *reinterpret_cast<float4*>(Xs + b * PJ + 4 * v) = ld4<TX>(src + b * sample_stride + 4 * v);
    }
  }
}

// Role C of the first pass takes the positions of a sample in NQ parts.  S = 7: the whole map.  Larger
// maps: four parts that start on 16-byte boundaries -- 14 x 14 splits its 49 float4 per channel as
// 13 + 12 + 12 + 12 (parts 1..3 carry four zero columns), 16 x 16 as 4 x 16.
__host__ __device__ constexpr int role_c_hwc(int S) { return S == 7 ? 49 : (S == 14 ? 52 : S * S / 4); }
__host__ __device__ constexpr int role_c_pitch(int S) { return S == 7 ? 49 : pitch4(role_c_hwc(S)); }

template <int S, int R, bool ANY, typename TX>
__device__ __forceinline__ void sm_tile1_cta(const SmTile1Args& p, const int bid) {
  constexpr bool kBulk = std::is_same<TX, float>::value && !ANY;
  constexpr bool kGram = (S == 7);                   // modes 3, 4 as Gram matrices A_m A_m^T (7 x 7)
  constexpr bool kGram14 = (S == 14);                // ... as 14 x 14 Gram matrices in four 7 x 7 blocks
  constexpr int HW = S * S;
  constexpr int CC = (S == 7) ? 4 : 1;               // channels per role-B tile
  constexpr int J = CC * HW;                         // contiguous elements per sample in a tile
  constexpr int PJ = pitch4(J);                      // row pitch == 4 (mod 32): conflict-free (b, j) reads
  constexpr int NH1 = batch_groups(kNG, J);
  extern __shared__ __align__(128) float smem[];
  __shared__ __align__(8) uint64_t s_bar;
  __shared__ int s_flag;
  const int tid = threadIdx.x, lane = tid & 31;
  const TX* __restrict__ A = reinterpret_cast<const TX*>(p.act);
  const int B = p.B, C = p.C;

  pdl_wait();                                        // the first kernel of a call
  if (bid == 0 && tid < 241) p.status[tid == 0 ? 0 : 15 + tid] = 0;  // status word, counters 16..255

  constexpr int kNQ = (S == 7) ? 1 : 4;             // role-C CTAs per sample
  if (bid >= B * kNQ) {
    // ---------------- role B: modes 1, 3, 4 on tile [B x J] ----------------
    const int tile = bid - B * kNQ;
    float* Xs = smem;                                // [B][PJ]
    float* U1s = Xs + B * PJ;                        // [B][R]
    float* U3s = U1s + B * R;                        // [S][R]
    float* U4s = U3s + S * R;                        // [S][R]
    float* V1s = U4s + S * R;                        // [J][R]
    float* part = V1s + J * R;                       // [NH1][J][R] (NH1 > 1 only)
    float* red = part + (NH1 > 1 ? NH1 : 0) * J * R; // [8][32], S = 14: [8 + 16][32]
    fac_issue_padded<R, kTT>(p.U_prev + p.u_off[0], U1s, B, p.r[0]);
    if constexpr (!kGram && !kGram14) {
      fac_issue_padded<R, kTT>(p.U_prev + p.u_off[2], U3s, S, p.r[2]);
      fac_issue_padded<R, kTT>(p.U_prev + p.u_off[3], U4s, S, p.r[3]);
    }
    stage_tile_begin<ANY, TX>(A + (int64_t)tile * J, (int64_t)C * HW, Xs, B, J, PJ);
    fac_wait();
    __syncthreads();
    const int t = tid & (kNG - 1), wg = t >> 5;
    if (tid < kNG) {
      // ---- half 0: mode 1.  V[j,:] = sum_b X[b,j] U1[b,:], then P1[b,:] = sum_j X[b,j] V[j,:]
      project_batch<R>(Xs, PJ, U1s, B, J, part, V1s, t, kNG, 1);
      float* P1 = p.Pp[0] + (int64_t)tile * B * p.r[0];
      const int bl = lane >> 2, jl = lane & 3;       // a warp covers 8 samples x 4 column phases
      for (int b0 = wg * 8; b0 < B; b0 += 64) {
        const int b = b0 + bl;
        float acc[R];
#pragma unroll
        for (int q = 0; q < R; ++q) acc[q] = 0.f;
#pragma unroll 7
        for (int jj = jl; jj < J; jj += 4) fma_row<R>(acc, Xs[b * PJ + jj], V1s + jj * R);
#pragma unroll
        for (int q = 0; q < R; ++q) {
          acc[q] += __shfl_xor_sync(0xffffffffu, acc[q], 1);
          acc[q] += __shfl_xor_sync(0xffffffffu, acc[q], 2);
        }
        if (jl == 0) {
#pragma unroll
          for (int q = 0; q < R; ++q)
            if (q < p.r[0]) P1[b * p.r[0] + q] = acc[q];
        }
      }
    } else if constexpr (kGram) {
      // ---- half 1, S = 7: G_m = A_m A_m^T for m = 3, 4, one plane (b, c) per thread at a time; the
      // 32 lanes of a warp touch 32 different banks.  P_m = G_m U_m^prev follows in k_sm_reduce.
      constexpr int NACC = 32;
      static_assert(S * (S + 1) / 2 <= NACC, "upper triangle of the Gram matrix");
      const int nplanes = B * CC;
#pragma unroll 1
      for (int mode = 2; mode <= 3; ++mode) {
        const int es = (mode == 2) ? S : 1;          // step between the elements of a fiber
        const int cs = (mode == 2) ? 1 : S;          // step between neighbouring fibers
        float* Gm = p.Pp[mode] + (int64_t)tile * HW;
        float acc[NACC];
#pragma unroll
        for (int i = 0; i < NACC; ++i) acc[i] = 0.f;
        for (int pl = t; pl < nplanes; pl += kNG) {
          const int b = pl / CC, cl = pl % CC;
          const float* base = Xs + b * PJ + cl * HW;
#pragma unroll 1
          for (int col = 0; col < S; ++col) {
            const float* colp = base + col * cs;
            float x[S];
#pragma unroll
            for (int k = 0; k < S; ++k) x[k] = colp[k * es];
#pragma unroll
            for (int k = 0; k < S; ++k)
#pragma unroll
              for (int k2 = k; k2 < S; ++k2) acc[tri_index(S, k, k2)] = fmaf(x[k], x[k2], acc[tri_index(S, k, k2)]);
          }
        }
        warp_reduce_scatter<NACC>(acc, lane);
        red[wg * 32 + scatter_base<NACC>(lane)] = acc[0];
        bar_sync(2, kNG);
        for (int o = t; o < HW; o += kNG) {
          const int k = o / S, k2 = o % S;
          const int e = (k <= k2) ? tri_index(S, k, k2) : tri_index(S, k2, k);
          float s = 0.f;
#pragma unroll
          for (int w = 0; w < 8; ++w) s += red[w * 32 + e];
          Gm[o] = s;
        }
        bar_sync(2, kNG);
      }
    } else if constexpr (kGram14) {
      // ---- half 1, S = 14: G_3 = A_3 A_3^T (see gram14_accumulate); G_4 follows on all sixteen warps
      const int role = wg & 3;
      float* Gm = p.Pp[2] + (int64_t)tile * HW;
      float acc[32];
      gram14_accumulate<S, 1>(Xs, PJ, B * 4, (wg >> 2) * 32 + lane, 64, role, acc);
      warp_reduce_scatter<32>(acc, lane);
      red[wg * 32 + scatter_base<32>(lane)] = acc[0];
      bar_sync(2, kNG);
      for (int o = t; o < HW; o += kNG) {
        int rl, e;
        gram14_slot(o, rl, e);
        Gm[o] = red[rl * 32 + e] + red[(rl + 4) * 32 + e];
      }
    } else {
      // ---- half 1, other sizes: P_m = A_m (A_m^T U_m^prev) for m = 3, 4.  A unit is a quarter of a plane
      // (columns == part mod 4); unit -> thread so that the 32 lanes of a warp touch 32 different
      // banks.  Each thread owns 2 columns of the factor; warp w serves column pair w mod JH.
      constexpr int TPP = 4, JT = 2, JH = R / JT, NACC = 32;
      static_assert(S * JT <= NACC, "accumulators of one thread");
      const int jh = wg % JH;
      const int u0 = (wg / JH) * 32 + lane;
      const int nunits = B * CC * TPP;
#pragma unroll 1
      for (int mode = 2; mode <= 3; ++mode) {
        const float* Us = ((mode == 2) ? U3s : U4s) + jh * JT;
        const int es = (mode == 2) ? S : 1;
        const int cs = (mode == 2) ? 1 : S;
        const int rm = p.r[mode];
        float* Pm = p.Pp[mode] + (int64_t)tile * S * rm;
        float acc[NACC];
#pragma unroll
        for (int i = 0; i < NACC; ++i) acc[i] = 0.f;
        for (int un = u0; un < nunits; un += kNG / JH) {
          const int pl = un / TPP, part_ = un % TPP;
          const int b = pl / CC, cl = pl % CC;
          const float* base = Xs + b * PJ + cl * HW;
#pragma unroll 1
          for (int col = part_; col < S; col += TPP) {
            const float* colp = base + col * cs;
            float x[S], v0 = 0.f, v1 = 0.f;
#pragma unroll
            for (int k = 0; k < S; ++k) {
              x[k] = colp[k * es];
              const float2 u = *reinterpret_cast<const float2*>(Us + k * R);
              v0 = fmaf(x[k], u.x, v0);
              v1 = fmaf(x[k], u.y, v1);
            }
#pragma unroll
            for (int k = 0; k < S; ++k) {
              acc[2 * k] = fmaf(x[k], v0, acc[2 * k]);
              acc[2 * k + 1] = fmaf(x[k], v1, acc[2 * k + 1]);
            }
          }
        }
        warp_reduce_scatter<NACC>(acc, lane);
        red[wg * 32 + scatter_base<NACC>(lane)] = acc[0];
        bar_sync(2, kNG);
        for (int o = t; o < S * R; o += kNG) {
          const int k = o / R, j = o % R;
          const int e = k * JT + (j % JT);
          float s = 0.f;
          for (int w = j / JT; w < 8; w += JH) s += red[w * 32 + e];
          if (j < rm) Pm[k * rm + j] = s;
        }
        bar_sync(2, kNG);
      }
    }
    if constexpr (kGram14) {
      // ---- S = 14, G_4 = A_4 A_4^T: each half joins as it finishes its first job (mode 1 or G_3)
      const int gw = tid >> 5, role = gw & 3;
      float* red4 = red + 8 * 32;                    // [16][32]
      float acc[32];
      gram14_accumulate<1, S>(Xs, PJ, B * 4, (gw >> 2) * 32 + lane, 128, role, acc);
      warp_reduce_scatter<32>(acc, lane);
      red4[gw * 32 + scatter_base<32>(lane)] = acc[0];
      __syncthreads();
      float* Gm = p.Pp[3] + (int64_t)tile * HW;
      for (int o = tid; o < HW; o += kTT) {
        int rl, e;
        gram14_slot(o, rl, e);
        Gm[o] = ((red4[rl * 32 + e] + red4[(rl + 4) * 32 + e]) + red4[(rl + 8) * 32 + e]) + red4[(rl + 12) * 32 + e];
      }
    }
  } else {
    // ---------------- role C: mode 2 on block [C x HWC] of one sample ----------------
    // S = 7: the whole sample (contiguous, staged by the bulk-copy engine, odd row pitch for the
    // row-per-thread reads below); larger maps: one part of the positions, rows staged by 16-byte
    // cp.async at a pitch == 4 (mod 32), read back as float4.
    constexpr int NQ = (S == 7) ? 1 : 4;
    constexpr int HWC = role_c_hwc(S);
    constexpr int PC = role_c_pitch(S);
    constexpr int G = kTT / HWC;
    constexpr bool kBulkC = kBulk && NQ == 1;
    const int b = bid / NQ, q = bid % NQ;
    const int hw0 = (S == 14) ? (q == 0 ? 0 : 4 + 48 * q) : q * HWC;     // first position of this part
    const int nval = (S == 14 && q > 0) ? 48 : HWC;                      // positions it holds
    float* Xs = smem;                                // [C][PC]
    float* U2s = Xs + ((C * PC + 3) & ~3);           // [C][R]
    float* V2s = U2s + C * R;                        // [HWC][R]
    float* Vp = (C >= (G - 1) * HWC) ? U2s : V2s + HWC * R;   // [G-1][HWC][R]: on top of U2s when it fits
    const TX* Xb = A + (int64_t)b * C * HW + hw0;
    if constexpr (kBulkC)
      stage_block(&s_bar, reinterpret_cast<char*>(Xs), reinterpret_cast<const char*>(Xb), (uint32_t)C * HW * 4u,
                  p.stall_copy != 0);
    fac_issue_padded<R, kTT>(p.U_prev + p.u_off[1], U2s, C, p.r[1]);
    if constexpr (ANY) {                             // one value at a time
      for (int c = tid >> 5; c < C; c += kTT / 32)
        for (int v = lane; v < HWC; v += 32) Xs[c * PC + v] = v < nval ? to_f(Xb[(int64_t)c * HW + v]) : 0.f;
    } else if constexpr (kBulkC) {
    } else if constexpr (NQ == 1) {
      const int n4 = C * HW / 4;
      for (int idx = tid; idx < n4; idx += kTT) *reinterpret_cast<float4*>(Xs + 4 * idx) = ld4<TX>(Xb + 4 * idx);
    } else {
      constexpr int NV = HWC / 4;
      const int n = C * NV;
#pragma unroll 1
      for (int idx = tid; idx < n; idx += kTT) {
        const int c = idx / NV, v = idx - c * NV;
        float* dst = Xs + c * PC + 4 * v;
        const TX* src = Xb + (int64_t)c * HW + 4 * v;
        if (4 * v >= nval) {
          *reinterpret_cast<float4*>(dst) = make_float4(0.f, 0.f, 0.f, 0.f);
        } else if constexpr (kBulk) {
          asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
        } else {
          *reinterpret_cast<float4*>(dst) = ld4<TX>(src);
        }
      }
    }
    fac_wait();
    if constexpr (kBulkC) {
      if (!cta_wait_tile(&s_bar, &s_flag, p.status, p.wait_ns)) return;
    } else {
      __syncthreads();
    }
    project_channels<HWC, PC, R>(Xs, U2s, Vp, V2s, C);
    // expansion: P2[c,:] = sum_hw X[c,hw] V2[hw,:], one channel row per thread
    float* P2 = p.Pp[1] + (int64_t)bid * C * p.r[1];
    for (int c = tid; c < C; c += kTT) {
      const float* row = Xs + c * PC;
      float acc[R];
#pragma unroll
      for (int j = 0; j < R; ++j) acc[j] = 0.f;
      if constexpr (NQ == 1) {
#pragma unroll 7
        for (int hw = 0; hw < HWC; ++hw) fma_row<R>(acc, row[hw], V2s + hw * R);
      } else {
#pragma unroll 2
        for (int hw = 0; hw < HWC; hw += 4) {
          const float4 x = *reinterpret_cast<const float4*>(row + hw);
          fma_row<R>(acc, x.x, V2s + hw * R);
          fma_row<R>(acc, x.y, V2s + (hw + 1) * R);
          fma_row<R>(acc, x.z, V2s + (hw + 2) * R);
          fma_row<R>(acc, x.w, V2s + (hw + 3) * R);
        }
      }
#pragma unroll
      for (int j = 0; j < R; ++j)
        if (j < p.r[1]) P2[c * p.r[1] + j] = acc[j];
    }
  }
}

// A launch over several layers at once: the CTAs of layer l are [first[l], first[l + 1]).
constexpr int kMaxBatch = 8;
template <typename Args>
struct SmBatch {
  Args a[kMaxBatch];
  int first[kMaxBatch + 1];
  int n;
};
template <typename Args>
__device__ __forceinline__ int batch_layer(const SmBatch<Args>& b, int bid) {
  int l = 0;
  while (l + 1 < b.n && bid >= b.first[l + 1]) ++l;
  return l;
}

template <int S, int R, bool ANY, typename TX>
__global__ void __launch_bounds__(kTT, 2) k_sm_tile1(const __grid_constant__ SmTile1Args p) {
  sm_tile1_cta<S, R, ANY, TX>(p, (int)blockIdx.x);
}
template <int S, int R, typename TX>
__global__ void __launch_bounds__(kTT, 2) k_sm_tile1_b(const __grid_constant__ SmBatch<SmTile1Args> b) {
  const int l = batch_layer(b, (int)blockIdx.x);
  sm_tile1_cta<S, R, false, TX>(b.a[l], (int)blockIdx.x - b.first[l]);
}

template <int KIND, int R, bool ANY, typename TX>
__global__ void __launch_bounds__(kPT, R == 4 ? 4 : 2) k_sm_pass1(const __grid_constant__ SmPass1Args p) {
  sm_pass1_cta<KIND, R, ANY, TX>(p, (int)blockIdx.x);
}
template <int KIND, int R, typename TX>
__global__ void __launch_bounds__(kPT, R == 4 ? 4 : 2) k_sm_pass1_b(const __grid_constant__ SmBatch<SmPass1Args> b) {
  const int l = batch_layer(b, (int)blockIdx.x);
  sm_pass1_cta<KIND, R, false, TX>(b.a[l], (int)blockIdx.x - b.first[l]);
}

// ---------------------------------------------------------------------------------------------
// k_sm_reduce: CTA (c, m) sums rows [16 c, 16 c + 16) of the per-tile partials of P_m in fp64 in a
// fixed order (thread (e, sg) takes the partials s == sg (mod SG); the SG sums meet in shared memory
// in index order), stores them in fp64 and adds its share of P_m^T P_m.  A mode whose partials are
// Gram matrices A_m A_m^T (a <= 16) is summed the same way, a slice of the a x a elements per CTA.
// With args.factor the last CTA of a mode to finish then factors the mode once for all CTAs of the
// core kernel: it sums the shares of P_m^T P_m (a Gram mode: forms P_m = G_m U_m^prev first), and
// leaves the Cholesky factor R_m and 1 / diag(R_m) in args.Rf; LARGE also solves for the rows of U_m.
// LARGE (the layers of large maps, 148 to 296 partials a mode, at most kSolveRows rows): a chain of round trips to memory, so 512 threads with sixteen
// partials each in flight, and the rows solved here: 10.7 us where 256 threads took 11.7 and a launch for the rows 3.5 more
// (128 x 128 x 28 x 28 bf16, one layer's step 91.3 -> 89.2 us).  Fused layers lose by it (MobileNetV2 tail 165 -> 168 us).
// ---------------------------------------------------------------------------------------------
template <bool LARGE>
__device__ __forceinline__ void sm_reduce_cta(const SmReduceArgs& args, const int c, const int mode) {
  constexpr int RM = 8, RPC = kRedRows, NT = LARGE ? kRedNTLarge : kRedNT;
  const SmReduceMode M = args.m[mode];   // a copy in registers: reading the fields through the parameter each time cost 9 % of a step
  pdl_launch_dependents();
  if (c >= M.nchunk) return;
  pdl_wait();                                      // the partials come from the previous kernel
  __shared__ double part[NT];
  __shared__ double Ps[RPC][RM];
  const int tid = threadIdx.x;
  const int r = M.r, a = M.a;
  // a Gram mode: CTA c sums elements [c*per, c*per + per) of G_m = A_m A_m^T over the tiles;
  // otherwise rows [16 c, 16 c + 16) of P_m
  const int per = M.gram ? (a * a + M.nchunk - 1) / M.nchunk : 0;
  const int first = M.gram ? c * per : c * RPC * r;
  const int row0 = c * RPC;
  const int nrow = (a - row0 < RPC) ? (a - row0) : RPC;
  const int E = M.gram ? ((a * a - first < per) ? a * a - first : per) : nrow * r;   // <= 128
  const int64_t stride = M.gram ? (int64_t)a * a : (int64_t)a * r;
  int EP = 32;
  while (EP < E) EP <<= 1;
  const int SG = NT / EP;
  {
    const int e = tid & (EP - 1), sg = tid >> (31 - __clz(EP));
    double acc = 0.0;
    if (e < E) {
      const float* ptr = M.Pp + first + e;
      if constexpr (LARGE) {                         // sixteen partials in flight, the last batch too
#pragma unroll 1
        for (int s = sg; s < M.nsplit; s += 16 * SG) {
          float v[16];
#pragma unroll
          for (int u = 0; u < 16; ++u) v[u] = s + u * SG < M.nsplit ? __ldcg(ptr + (s + u * SG) * stride) : 0.f;
#pragma unroll
          for (int u = 0; u < 16; ++u) acc += (double)v[u];
        }
      } else {
#pragma unroll 8
        for (int s = sg; s < M.nsplit; s += SG) acc += (double)__ldcg(ptr + s * stride);
      }
    }
    part[tid] = acc;
  }
  for (int idx = tid; idx < RPC * RM; idx += NT) Ps[idx / RM][idx % RM] = 0.0;
  __syncthreads();
  if (tid < E) {
    double v = 0.0;
    for (int sg = 0; sg < SG; ++sg) v += part[sg * EP + tid];
    M.Pred[first + tid] = v;                       // P_m rows, or G_m elements for a Gram mode
    if (!M.gram) {
      const FDiv dr(r);
      int k, j;
      dr.divmod(tid, k, j);
      Ps[k][j] = v;
    }
  }
  if (!M.gram) {
    __syncthreads();
    if (tid < r * r) {
      const FDiv dr(r);
      int i, j;
      dr.divmod(tid, i, j);
      double g = 0.0;
      if (j >= i) {
#pragma unroll 4
        for (int rl = 0; rl < RPC; ++rl) g = fma(Ps[rl][i], Ps[rl][j], g);
      }
      M.Gp[((int64_t)c * r + i) * r + j] = g;
    }
  }
  if (!args.factor) return;
  // ---- the last CTA of a mode to get here factors the mode once for every CTA of the core kernel:
  // G_m = P_m^T P_m = R_m^T R_m (Cholesky), stored as the rows of R_m and 1 / diag(R_m)
  __shared__ int s_last;
  __shared__ double Gq[8][RM * RM];
  __shared__ double Gs[RM][RM + 1];
  __shared__ double Dinv[RM];
  __shared__ double Gfull[16 * 16];
  __shared__ double Pm[16][RM];
  __shared__ float Ups[16 * RM];
  __threadfence();
  __syncthreads();
  if (tid == 0) s_last = (atomicAdd(args.counter + mode, 1) == M.nchunk - 1);
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  const int lane = tid & 31, warp = tid >> 5;
  if (!M.gram) {
    // warp q sums the shares of the chunks == q (mod 8); the eight sums meet in index order
    for (int e = lane; e < r * r && warp < 8; e += 32) {
      double g = 0.0;
#pragma unroll 8
      for (int cc = warp; cc < M.nchunk; cc += 8) g += __ldcg(M.Gp + (int64_t)cc * r * r + e);
      Gq[warp][e] = g;
    }
    __syncthreads();
    if (tid < r * r) {
      double g = Gq[0][tid];
#pragma unroll
      for (int q = 1; q < 8; ++q) g += Gq[q][tid];
      const int i = tid / r, k = tid - i * r;
      Gs[i][k] = g;
    }
  } else {
    // Gram mode (a <= 16): P_m = G_m U_m^prev (Algorithm 1: A_m (A_m^T U)), kept in fp64 for the row
    // solves of the core kernel, then its Gram matrix
    for (int e = tid; e < a * a; e += NT) Gfull[e] = __ldcg(M.Pred + e);
    for (int e = tid; e < a * r; e += NT) Ups[e] = __ldg(M.U_prev + e);
    __syncthreads();
    if (tid < a * r) {
      const int k = tid / r, j = tid - k * r;
      double v = 0.0;
      for (int k2 = 0; k2 < a; ++k2) v = fma(Gfull[k * a + k2], (double)Ups[k2 * r + j], v);
      Pm[k][j] = v;
      M.Pg[tid] = v;
    }
    __syncthreads();
    if (tid < r * r) {
      const int i = tid / r, k = tid - i * r;
      double g = 0.0;
      if (k >= i)
        for (int kk = 0; kk < a; ++kk) g = fma(Pm[kk][i], Pm[kk][k], g);
      Gs[i][k] = g;
    }
  }
  __syncthreads();
  if (warp == 0) {
    // right-looking Cholesky G = R^T R on one warp; lane owns entries e0 = lane and e1 = lane + 32
    const int e0 = lane, e1 = lane + 32;
    const int i0 = e0 / r, k0 = e0 - i0 * r, i1 = e1 / r, k1 = e1 - i1 * r;
    const bool in0 = e0 < r * r, in1 = e1 < r * r;
    double trace = 0.0;
    for (int i = 0; i < r; ++i) trace += Gs[i][i];
    const double floor_d = 1e-12 * trace;
    for (int j = 0; j < r; ++j) {
      double d = Gs[j][j];
      if (!(d > floor_d)) {
        if (lane == 0) atomicMax(args.status, (int)ASI_ERR_RANK_DEFICIENT);
        d = (floor_d > 0.0) ? floor_d : 1.0;
      }
      const double inv = rsqrt(d);
      __syncwarp();
      if (lane == j) {
        Gs[j][j] = d * inv;
        Dinv[j] = inv;
      } else if (lane > j && lane < r) {
        Gs[j][lane] *= inv;
      }
      __syncwarp();
      if (in0 && i0 > j && k0 >= i0) Gs[i0][k0] -= Gs[j][i0] * Gs[j][k0];
      if (in1 && i1 > j && k1 >= i1) Gs[i1][k1] -= Gs[j][i1] * Gs[j][k1];
      __syncwarp();
    }
    double* Rf = args.Rf + mode * kRfStride;
    if (in0) Rf[i0 * RM + k0] = Gs[i0][k0];
    if (in1) Rf[i1 * RM + k1] = Gs[i1][k1];
    if (lane < r) Rf[RM * RM + lane] = Dinv[lane];
    if (lane == 0) args.counter[mode] = 0;
  }
  if constexpr (!LARGE) return;
  // ---- U_m = P_m R_m^{-1}, a row per thread (a launch of its own took 3.5 us of the chain)
  __syncthreads();
  if (tid >= a) return;
  double q[RM];
#pragma unroll
  for (int j = 0; j < RM; ++j) q[j] = j < r ? __ldcg(M.Pred + (int64_t)tid * r + j) : 0.0;
#pragma unroll
  for (int j = 0; j < RM; ++j)
    if (j < r) {
#pragma unroll
      for (int i = 0; i < RM; ++i)
        if (i < j) q[j] = fma(-q[i], Gs[i][j], q[j]);
      q[j] *= Dinv[j];
      M.U[(int64_t)tid * r + j] = (float)q[j];
    }
}

__global__ void __launch_bounds__(kRedNT) k_sm_reduce(const __grid_constant__ SmReduceArgs args) {
  sm_reduce_cta<false>(args, (int)blockIdx.x, (int)blockIdx.y);
}
__global__ void __launch_bounds__(kRedNTLarge) k_sm_reduce_large(const __grid_constant__ SmReduceArgs args) {
  sm_reduce_cta<true>(args, (int)blockIdx.x, (int)blockIdx.y);
}
__global__ void __launch_bounds__(kRedNT) k_sm_reduce_b(const __grid_constant__ SmBatch<SmReduceArgs> b) {
  const int l = batch_layer(b, (int)blockIdx.x);
  sm_reduce_cta<false>(b.a[l], (int)blockIdx.x - b.first[l], (int)blockIdx.y);
}

cudaError_t launch_sm_reduce(const SmReduceArgs& p, int nd, int max_chunks, cudaStream_t st) {
  double bytes = 0.0;
  for (int m = 0; m < nd; ++m)
    bytes += 4.0 * p.m[m].nsplit * p.m[m].a * (p.m[m].gram ? p.m[m].a : p.m[m].r) + 8.0 * p.m[m].a * p.m[m].r;
  ProfScope prof(ASI_K_QR, st, bytes);
  dim3 grid((unsigned)max_chunks, (unsigned)nd);
  if (p.large) return launch_pdl(k_sm_reduce_large, grid, dim3(kRedNTLarge), 0, st, p);
  return launch_pdl(k_sm_reduce, grid, dim3(kRedNT), 0, st, p);
}

// ---------------------------------------------------------------------------------------------
// k_sm_core.  Tile = CC whole channels (at most 256 columns (c, h, w)) of all samples:
//   prologue: one thread per needed factor row fetches the fp64 row of P_m and solves u = p R_m^{-1} with the
//     Cholesky factor the reduction kernel left -- all of U_1, the tile's own rows of U_2, all of U_3 and U_4 -- and
//     the owners write them to U_new; the first samples of the tile are already on their way;
//   W[c,h,w][i] = sum_b U1[b,i] X[b][c,h,w] straight from memory in registers (the activation is in L2 or streams
//     from HBM; nothing is staged, so several CTAs share an SM), or, in launches of few CTAs, from a tile in shared
//     memory (choose_core);
//   M[c][i,k,l] = W x_3 U3^T x_4 U4^T per channel -- the spatial modes before the channel mode: r1 r3 (W + r4) short
//     sums per channel instead of r1 r2 HW, and r1 r3 r4 numbers leave a channel instead of a whole core;
//   core[i,j,k,l] = sum_c U2[c,j] M[c][i,k,l] by the last CTA of every group of tiles, then over the groups by the last
//     group, both in index order.
// ---------------------------------------------------------------------------------------------
// ---- A tile [B x J] (J a multiple of four) whole in shared memory: k_sm_core and k_sm_wgrad where a launch has few CTAs.
// Every value is requested before there is anything to wait for, by 512 threads; the streamed forms of the same sums
// hold eight samples a thread, so that four CTAs share an SM.  The bits are the same: sample b goes to share b mod NH, and
// the shares meet in order.
template <typename TX>
__host__ __device__ constexpr int tile_pitch(int J) { return sizeof(TX) == 4 ? J + 4 : J + 8; }   // rows stay 16 (bf16: 8) byte aligned
template <typename TX>
__host__ __device__ constexpr size_t tile_floats(int B, int J) { return ((size_t)B * tile_pitch<TX>(J) * sizeof(TX) + 3) / 4; }
template <typename TX>
__device__ __forceinline__ void tile_issue(const TX* __restrict__ A, int64_t sstride, int B, int J, int jvalid, TX* __restrict__ Xs) {
  const int JV = J / 4, PJ = tile_pitch<TX>(J);
  const FDiv dJ(JV);
  int b, q, sb, sq;
  dJ.divmod((int)threadIdx.x, b, q);
  dJ.divmod(kTT, sb, sq);
  while (b < B) {
    if (4 * q < jvalid) {
      const TX* src = A + (int64_t)b * sstride + 4 * q;
      if constexpr (sizeof(TX) == 4)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(Xs + b * PJ + 4 * q)), "l"(src) : "memory");
      else
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(smem_u32(Xs + b * PJ + 4 * q)), "l"(src) : "memory");
    }
    b += sb;
    q += sq;
    if (q >= JV) { q -= JV; ++b; }
  }
}
// acc[c][j / 2] = sum over the samples b == h (mod NH) of X[b][4 jq + c] (U1[b][j], U1[b][j + 1])
template <int R, typename TX>
__device__ __forceinline__ void tile_project(const TX* Xs, int B, int PJ, int NH, int h, int jq, const float* __restrict__ U1s,
                                             f2 (&acc)[4][R / 2]) {
#pragma unroll
  for (int c = 0; c < 4; ++c)
#pragma unroll
    for (int j = 0; j < R / 2; ++j) acc[c][j] = 0ull;
  const TX* src = Xs + 4 * jq;
#pragma unroll 4
  for (int b = h; b < B; b += NH) {
    const float4 x = ld4<TX>(src + b * PJ);
    const float xs[4] = {x.x, x.y, x.z, x.w};
    const float* u = U1s + b * R;
#pragma unroll
    for (int j = 0; j < R / 2; j += 2) {
      const ulonglong2 uj = *reinterpret_cast<const ulonglong2*>(u + 2 * j);
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const f2 xc = pack2(xs[c], xs[c]);
        ffma2(acc[c][j], xc, uj.x);
        ffma2(acc[c][j + 1], xc, uj.y);
      }
    }
  }
}

// W[col][:] = sum_b X[b][col] U1[b][:] for the tile's J columns (jvalid of them exist): thread = VW neighbouring columns
// and the samples b == h (mod NH), eight in flight, the NH shares meet in order.  The first eight are requested before
// `factors` (the row solves, which end with a barrier) runs.  Shares are stored by rank, columns side by side: stored by
// column they cost four times the shared-memory cycles (ResNet-18 tail at 64: 26.6 -> 24.5 us).
template <int R, int VW, typename TX, typename F>
__device__ __forceinline__ void core_project(const TX* __restrict__ A, int64_t chw, int B, int J, int jvalid,
                                             const float* __restrict__ U1s, float* __restrict__ part, float* __restrict__ Ws,
                                             F&& factors) {
  constexpr int U = 8;
  const int tid = threadIdx.x;
  const int JV = (J + VW - 1) / VW, NH = kPT / JV;
  const FDiv dJ(JV);
  int h, jq;
  dJ.divmod(tid, h, jq);
  const bool on = h < NH && jq * VW < jvalid;
  const TX* src = A + (on ? jq * VW : 0);
  f2 acc[VW][R / 2];                                 // pairs of ranks
#pragma unroll
  for (int c = 0; c < VW; ++c)
#pragma unroll
    for (int j = 0; j < R / 2; ++j) acc[c][j] = 0ull;
  const int nb = on && B > h ? (B - h + NH - 1) / NH : 0;   // samples of this thread
  if (!on) h = 0;
  src += (int64_t)h * chw;
  const int64_t step = (int64_t)NH * chw;
  bool first = true;
#pragma unroll 1
  for (int t0 = 0; t0 < nb || first; t0 += U) {
    RawCol<TX, VW> x[U];
#pragma unroll
    for (int t = 0; t < U; ++t) x[t].load(src + (int64_t)(t0 + t < nb ? t0 + t : 0) * step);
    if (first) {                                     // uniform: every thread's first batch
      factors();
      first = false;
    }
#pragma unroll
    for (int t = 0; t < U; ++t)
      if (t0 + t < nb) {
        float xs[VW];
        x[t].get(xs);
        const float* u = U1s + (h + (t0 + t) * NH) * R;
#pragma unroll
        for (int j = 0; j < R / 2; j += 2) {
          const ulonglong2 uj = *reinterpret_cast<const ulonglong2*>(u + 2 * j);
#pragma unroll
          for (int c = 0; c < VW; ++c) {
            const f2 xc = pack2(xs[c], xs[c]);
            ffma2(acc[c][j], xc, uj.x);
            ffma2(acc[c][j + 1], xc, uj.y);
          }
        }
      }
  }
  if (on) {
    float* dst = part + h * J * R + jq * VW;         // [h][j][J]: neighbours write neighbouring quads
#pragma unroll
    for (int j = 0; j < R; j += 2) {
      float2 v[VW];
#pragma unroll
      for (int c = 0; c < VW; ++c) v[c] = unpack2(acc[c][j / 2]);
      if constexpr (VW == 4) {
        *reinterpret_cast<float4*>(dst + j * J) = make_float4(v[0].x, v[1].x, v[2].x, v[3].x);
        *reinterpret_cast<float4*>(dst + (j + 1) * J) = make_float4(v[0].y, v[1].y, v[2].y, v[3].y);
      } else {
        dst[j * J] = v[0].x;
        dst[(j + 1) * J] = v[0].y;
      }
    }
  }
  __syncthreads();
  for (int idx = tid; idx < J * R; idx += kPT) {
    float s = part[idx];
#pragma unroll 4
    for (int q = 1; q < NH; ++q) s += part[q * J * R + idx];
    Ws[idx] = s;
  }
  __syncthreads();
}

template <int R, typename TX>
__device__ __forceinline__ void core_project_staged(const TX* Xs, int B, int J, int jvalid, const float* __restrict__ U1s,
                                                    float* part, float* __restrict__ Ws) {
  const int tid = threadIdx.x, JV = J / 4, NH = kPT / JV;
  const FDiv dJ(JV);
  int h, jq;
  dJ.divmod(tid, h, jq);
  const bool on = h < NH && 4 * jq < jvalid;
  f2 acc[4][R / 2];
  if (on) tile_project<R>(Xs, B, tile_pitch<TX>(J), NH, h, jq, U1s, acc);
  __syncthreads();                                   // the tile has been read: the shares go over it
  if (on) {
    float* dst = part + h * J * R + 4 * jq;
#pragma unroll
    for (int j = 0; j < R; j += 2) {
      float2 v[4];
#pragma unroll
      for (int c = 0; c < 4; ++c) v[c] = unpack2(acc[c][j / 2]);
      *reinterpret_cast<float4*>(dst + j * J) = make_float4(v[0].x, v[1].x, v[2].x, v[3].x);
      *reinterpret_cast<float4*>(dst + (j + 1) * J) = make_float4(v[0].y, v[1].y, v[2].y, v[3].y);
    }
  }
  __syncthreads();
  for (int idx = tid; idx < J * R; idx += kTT) {
    float s = part[idx];
#pragma unroll 4
    for (int q = 1; q < NH; ++q) s += part[q * J * R + idx];
    Ws[idx] = s;
  }
  __syncthreads();
}

template <int R, bool STAGED, typename TX>
__device__ __forceinline__ void sm_core_cta(const SmCoreArgs& p, const int bid) {
  constexpr int NT = STAGED ? kTT : kPT;
  extern __shared__ __align__(128) float smem[];
  __shared__ int s_last;
  __shared__ double Rs[4][kRfStride];   // per mode: rows of R_m (pitch 8), then 1 / diag(R_m) at [64..]
  const int tid = threadIdx.x;
  const int B = p.B, C = p.C, H = p.H, W = p.W, HW = H * W, CC = p.tile_c, J = CC * HW, tile = bid;
  const int r1 = p.r[0], r2 = p.r[1], r3 = p.r[2], r4 = p.r[3];
  const int c0 = tile * CC, ncl = (C - c0 < CC) ? C - c0 : CC, jvalid = ncl * HW;
  float* U1s = smem;                    // [B][R]
  float* U3s = U1s + ((B * R + 3) & ~3);   // [H][R]
  float* U4s = U3s + H * R;             // [W][R]
  float* Ws = U4s + W * R;              // [R][J]
  float* part = Ws + J * R;             // [NH][R][J], at most 256 * 4 R
  float* T1 = part;                     // [ncl r1][r3][W] after part is free
  auto factors = [&]() {
    pdl_wait();                         // P_m and the Cholesky factors come from the reduction kernel
    // factor rows: [U1: B rows][the tile's rows of U2][U3: H][U4: W]
    const int nrows = B + ncl + H + W;
    bool synced = false;
#pragma unroll 1
    for (int row = tid; row < nrows || !synced; row += NT) {
      int m = 0, k = row;
      float* rdst = U1s + k * R;
      bool owner = tile == 0;
      if (row >= B + ncl + H) { m = 3; k = row - B - ncl - H; rdst = U4s + k * R; }
      else if (row >= B + ncl) { m = 2; k = row - B - ncl; rdst = U3s + k * R; }
      else if (row >= B) { m = 1; k = c0 + row - B; rdst = nullptr; owner = true; }
      const int rr = p.r[m];
      const bool on = row < nrows;
      double q[R];
#pragma unroll
      for (int j = 0; j < R; ++j) q[j] = (on && j < rr) ? __ldcg(p.Pred[m] + (int64_t)k * rr + j) : 0.0;
      if (!synced) {                    // the Cholesky factors of the four modes travel with the first rows
        for (int e = tid; e < 4 * kRfStride; e += NT) (&Rs[0][0])[e] = __ldcg(p.Rf + e);
        __syncthreads();
        synced = true;
      }
      if (!on) break;
      float* gdst = p.U_new + p.u_off[m] + (int64_t)k * rr;
#pragma unroll
      for (int j = 0; j < R; ++j) {
        float out = 0.f;
        if (j < rr) {
#pragma unroll
          for (int i = 0; i < R; ++i)
            if (i < j) q[j] = fma(-q[i], Rs[m][i * 8 + j], q[j]);
          q[j] *= Rs[m][64 + j];
          out = (float)q[j];
          if (owner) gdst[j] = out;
        }
        if (rdst) rdst[j] = out;
      }
    }
    __syncthreads();
  };
  const TX* A = reinterpret_cast<const TX*>(p.act) + (int64_t)c0 * HW;
  const int64_t chw = (int64_t)C * HW;
  if constexpr (STAGED) {
    TX* Xs = reinterpret_cast<TX*>(part);
    tile_issue(A, chw, B, J, jvalid, Xs);
    factors();
    fac_wait();
    __syncthreads();
    core_project_staged<R>(Xs, B, J, jvalid, U1s, part, Ws);
  } else if (p.vec4) core_project<R, 4, TX>(A, chw, B, J, jvalid, U1s, part, Ws, factors);
  else core_project<R, 1, TX>(A, chw, B, J, jvalid, U1s, part, Ws, factors);
  // T1[cl,i][k][w] = sum_h W[cl,h,w][i] U3[h][k]
  const FDiv dW(W), d_r1(r1), d_r3(r3), d_r4(r4);
  for (int idx = tid; idx < ncl * r1 * r3 * W; idx += NT) {
    int t, w, ci, k, cl, i;
    dW.divmod(idx, t, w);
    d_r3.divmod(t, ci, k);
    d_r1.divmod(ci, cl, i);
    const float* ws = Ws + i * J + cl * HW + w;
    float s = 0.f;
#pragma unroll 4
    for (int h = 0; h < H; ++h) s = fmaf(ws[h * W], U3s[h * R + k], s);
    T1[idx] = s;
  }
  __syncthreads();
  // M[c][i,k,l] = sum_w T1[cl,i][k][w] U4[w][l]
  const int ce3 = r1 * r3 * r4;
  for (int idx = tid; idx < ncl * ce3; idx += NT) {
    int t, l;
    d_r4.divmod(idx, t, l);
    const float* ts = T1 + t * W;
    float s = 0.f;
#pragma unroll 4
    for (int w = 0; w < W; ++w) s = fmaf(ts[w], U4s[w * R + l], s);
    p.Tp[(int64_t)c0 * ce3 + idx] = s;
  }
  // ---- groups of gs tiles, then the groups, both by the last CTA and in index order
  __threadfence();
  __syncthreads();
  const int grp = tile / p.gs, gfirst = grp * p.gs, ce = ce3 * r2;
  const int gsize = (p.n_tiles - gfirst < p.gs) ? p.n_tiles - gfirst : p.gs;
  const int ngroups = (p.n_tiles + p.gs - 1) / p.gs;
  if (tid == 0) s_last = (atomicAdd(p.gcount + grp, 1) == gsize - 1);
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  {
    const int ch0 = gfirst * CC, nch = ((gfirst + gsize) * CC < C ? (gfirst + gsize) * CC : C) - ch0;
    float* u2 = part;                   // [nch][R] (gs CC R floats: fits, checked by the host)
    for (int e = tid; e < nch * R; e += NT) {
      const int c = e / R, j = e % R;
      u2[e] = j < r2 ? __ldcg(p.U_new + p.u_off[1] + (int64_t)(ch0 + c) * r2 + j) : 0.f;
    }
    __syncthreads();
    // thread = one (i, k, l), all j: the channels' numbers are read once, 16 in flight
    for (int e = tid; e < ce3; e += NT) {
      float s[R];
#pragma unroll
      for (int j = 0; j < R; ++j) s[j] = 0.f;
      const float* src = p.Tp + (int64_t)ch0 * ce3 + e;
#pragma unroll 1
      for (int c = 0; c < nch; c += 16) {
        float v[16];
#pragma unroll
        for (int q = 0; q < 16; ++q) v[q] = __ldcg(src + (int64_t)(c + q < nch ? c + q : c) * ce3);
#pragma unroll
        for (int q = 0; q < 16; ++q)
          if (c + q < nch) fma_row<R>(s, v[q], u2 + (c + q) * R);
      }
      const int i = e / (r3 * r4), kl = e - i * (r3 * r4);
      float* dst = p.Tg + (int64_t)grp * ce + (int64_t)i * r2 * r3 * r4 + kl;
#pragma unroll
      for (int j = 0; j < R; ++j)
        if (j < r2) dst[j * r3 * r4] = s[j];
    }
  }
  __threadfence();
  __syncthreads();
  if (tid == 0) {
    p.gcount[grp] = 0;
    s_last = (atomicAdd(p.counter, 1) == ngroups - 1);
  }
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  // few core elements: thread (e, q) sums the groups == q (mod nq) of element e, the nq sums meet in index order
  if (ce > kPT && ngroups <= 8) {       // a wide core from few groups: four elements x eight groups in flight
#pragma unroll 1
    for (int e0 = tid; e0 < ce; e0 += 4 * NT) {
      float v[4][8];
#pragma unroll
      for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int k = 0; k < 8; ++k)
          v[u][k] = __ldcg(p.Tg + (int64_t)(k < ngroups ? k : 0) * ce + (e0 + u * NT < ce ? e0 + u * NT : e0));
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        float s = v[u][0];
#pragma unroll
        for (int k = 1; k < 8; ++k) s += k < ngroups ? v[u][k] : 0.f;
        if (e0 + u * NT < ce) p.core[e0 + u * NT] = s;
      }
    }
    if (tid == 0) *p.counter = 0;
    return;
  }
  int nq = kPT / ce;                   // (the order of these sums does not depend on NT)
  nq = nq > 8 ? 8 : (nq < 1 ? 1 : nq);
  float* fold = part;                   // [nq][ce]
  for (int it = tid; it < nq * ce; it += NT) {
    const int q = it / ce, e = it - q * ce;
    const float* src = p.Tg + e;
    float s = 0.f;
#pragma unroll 1
    for (int g0 = q; g0 < ngroups; g0 += 16 * nq) {
      float v[16];
#pragma unroll
      for (int k = 0; k < 16; ++k) v[k] = __ldcg(src + (int64_t)(g0 + k * nq < ngroups ? g0 + k * nq : g0) * ce);
#pragma unroll
      for (int k = 0; k < 16; ++k) s += (g0 + k * nq < ngroups) ? v[k] : 0.f;
    }
    if (nq > 1) fold[it] = s;
    else p.core[e] = s;
  }
  if (nq > 1) {
    __syncthreads();
    if (tid < ce) {
      float s = fold[tid];
      for (int q = 1; q < nq; ++q) s += fold[q * ce + tid];
      p.core[tid] = s;
    }
  }
  if (tid == 0) *p.counter = 0;
}

template <int R, typename TX>
__global__ void __launch_bounds__(kPT, R == 4 ? 4 : 3) k_sm_core(const __grid_constant__ SmCoreArgs p) {
  sm_core_cta<R, false, TX>(p, (int)blockIdx.x);
}
template <int R, typename TX>
__global__ void __launch_bounds__(kPT, R == 4 ? 4 : 3) k_sm_core_b(const __grid_constant__ SmBatch<SmCoreArgs> b) {
  const int l = batch_layer(b, (int)blockIdx.x);
  sm_core_cta<R, false, TX>(b.a[l], (int)blockIdx.x - b.first[l]);
}
template <int R, typename TX>
__global__ void __launch_bounds__(kTT, 2) k_sm_core_staged(const __grid_constant__ SmCoreArgs p) {
  sm_core_cta<R, true, TX>(p, (int)blockIdx.x);
}
template <int R, typename TX>
__global__ void __launch_bounds__(kTT, 2) k_sm_core_staged_b(const __grid_constant__ SmBatch<SmCoreArgs> b) {
  const int l = batch_layer(b, (int)blockIdx.x);
  sm_core_cta<R, true, TX>(b.a[l], (int)blockIdx.x - b.first[l]);
}

// ---------------------------------------------------------------------------------------------
// k_sm_wgrad: CTA owns cpb consecutive output channels, i.e. the dY tile [B x J], J = cpb*Ho*Wo
// contiguous values per sample.
//   Z1 = dY x_1 U1^T on the CTA's channels, straight from memory in registers (no staged tile: 100 KB less shared
//     memory, so two CTAs share an SM and the set-up of one hides behind the stream of the other), or, in launches of at
//     most a CTA an SM, from a staged tile with Z3 formed while it is on its way (wgrad_staged);
//   Z3 = core x_3 U3 x_4 U4 (recomputed per CTA);
//   Z4[c',j,kh,kw] = sum_{i,h',w'} Z1[i,c',h',w'] Z3pad[i,j,h's+kh-p,w's+kw-p];  dW = Z4 x_2 U2.
// ---------------------------------------------------------------------------------------------
// Term 5: dW[c0+cl, c, t] = sum_j Z4[cl][t][j] U2[(g cg + c), j].  The rows of Z4 are the same for every
// thread, so each 16-byte shared-memory read of one costs a full warp-wide transfer; a thread therefore
// owns up to four input channels (their rows of U2 stay in registers) and every row of Z4 it reads feeds
// four dot products (fewer, busier threads: the shared-memory pipe is the limit).  p.ncl output channels
// are expanded per round, one thread group each, into a staging block [ncl][cg x kk] in shared memory
// that then leaves for global memory in one piece per channel -- by the bulk-copy engine
// (cp.async.bulk shared -> global) when a channel's block is 16-byte sized and aligned, else by
// coalesced stores.  With more than one round there are two staging blocks, so that a round's stores
// run under the next round's arithmetic: the write of dW by all CTAs at once is DRAM-bound.
template <int R, int kNT>
__device__ __forceinline__ void wgrad_expand_rows(const SmWgradArgs& p, const float* __restrict__ Z4s,
                                                  const float* __restrict__ U2s, float* stage, int c0) {
  const int kk = p.kh * p.kw;
  const int cg = p.C / p.groups, og = p.Cout / p.groups;
  const int tid = threadIdx.x;
  const int nblk = cg * kk;
  const int lg = (p.ncl == 4) ? 2 : (p.ncl == 2 ? 1 : 0);
  const int TG = kNT >> lg;                          // threads per output channel
  const int grp = tid / TG, tg = tid - grp * TG;
  int ta = (((cg + 3) >> 2) + 31) & ~31;             // active threads of a group: four channels each
  if (ta > TG) ta = TG;
  const int rounds = p.cpb / p.ncl;
#pragma unroll 1
  for (int rd = 0; rd < rounds; ++rd) {
    const int cl = rd * p.ncl + grp;
    const int co = c0 + cl;
    const int g = co / og;
    float* dw = p.dW + (int64_t)(c0 + rd * p.ncl) * nblk;
    const float* u2 = U2s + (int64_t)g * cg * R;
    float* buf = stage + (p.nbuf == 2 ? (rd & 1) : 0) * p.ncl * nblk;
    if (rd >= p.nbuf) {                              // the block's last round has left it
      if (p.bulk_store && tid == 0) {
        if (p.nbuf == 2) asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");
        else asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
      }
      __syncthreads();
    }
    float* out = buf + grp * nblk;
    const float* z = Z4s + cl * kk * R;
#pragma unroll 1
    for (int cb = tg; cb < cg && tg < ta; cb += 4 * ta) {
      float u[4][R];
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        const int c = cb + m * ta;
#pragma unroll
        for (int j = 0; j < R; j += 4) {
          float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
          if (c < cg) v = *reinterpret_cast<const float4*>(u2 + c * R + j);
          u[m][j] = v.x; u[m][j + 1] = v.y; u[m][j + 2] = v.z; u[m][j + 3] = v.w;
        }
      }
#pragma unroll 3
      for (int t = 0; t < kk; ++t) {
        float v[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int j = 0; j < R; j += 4) {
          const float4 zz = *reinterpret_cast<const float4*>(z + t * R + j);
#pragma unroll
          for (int m = 0; m < 4; ++m) {
            v[m] = fmaf(zz.x, u[m][j], v[m]);
            v[m] = fmaf(zz.y, u[m][j + 1], v[m]);
            v[m] = fmaf(zz.z, u[m][j + 2], v[m]);
            v[m] = fmaf(zz.w, u[m][j + 3], v[m]);
          }
        }
#pragma unroll
        for (int m = 0; m < 4; ++m) {
          const int c = cb + m * ta;
          if (c < cg) out[c * kk + t] = v[m];
        }
      }
    }
    if (p.bulk_store) {
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncthreads();
      if (tid == 0) {
        for (int q = 0; q < p.ncl; ++q)
          asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dw + (int64_t)q * nblk),
                       "r"(smem_u32(buf + q * nblk)), "r"((uint32_t)nblk * 4u)
                       : "memory");
        asm volatile("cp.async.bulk.commit_group;" ::: "memory");
      }
    } else {
      __syncthreads();
      for (int idx = tid; idx < p.ncl * nblk; idx += kNT) dw[idx] = buf[idx];
    }
  }
  if (p.bulk_store && tid == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
}

// groups of samples a CTA of k_sm_wgrad splits the batch over (JV column items)
__host__ __device__ inline int wgrad_groups(int JV, int nt) {
  const int n = nt / (JV < nt ? JV : nt);
  return n > 8 ? 8 : n;
}
// Z1[j][:] = sum_b dY[b][j] U1[b][:] for the CTA's J columns; thread = VW neighbouring columns and the samples
// b == h (mod NH), eight of them in flight; the NH shares meet in order.  The factors' asynchronous copies of this
// thread are waited for behind the first loads.
template <int R, int VW, int kNT, typename TX>
__device__ __forceinline__ void wgrad_project(const TX* __restrict__ dY, int64_t sstride, int B, int J, int NH,
                                              const float* __restrict__ U1s, float* __restrict__ part, float* __restrict__ Z1s) {
  constexpr int U = 8;
  const int tid = threadIdx.x, JV = (J + VW - 1) / VW;
  const FDiv dJ(JV);
  bool waited = false;
  for (int it = tid; it < NH * JV || !waited; it += kNT) {      // one round unless there are more columns than threads
    int h, jq;
    dJ.divmod(it, h, jq);
    const bool on = h < NH;
    const TX* src = dY + (on ? jq * VW : 0);
    if (!on) h = 0;
    src += (int64_t)h * sstride;
    const int nb = on && B > h ? (B - h + NH - 1) / NH : 0;     // samples of this thread
    const int64_t step = (int64_t)NH * sstride;
    float acc[VW][R];
#pragma unroll
    for (int c = 0; c < VW; ++c)
#pragma unroll
      for (int j = 0; j < R; ++j) acc[c][j] = 0.f;
#pragma unroll 1
    for (int t0 = 0; t0 < nb || !waited; t0 += U) {
      RawCol<TX, VW> x[U];
#pragma unroll
      for (int u = 0; u < U; ++u) x[u].load(src + (int64_t)(t0 + u < nb ? t0 + u : 0) * step);
      if (!waited) {
        fac_wait();
        __syncthreads();
        waited = true;
      }
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (t0 + u < nb) {
          float xs[VW];
          x[u].get(xs);
          const float* u1 = U1s + (h + (t0 + u) * NH) * R;
#pragma unroll
          for (int c = 0; c < VW; ++c) fma_row<R>(acc[c], xs[c], u1);
        }
    }
    if (on) {
      float* dst = part + (h * J + jq * VW) * R;
#pragma unroll
      for (int c = 0; c < VW; ++c)
#pragma unroll
        for (int j = 0; j < R; j += 4)
          *reinterpret_cast<float4*>(dst + c * R + j) = make_float4(acc[c][j], acc[c][j + 1], acc[c][j + 2], acc[c][j + 3]);
    }
  }
  __syncthreads();
  for (int idx = tid; idx < J * R; idx += kNT) {
    float s = part[idx];
    for (int q = 1; q < NH; ++q) s += part[q * J * R + idx];
    Z1s[idx] = s;
  }
}

template <int R, int kNT, bool STAGED, typename TX>
__device__ __forceinline__ void sm_wgrad_cta(const SmWgradArgs& p, const int bid) {
  extern __shared__ __align__(128) float smem[];
  pdl_wait();                                        // the only kernel of a call
  const int tid = threadIdx.x;
  const int r1 = p.r[0], r2 = p.r[1], r3 = p.r[2], r4 = p.r[3];
  const int H = p.H, W = p.W, HoWo = p.Ho * p.Wo, kk = p.kh * p.kw;
  const int J = p.cpb * HoWo;                        // dY columns of this CTA, contiguous per sample
  const int c0 = bid * p.cpb;
  // staging blocks of term 5 reuse the tile's space: ncl channels per round, nbuf of them when rounds follow
  const int n_stage = (p.cpb > p.ncl ? p.nbuf : 1) * p.ncl * (p.C / p.groups) * kk;
  const int nt = STAGED ? p.nt : kNT;                // the thread count that the sums are split by
  const int VW = p.vec4 ? 4 : 1, JV = (J + VW - 1) / VW, NH = wgrad_groups(JV, nt);
  const int n_tile = STAGED ? (int)tile_floats<TX>(p.B, J) : 0;
  float* stage = smem;                               // term 5's blocks; before that the shares of Z1 [NH][J][R]
  float* part = smem;                                // (and before these the tile of dY)
  int n_head = NH * J * R > n_stage ? NH * J * R : n_stage;
  if (n_tile > n_head) n_head = n_tile;
  float* U1s = smem + (n_head + 3) / 4 * 4;          // [B][R]
  float* U2s = U1s + p.B * R;                        // [C][R]
  float* Z1s = U2s + p.C * R;                        // [J][R]
  float* Ss = Z1s + J * R;                           // [r1 r2][R (l)][R (k)]: core, modes 3 and 4 swapped, zero-padded
  float* U3s = Ss + r1 * r2 * R * R;                 // [H][R]
  float* U4s = U3s + H * R;                          // [W][R]
  float* Tm = U4s + W * R;                           // [r1 r2][H][R]
  const int Hp = H + 2 * p.ph, Wp = W + 2 * p.pw;    // Z3 is kept zero-padded: term 4 needs no bounds logic
  float* Z3s = Tm + r1 * r2 * H * R;                 // [r1 r2][Hp][Wp]
  float* Z4s = smem + ((Z3s + r1 * r2 * Hp * Wp) - smem + 3) / 4 * 4;   // [cpb][kk][R], 16-byte aligned (rank index fastest, zero-padded)
  float* red = Z4s + p.cpb * kk * R;                 // [G4][cpb][r2 kk]

  const TX* dY = reinterpret_cast<const TX*>(p.dY) + (int64_t)c0 * HoWo;
  const int64_t sstride = (int64_t)p.Cout * HoWo;
  {
#pragma unroll 1
    for (int idx = tid; idx < r1 * r2 * R * R; idx += kNT) {      // Ss[ij][l][k] = core[ij][k][l]
      const int k = idx % R, l = (idx / R) % R, ij = idx / (R * R);
      const bool in = k < r3 && l < r4;
      cp_async4(Ss + idx, p.core + (in ? (ij * r3 + k) * r4 + l : 0), in ? 4 : 0);
    }
    fac_issue_padded<R, kNT>(p.U + p.u_off[2], U3s, H, r3);
    fac_issue_padded<R, kNT>(p.U + p.u_off[3], U4s, W, r4);
    fac_issue_padded<R, kNT>(p.U + p.u_off[0], U1s, p.B, r1);
    fac_issue_padded<R, kNT>(p.U + p.u_off[1], U2s, p.C, r2);
    if constexpr (STAGED) {                          // Z3 is formed while the tile is on its way
      asm volatile("cp.async.commit_group;" ::: "memory");
      tile_issue(dY, sstride, p.B, J, J, reinterpret_cast<TX*>(smem));
      asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 1;" ::: "memory");
      __syncthreads();
    } else if (p.vec4) wgrad_project<R, 4, kNT, TX>(dY, sstride, p.B, J, NH, U1s, part, Z1s);
    else wgrad_project<R, 1, kNT, TX>(dY, sstride, p.B, J, NH, U1s, part, Z1s);
  }
  // terms 2-3: Tm[ij][h][l] = sum_k S[ij][k][l] U3[h][k];  Z3[ij][h][w] = sum_l Tm[ij][h][l] U4[w][l]
  // (rank indices padded to R with zeros: every sum is a fixed-length dot product of 16-byte reads)
  const FDiv d_H(H), d_Wp(Wp), d_Hp(Hp), d_kk(kk), d_kw(p.kw);
  for (int idx = tid; idx < r1 * r2 * H * R; idx += kNT) {
    const int l = idx % R, t0 = idx / R;
    int ij, h;
    d_H.divmod(t0, ij, h);
    const float* sp = Ss + (ij * R + l) * R;
    const float* up = U3s + h * R;
    float s = 0.f;
#pragma unroll
    for (int k = 0; k < R; k += 4) {
      const float4 a = *reinterpret_cast<const float4*>(sp + k), b = *reinterpret_cast<const float4*>(up + k);
      s = fmaf(a.x, b.x, s); s = fmaf(a.y, b.y, s); s = fmaf(a.z, b.z, s); s = fmaf(a.w, b.w, s);
    }
    Tm[idx] = s;
  }
  __syncthreads();
  for (int idx = tid; idx < r1 * r2 * Hp * Wp; idx += kNT) {
    int t0, wp, ij, hp;
    d_Wp.divmod(idx, t0, wp);
    d_Hp.divmod(t0, ij, hp);
    const int h = hp - p.ph, w = wp - p.pw;
    float s = 0.f;
    if (h >= 0 && h < H && w >= 0 && w < W) {
      const float* tp = Tm + (ij * H + h) * R;
      const float* up = U4s + w * R;
#pragma unroll
      for (int l = 0; l < R; l += 4) {
        const float4 a = *reinterpret_cast<const float4*>(tp + l), b = *reinterpret_cast<const float4*>(up + l);
        s = fmaf(a.x, b.x, s); s = fmaf(a.y, b.y, s); s = fmaf(a.z, b.z, s); s = fmaf(a.w, b.w, s);
      }
    }
    Z3s[idx] = s;
  }
  if constexpr (STAGED) {
    fac_wait();
    __syncthreads();
    const FDiv dJ(JV);
    int h, jq;
    dJ.divmod(tid, h, jq);
    const bool on = h < NH;
    f2 acc[4][R / 2];
    if (on) tile_project<R>(reinterpret_cast<const TX*>(smem), p.B, tile_pitch<TX>(J), NH, h, jq, U1s, acc);
    __syncthreads();                                 // the tile has been read: the shares go over it
    if (on)
#pragma unroll
      for (int c = 0; c < 4; ++c)
#pragma unroll
        for (int j = 0; j < R; j += 4) {
          const float2 a = unpack2(acc[c][j / 2]), b = unpack2(acc[c][j / 2 + 1]);
          *reinterpret_cast<float4*>(part + (h * J + 4 * jq + c) * R + j) = make_float4(a.x, a.y, b.x, b.y);
        }
    __syncthreads();
    for (int idx = tid; idx < J * R; idx += kNT) {
      float s = part[idx];
      for (int q = 1; q < NH; ++q) s += part[q * J * R + idx];
      Z1s[idx] = s;
    }
  }
  __syncthreads();
  // term 4: thread (n, g): outputs n = (j, kh, kw) of all cpb channels and every G-th pair (i, h') of
  // the reduction; one Z3 operand feeds cpb FMAs.  The G partial sums meet in order.
  const int N4 = r2 * kk;
  int G4 = (N4 <= nt) ? nt / N4 : 1;
  if (G4 > r1 * p.Ho) G4 = r1 * p.Ho;
  const FDiv d_Ho(p.Ho), d_N4(N4);
  for (int it = tid; it < N4 * G4; it += kNT) {
    int g, n, j, tt, ky, kx;
    d_N4.divmod(it, g, n);
    d_kk.divmod(n, j, tt);
    d_kw.divmod(tt, ky, kx);
    const float* z3 = Z3s + (j * Hp + ky) * Wp + kx;
    float acc[4] = {0.f, 0.f, 0.f, 0.f};
    for (int q = g; q < r1 * p.Ho; q += G4) {
      int i, ho;
      d_Ho.divmod(q, i, ho);
      const float* z1r = Z1s + ho * p.Wo * R + i;
      const float* z3r = z3 + (i * r2 * Hp + ho * p.sh) * Wp;
#pragma unroll 7
      for (int wo = 0; wo < p.Wo; ++wo) {
        const float b = z3r[wo * p.sw];
#pragma unroll
        for (int cl = 0; cl < 4; ++cl)
          if (cl < p.cpb) acc[cl] = fmaf(z1r[(cl * HoWo + wo) * R], b, acc[cl]);
      }
    }
#pragma unroll
    for (int cl = 0; cl < 4; ++cl)
      if (cl < p.cpb) red[(g * p.cpb + cl) * N4 + n] = acc[cl];
  }
  __syncthreads();
  for (int o = tid; o < p.cpb * kk * R; o += kNT) {
    const int j = o % R, ct = o / R;                 // ct = cl*kk + t
    int cl, tt;
    d_kk.divmod(ct, cl, tt);
    float v = 0.f;
    if (j < r2)
      for (int g = 0; g < G4; ++g) v += red[(g * p.cpb + cl) * N4 + j * kk + tt];
    Z4s[o] = v;
  }
  __syncthreads();
  // term 5: dW[c0+cl, c, t] = sum_j Z4[cl][j][t] U2[(g cg + c), j]
  wgrad_expand_rows<R, kNT>(p, Z4s, U2s, stage, c0);
}

template <int R, int NT, typename TX>
__global__ void __launch_bounds__(NT, (R == 4 ? 1024 : 512) / NT) k_sm_wgrad(const __grid_constant__ SmWgradArgs p) {
  sm_wgrad_cta<R, NT, false, TX>(p, (int)blockIdx.x);
}
template <int R, int NT, typename TX>
__global__ void __launch_bounds__(NT, (R == 4 ? 1024 : 512) / NT) k_sm_wgrad_b(const __grid_constant__ SmBatch<SmWgradArgs> b) {
  const int l = batch_layer(b, (int)blockIdx.x);
  sm_wgrad_cta<R, NT, false, TX>(b.a[l], (int)blockIdx.x - b.first[l]);
}
template <int R, typename TX>
__global__ void __launch_bounds__(kTT, R == 4 ? 2 : 1) k_sm_wgrad_staged(const __grid_constant__ SmWgradArgs p) {
  sm_wgrad_cta<R, kTT, true, TX>(p, (int)blockIdx.x);
}
template <int R, typename TX>
__global__ void __launch_bounds__(kTT, R == 4 ? 2 : 1) k_sm_wgrad_staged_b(const __grid_constant__ SmBatch<SmWgradArgs> b) {
  const int l = batch_layer(b, (int)blockIdx.x);
  sm_wgrad_cta<R, kTT, true, TX>(b.a[l], (int)blockIdx.x - b.first[l]);
}

// ---------------------------------------------------------------------------------------------
// host-side launchers
// ---------------------------------------------------------------------------------------------
int sm_tile1_role_c_ctas(int S, int B) { return (S == 7) ? B : 4 * B; }

size_t sm_tile1_smem(int S, int R, int B, int C) {
  const int HW = S * S, CC = (S == 7) ? 4 : 1, J = CC * HW, PJ = pitch4(J);
  const int NH1 = batch_groups(kNG, J);
  const size_t role_b = (size_t)B * PJ + (size_t)B * R + 2 * S * R + (size_t)J * R +
                        (NH1 > 1 ? (size_t)NH1 * J * R : 0) + 24 * 32;
  const int HWC = role_c_hwc(S), PC = role_c_pitch(S);
  const int G = kTT / HWC;
  const size_t vp = (C >= (G - 1) * HWC) ? 0 : (size_t)(G - 1) * HWC * R;
  const size_t role_c = (size_t)((C * PC + 3) & ~3) + (size_t)C * R + (size_t)HWC * R + vp;
  return 4 * (role_b > role_c ? role_b : role_c);
}

int sm_pass1_pitch(int HW) { return HW % 4 == 0 && (HW / 4) % 2 == 0 ? HW + 4 : HW; }

// CTAs per sample (they share a cluster) and channels per CTA: about 48 KB of the sample each, so that four CTAs share
// an SM; a CTA of a few KB pays more for its set-up and reductions than for its share (a 160-channel 7 x 7 layer split
// over four was slower than whole), but a small batch is spread over at least one CTA per SM
void sm_pass1_split(int HW, int C, int B, int* cs, int* cc) {
  int n = 1;
  auto per = [&](int k) { return ((C + k - 1) / k + 3) / 4 * 4; };
  while (n < 8 && ((size_t)per(n) * sm_pass1_pitch(HW) * 4 > 50 * 1024 || (B * n < 148 && per(n) >= 16))) n *= 2;
  *cs = n;
  *cc = per(n);
}
int sm_pass1_off_u2(int R, int cc, int pitch) {
  const int tile = (cc * pitch + 3) & ~3, red = 4 * kPT * R;
  return tile > red ? tile : red;
}

size_t sm_pass1_smem(const SmPass1Args& p, int kind, int R) {
  const int HW = p.H * p.W, JT = p.vec4 ? 128 : 32;
  const size_t role_b = (size_t)2 * p.B * R + (size_t)9 * JT * R;
  const size_t role_c = (size_t)p.off_u2 + (size_t)p.cc * R + (size_t)2 * HW * R + (size_t)(kPT / HW) * HW * R +
                        (kind == 0 ? (size_t)(p.H + p.W + 3 * 8 * 32) * R : 0);
  return 4 * (role_b > role_c ? role_b : role_c);
}
int sm_pass1_tiles_b(int64_t chw, bool vec4) { return (int)((chw + (vec4 ? 127 : 31)) / (vec4 ? 128 : 32)); }

// channels per tile of k_sm_core: as many as 256 columns hold, a multiple of four where that makes the tile's base
// 16-byte aligned
int sm_core_tile_c(int HW, int C) {
  int cc = 256 / HW;
  if (HW % 4 != 0 && cc >= 4) cc = cc / 4 * 4;
  return cc < C ? cc : C;
}
size_t sm_core_smem(const SmCoreArgs& p, int R, bool bf16) {
  const int HW = p.H * p.W, J = p.tile_c * HW, VW = p.vec4 ? 4 : 1, JV = (J + VW - 1) / VW;
  size_t part = (size_t)(kPT / JV) * J * R;
  const size_t t1 = (size_t)p.tile_c * p.r[0] * p.r[2] * p.W, u2 = (size_t)p.gs * p.tile_c * R;
  const size_t tile = p.staged ? (bf16 ? tile_floats<__nv_bfloat16>(p.B, J) : tile_floats<float>(p.B, J)) : 0;
  if (t1 > part) part = t1;
  if (u2 > part) part = u2;
  if (tile > part) part = tile;
  if (part < 8 * kPT) part = 8 * kPT;                // the final fold
  return 4 * ((size_t)((p.B * R + 3) & ~3) + (size_t)(p.H + p.W) * R + (size_t)J * R + part);
}

size_t sm_wgrad_smem(const SmWgradArgs& p, int R, bool staged, bool bf16) {
  const int r1 = p.r[0], r2 = p.r[1];
  const int J = p.cpb * p.Ho * p.Wo, kk = p.kh * p.kw, JV = p.vec4 ? J / 4 : J;
  const int N4 = r2 * kk;
  const size_t part = (size_t)wgrad_groups(JV, p.nt) * J * R,
               stage = (size_t)(p.cpb > p.ncl ? p.nbuf : 1) * p.ncl * (p.C / p.groups) * kk;
  const size_t tile = staged ? (bf16 ? tile_floats<__nv_bfloat16>(p.B, J) : tile_floats<float>(p.B, J)) : 0;
  size_t head = part > stage ? part : stage;
  if (tile > head) head = tile;
  size_t n = (head + 3) / 4 * 4 + (size_t)p.B * R + (size_t)p.C * R + (size_t)J * R +
             (size_t)r1 * r2 * R * R + (size_t)p.H * R + (size_t)p.W * R +
             (size_t)r1 * r2 * p.H * R + ((size_t)r1 * r2 * (p.H + 2 * p.ph) * (p.W + 2 * p.pw) + 3) / 4 * 4 +
             (size_t)p.cpb * kk * R + (size_t)p.cpb * (N4 > p.nt ? N4 : p.nt);
  return 4 * n + 64;
}

// a launch in clusters of cs CTAs
template <typename Arg>
static cudaError_t launch_clustered(void (*kernel)(Arg), int grid, int cs, size_t smem, cudaStream_t st, const Arg& arg) {
  cudaError_t e = opt_in_smem(reinterpret_cast<const void*>(kernel), smem);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3(kPT);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  at[1].id = cudaLaunchAttributeClusterDimension;
  at[1].val.clusterDim.x = (unsigned)cs;
  at[1].val.clusterDim.y = 1;
  at[1].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = cs > 1 ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, kernel, arg);
}
static int pass1_grid(const SmPass1Args& p) {
  return (p.B * p.cs + p.cl - 1) / p.cl * p.cl + (p.n_tiles_b + p.cl - 1) / p.cl * p.cl;
}

template <int KIND, int R, typename TX>
static cudaError_t launch_pass1_t(const SmPass1Args& p, size_t smem, cudaStream_t st) {
  return launch_clustered(p.aligned || !p.vec4 ? k_sm_pass1<KIND, R, false, TX> : k_sm_pass1<KIND, R, true, TX>, pass1_grid(p),
                          p.cl, smem, st, p);
}
// Which form a launch takes, by what it and the fused launches of the same call beside it (`beside` CTAs) bring to the
// machine; results do not depend on it.  The staged forms need whole groups of four.
//
// Core: staged up to 296 CTAs (two an SM: one wave), and where a thread of the streamed form takes more than two rounds
// of eight samples, each a round trip to memory.  One layer's step, streamed / staged: 64 x 512 x 7 x 7 (128 CTAs, two
// rounds) 40.4 / 38.8 us, 128 x 960 x 7 x 7 (240, four) 63.9 / 57.7, 128 x 256 x 14 x 14 (256, four) 80.5 / 74.1; five
// layers of 7 x 7 at 128 in a launch (840, four) 169.4 / 165.1; but the ResNet-18 tail at 64 (640 side by side, two rounds)
// 91.0 / 95.2.  Up to 113 KB, two CTAs an SM (up to 208 KB: no difference on these).
// All layers of a launch take one form.
static void choose_core(SmCoreArgs* a, int n, int R, bool bf16, int beside) {
  int ctas = beside, rounds = 0;
  bool ok = true;
  for (int l = 0; l < n; ++l) {
    SmCoreArgs& p = a[l];
    p.staged = 1;
    ok = ok && p.vec4 && sm_core_smem(p, R, bf16) <= 113 * 1024;
    if (!ok) break;
    ctas += p.n_tiles;
    const int per = 8 * (kPT / (p.tile_c * p.H * p.W / 4)), rd = (p.B + per - 1) / per;
    if (rd > rounds) rounds = rd;
  }
  ok = ok && (ctas <= 296 || rounds > 2);
  for (int l = 0; l < n; ++l) a[l].staged = ok ? 1 : 0;
}
// Weight gradient: staged up to one CTA an SM, where nothing else hides the stream of dY (64 x 512 x 7 x 7 layer, 128
// CTAs, one layer's step: 38.8 / 37.5 us; 128 x 256 x 14 x 14 with stride two, 128 CTAs: 67.7 / 62.9; but 256 CTAs at 128 x
// 14 x 14 74.1 / 75.0, and five layers at once 165 / 184).
static bool wgrad_staged(const SmWgradArgs* a, int n, int R, bool bf16, int beside) {
  int ctas = beside;
  for (int l = 0; l < n; ++l) {
    if (!a[l].vec4 || a[l].cpb * a[l].Ho * a[l].Wo / 4 > kTT || sm_wgrad_smem(a[l], R, true, bf16) > 208 * 1024) return false;
    ctas += a[l].Cout / a[l].cpb;
  }
  return ctas <= 148;
}

template <int R, typename TX>
static cudaError_t launch_core_t(const SmCoreArgs& p, size_t smem, cudaStream_t st) {
  auto kernel = p.staged ? k_sm_core_staged<R, TX> : k_sm_core<R, TX>;
  cudaError_t e = opt_in_smem(reinterpret_cast<const void*>(kernel), smem);
  if (e != cudaSuccess) return e;
  return launch_pdl(kernel, dim3(p.n_tiles), dim3(p.staged ? kTT : kPT), smem, st, p);
}

template <int R, typename TX>
static cudaError_t launch_wgrad_t(const SmWgradArgs& p, int beside, cudaStream_t st) {
  const bool bf16 = sizeof(TX) == 2, staged = wgrad_staged(&p, 1, R, bf16, beside);
  const size_t smem = sm_wgrad_smem(p, R, staged, bf16);
  auto kernel = staged ? k_sm_wgrad_staged<R, TX> : (p.nt == 512 ? k_sm_wgrad<R, 512, TX> : k_sm_wgrad<R, 256, TX>);
  cudaError_t e = opt_in_smem(reinterpret_cast<const void*>(kernel), smem);
  if (e != cudaSuccess) return e;
  return launch_pdl(kernel, dim3(p.Cout / p.cpb), dim3(staged ? kTT : p.nt), smem, st, p);
}

template <int S, int R, typename TX>
static cudaError_t launch_tile1_t(const SmTile1Args& p, cudaStream_t st) {
  const size_t smem = sm_tile1_smem(S, R, p.B, p.C);
  auto kernel = p.aligned ? k_sm_tile1<S, R, false, TX> : k_sm_tile1<S, R, true, TX>;
  cudaError_t e = opt_in_smem(reinterpret_cast<const void*>(kernel), smem);
  if (e != cudaSuccess) return e;
  return launch_pdl(kernel, dim3(p.n_tiles_b + sm_tile1_role_c_ctas(S, p.B)), dim3(kTT), smem, st, p);
}
template <int S, int R, typename TX>
static cudaError_t launch_tile1_bt(const SmBatch<SmTile1Args>& b, size_t smem, cudaStream_t st) {
  cudaError_t e = opt_in_smem(reinterpret_cast<const void*>(k_sm_tile1_b<S, R, TX>), smem);
  if (e != cudaSuccess) return e;
  return launch_pdl(k_sm_tile1_b<S, R, TX>, dim3(b.first[b.n]), dim3(kTT), smem, st, b);
}

// FN<kind, R, TX> and FN<R, TX> for the plan's variant
#define ASI_DISPATCH_KR(FN, ...)                                                                         \
  do {                                                                                                   \
    if (kind == 7) {                                                                                     \
      if (R == 4) return bf16 ? FN<7, 4, __nv_bfloat16>(__VA_ARGS__) : FN<7, 4, float>(__VA_ARGS__);     \
      return bf16 ? FN<7, 8, __nv_bfloat16>(__VA_ARGS__) : FN<7, 8, float>(__VA_ARGS__);                 \
    }                                                                                                    \
    if (kind == 14) {                                                                                    \
      if (R == 4) return bf16 ? FN<14, 4, __nv_bfloat16>(__VA_ARGS__) : FN<14, 4, float>(__VA_ARGS__);   \
      return bf16 ? FN<14, 8, __nv_bfloat16>(__VA_ARGS__) : FN<14, 8, float>(__VA_ARGS__);               \
    }                                                                                                    \
    if (R == 4) return bf16 ? FN<0, 4, __nv_bfloat16>(__VA_ARGS__) : FN<0, 4, float>(__VA_ARGS__);       \
    return bf16 ? FN<0, 8, __nv_bfloat16>(__VA_ARGS__) : FN<0, 8, float>(__VA_ARGS__);                   \
  } while (0)
#define ASI_DISPATCH_R(FN, ...)                                                                          \
  do {                                                                                                   \
    if (R == 4) return bf16 ? FN<4, __nv_bfloat16>(__VA_ARGS__) : FN<4, float>(__VA_ARGS__);             \
    return bf16 ? FN<8, __nv_bfloat16>(__VA_ARGS__) : FN<8, float>(__VA_ARGS__);                         \
  } while (0)

#define ASI_DISPATCH_SR(FN, ...)                                                                         \
  do {                                                                                                   \
    if (S == 7) {                                                                                        \
      if (R == 4) return bf16 ? FN<7, 4, __nv_bfloat16>(__VA_ARGS__) : FN<7, 4, float>(__VA_ARGS__);     \
      return bf16 ? FN<7, 8, __nv_bfloat16>(__VA_ARGS__) : FN<7, 8, float>(__VA_ARGS__);                 \
    }                                                                                                    \
    if (S == 14) {                                                                                       \
      if (R == 4) return bf16 ? FN<14, 4, __nv_bfloat16>(__VA_ARGS__) : FN<14, 4, float>(__VA_ARGS__);   \
      return bf16 ? FN<14, 8, __nv_bfloat16>(__VA_ARGS__) : FN<14, 8, float>(__VA_ARGS__);               \
    }                                                                                                    \
    if (R == 4) return bf16 ? FN<16, 4, __nv_bfloat16>(__VA_ARGS__) : FN<16, 4, float>(__VA_ARGS__);     \
    return bf16 ? FN<16, 8, __nv_bfloat16>(__VA_ARGS__) : FN<16, 8, float>(__VA_ARGS__);                 \
  } while (0)

cudaError_t launch_sm_tile1(const SmTile1Args& p, int S, int R, bool bf16, cudaStream_t st) {
  ProfScope prof(ASI_K_SM_PASS1, st, (double)p.B * p.C * S * S * (bf16 ? 2 : 4));      // the activation, read once
  ASI_DISPATCH_SR(launch_tile1_t, p, st);
}

cudaError_t launch_sm_pass1(const SmPass1Args& p, int kind, int R, bool bf16, cudaStream_t st) {
  const size_t eb = bf16 ? 2 : 4;
  const double bytes = (double)p.B * p.C * p.H * p.W * eb;      // the activation, read once
  ProfScope prof(ASI_K_SM_PASS1, st, bytes);
  ASI_DISPATCH_KR(launch_pass1_t, p, sm_pass1_smem(p, kind, R), st);
}

cudaError_t launch_sm_core(const SmCoreArgs& p0, int R, bool bf16, int beside, cudaStream_t st) {
  SmCoreArgs p = p0;
  choose_core(&p, 1, R, bf16, beside);
  const size_t eb = bf16 ? 2 : 4;
  ProfScope prof(ASI_K_SM_CORE, st, (double)p.B * p.C * p.H * p.W * eb);
  ASI_DISPATCH_R(launch_core_t, p, sm_core_smem(p, R, bf16), st);
}

cudaError_t launch_sm_wgrad(const SmWgradArgs& p, int R, bool bf16, int beside, cudaStream_t st) {
  const size_t eb = bf16 ? 2 : 4;
  ProfScope prof(ASI_K_SM_WGRAD, st,
                 (double)p.B * p.Cout * p.Ho * p.Wo * eb +
                     4.0 * (double)p.Cout * (p.C / p.groups) * p.kh * p.kw);
  if (R == 4) return bf16 ? launch_wgrad_t<4, __nv_bfloat16>(p, beside, st) : launch_wgrad_t<4, float>(p, beside, st);
  return bf16 ? launch_wgrad_t<8, __nv_bfloat16>(p, beside, st) : launch_wgrad_t<8, float>(p, beside, st);
}

// ---------------------------------------------------------------------------------------------
// Batched launches: the same kernels over the tiles of up to kMaxBatch layers of one variant (map size,
// rank bucket, input type) in one grid.  The per-layer argument blocks travel as a kernel parameter; a CTA
// finds its layer from the table of first CTA indices.
// ---------------------------------------------------------------------------------------------
int sm_max_batch() { return kMaxBatch; }

template <int KIND, int R, typename TX>
static cudaError_t launch_pass1_bt(const SmBatch<SmPass1Args>& b, size_t smem, cudaStream_t st) {
  return launch_clustered(k_sm_pass1_b<KIND, R, TX>, b.first[b.n], b.a[0].cl, smem, st, b);
}
template <int R, typename TX>
static cudaError_t launch_core_bt(const SmBatch<SmCoreArgs>& b, size_t smem, cudaStream_t st) {
  const bool staged = b.a[0].staged != 0;            // all layers of a launch or none
  auto kernel = staged ? k_sm_core_staged_b<R, TX> : k_sm_core_b<R, TX>;
  cudaError_t e = opt_in_smem(reinterpret_cast<const void*>(kernel), smem);
  if (e != cudaSuccess) return e;
  return launch_pdl(kernel, dim3(b.first[b.n]), dim3(staged ? kTT : kPT), smem, st, b);
}
template <int R, typename TX>
static cudaError_t launch_wgrad_bt(const SmBatch<SmWgradArgs>& b, size_t smem, bool staged, cudaStream_t st) {
  auto kernel = staged ? k_sm_wgrad_staged_b<R, TX> : (b.a[0].nt == 512 ? k_sm_wgrad_b<R, 512, TX> : k_sm_wgrad_b<R, 256, TX>);
  cudaError_t e = opt_in_smem(reinterpret_cast<const void*>(kernel), smem);
  if (e != cudaSuccess) return e;
  return launch_pdl(kernel, dim3(b.first[b.n]), dim3(staged ? kTT : b.a[0].nt), smem, st, b);
}

cudaError_t launch_sm_tile1_batched(const SmTile1Args* a, int n, int S, int R, bool bf16, cudaStream_t st) {
  if (n < 1 || n > kMaxBatch) return cudaErrorInvalidValue;
  SmBatch<SmTile1Args> b;
  size_t smem = 0;
  double bytes = 0.0;
  b.n = n;
  b.first[0] = 0;
  for (int l = 0; l < n; ++l) {
    b.a[l] = a[l];
    b.first[l + 1] = b.first[l] + a[l].n_tiles_b + sm_tile1_role_c_ctas(S, a[l].B);
    const size_t need = sm_tile1_smem(S, R, a[l].B, a[l].C);
    if (need > smem) smem = need;
    bytes += (double)a[l].B * a[l].C * S * S * (bf16 ? 2 : 4);
  }
  ProfScope prof(ASI_K_SM_PASS1, st, bytes);
  ASI_DISPATCH_SR(launch_tile1_bt, b, smem, st);
}

cudaError_t launch_sm_pass1_batched(const SmPass1Args* a, int n, int kind, int R, bool bf16, cudaStream_t st) {
  if (n < 1 || n > kMaxBatch) return cudaErrorInvalidValue;
  SmBatch<SmPass1Args> b;
  size_t smem = 0;
  double bytes = 0.0;
  b.n = n;
  b.first[0] = 0;
  int cl = 1;                                        // the launch's cluster size: a multiple of every layer's split
  for (int l = 0; l < n; ++l) cl = a[l].cs > cl ? a[l].cs : cl;
  for (int l = 0; l < n; ++l) {
    b.a[l] = a[l];
    b.a[l].cl = cl;
    b.first[l + 1] = b.first[l] + pass1_grid(b.a[l]);
    const size_t need = sm_pass1_smem(a[l], kind, R);
    if (need > smem) smem = need;
    bytes += (double)a[l].B * a[l].C * a[l].H * a[l].W * (bf16 ? 2 : 4);
  }
  ProfScope prof(ASI_K_SM_PASS1, st, bytes);
  ASI_DISPATCH_KR(launch_pass1_bt, b, smem, st);
}

cudaError_t launch_sm_reduce_batched(const SmReduceArgs* a, const int* max_chunks, int n, cudaStream_t st) {
  if (n < 1 || n > kMaxBatch) return cudaErrorInvalidValue;
  SmBatch<SmReduceArgs> b;
  b.n = n;
  b.first[0] = 0;
  for (int l = 0; l < n; ++l) {
    b.a[l] = a[l];
    b.first[l + 1] = b.first[l] + max_chunks[l];
  }
  ProfScope prof(ASI_K_QR, st, 0.0);
  return launch_pdl(k_sm_reduce_b, dim3((unsigned)b.first[n], 4), dim3(kRedNT), 0, st, b);
}

cudaError_t launch_sm_core_batched(const SmCoreArgs* a, int n, int R, bool bf16, int beside, cudaStream_t st) {
  if (n < 1 || n > kMaxBatch) return cudaErrorInvalidValue;
  SmBatch<SmCoreArgs> b;
  size_t smem = 0;
  double bytes = 0.0;
  b.n = n;
  b.first[0] = 0;
  for (int l = 0; l < n; ++l) b.a[l] = a[l];
  choose_core(b.a, n, R, bf16, beside);
  for (int l = 0; l < n; ++l) {
    b.first[l + 1] = b.first[l] + a[l].n_tiles;
    const size_t need = sm_core_smem(b.a[l], R, bf16);
    if (need > smem) smem = need;
    bytes += (double)a[l].B * a[l].C * a[l].H * a[l].W * (bf16 ? 2 : 4);
  }
  ProfScope prof(ASI_K_SM_CORE, st, bytes);
  ASI_DISPATCH_R(launch_core_bt, b, smem, st);
}

cudaError_t launch_sm_wgrad_batched(const SmWgradArgs* a, int n, int R, bool bf16, int beside, cudaStream_t st) {
  if (n < 1 || n > kMaxBatch) return cudaErrorInvalidValue;
  const bool staged = wgrad_staged(a, n, R, bf16, beside);
  SmBatch<SmWgradArgs> b;
  size_t smem = 0;
  double bytes = 0.0;
  b.n = n;
  b.first[0] = 0;
  for (int l = 0; l < n; ++l) {
    b.a[l] = a[l];
    b.first[l + 1] = b.first[l] + a[l].Cout / a[l].cpb;
    const size_t need = sm_wgrad_smem(a[l], R, staged, bf16);
    if (need > smem) smem = need;
    bytes += (double)a[l].B * a[l].Cout * a[l].Ho * a[l].Wo * (bf16 ? 2 : 4) +
             4.0 * (double)a[l].Cout * (a[l].C / a[l].groups) * a[l].kh * a[l].kw;
  }
  ProfScope prof(ASI_K_SM_WGRAD, st, bytes);
  if (R == 4) return bf16 ? launch_wgrad_bt<4, __nv_bfloat16>(b, smem, staged, st) : launch_wgrad_bt<4, float>(b, smem, staged, st);
  return bf16 ? launch_wgrad_bt<8, __nv_bfloat16>(b, smem, staged, st) : launch_wgrad_bt<8, float>(b, smem, staged, st);
}

}  // namespace asi
