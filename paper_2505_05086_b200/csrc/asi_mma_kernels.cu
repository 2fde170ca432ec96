// Both products of a mode, V = A_m^T U and P = A_m V (Algorithm 1), with the short factor on the tensor cores and fp32
// accuracy.
//
//   k_mfiber : one mode with strided fibers
//   k_mplane : the two spatial modes of a conv activation, maps of 12 to 32 rows and columns
//
// A factor has 4 to 8 columns, so a product is one instruction deep in N and its cost lies in moving the factor past the
// activation: on the fp32 pipe every value needs the factor's row from shared memory and a sum over the lanes that share a
// column.  mma.sync.m16n8k8 (tf32) keeps the factor in registers for the whole kernel and adds over the lanes itself.  Its
// operands come straight from the fragments that the lanes load; a matrix unit fed from shared memory (tcgen05) would need
// both halves of every split value written back first, and with N = 8 it waits for its A operand (22 us for a traversal of
// 25.7 M values, where the register form needs 5.5).
//
// fp32 on tf32: x = hi + lo, hi the upper 19 bits of x -- which is all the unit reads, so x itself is the operand -- and lo the
// exact rest, of which the unit reads eleven bits.  V is split at its nearest tf32 value instead, and a factor's rest is rounded to
// the nearest one as well, because its error is the same for every column of the activation and does not average out.  The eight
// columns of the B operand are (hi | lo) of up to four factor columns, or with NB = 2 two operands of up to eight.  The
// unit's own sums truncate, so it never adds more than two steps of the leading term (16 products) before the sum goes to a
// register in round-to-nearest; the small terms go first.  bf16 values are exact in tf32.
// Against 64 bits, mean error of the factors of the batch, the channels, the rows and the columns in 1e-8 (the fp32 pipe in
// parentheses): 60 conv layers of ranks above four 3.10 3.34 3.14 3.23 (2.91 4.74 3.21 3.32), 60 of ranks up to four 2.66 2.78
// 2.72 2.76 (2.58 3.00 2.71 2.77), 60 bf16 2.90 3.79 2.89 2.96 (2.78 3.69 2.95 3.10); the batch of 60 token layers 3.08 (2.87); 40
// cold starts 44.1 45.5 42.6 48.5 (46.7 47.4 50.8 61.1).  2.4 of each warm figure is the rounding of the output; what the short modes have more is
// the last bit of the previous factor, which two terms of eleven bits do not hold.  (Rounding x to its nearest tf32 value takes a
// tenth off the excess of ranks above four, but makes infinities of the largest values; the product of the two rests for ranks above
// four takes 3.5 % of a compress of 50 x 116 x 27 x 27 for 1 to 3 % of the error.)
//
// The k order of an operand is free as long as both sides agree, and so is the order of rows: a lane takes four (bf16:
// eight) neighbouring columns by one 16-byte read, as four m-tiles' rows in one product and four k-steps in the other.
//
// Measured (one launch, cold caches): 128 x 64 x 56 x 56 fp32 along the batch 22.8 us and along the channels 21.2 (27.2 and
// 31.1 on the fp32 pipe; the tensor's bytes take 15.7), 128 x 128 x 28 x 28 15.2 each (17, 18) and bf16 12.0 and 11.2 (15.6, 17.0);
// planes of 128 x 128 x 28 x 28 25.1 us (29.1), bf16 19.2 (26.9), of 50 x 116 x 27 x 27 with ranks 5 17.7 (30.4).  What bounds
// them is the latency of chains of four dependent mma on twelve warps an SM (issue slots half used).
#include <cuda.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <cstring>
#include <mutex>

#include "asi_internal.h"

namespace asi {

namespace {

__device__ __forceinline__ uint32_t s_addr(const void* p) { return static_cast<uint32_t>(__cvta_generic_to_shared(p)); }

typedef unsigned long long f2;     // two packed fp32 values
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
__device__ __forceinline__ f2 fadd2(f2 a, f2 b) {
  f2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f2 fsub2(f2 a, f2 b) {
  f2 r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}

__device__ __forceinline__ uint32_t fbits(float x) { return __float_as_uint(x); }

// c += a b, and c = a b.  The unit reads the upper 19 bits of an operand: an fp32 value is its own leading term
__device__ __forceinline__ void mma8(float (&c)[4], const float* a, const float* b) {
  asm("mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(fbits(a[0])), "r"(fbits(a[1])), "r"(fbits(a[2])), "r"(fbits(a[3])), "r"(fbits(b[0])), "r"(fbits(b[1])));
}
__device__ __forceinline__ void mma8_first(float (&c)[4], const float* a, const float* b) {
  asm("mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%10,%10,%10};"
      : "=f"(c[0]), "=f"(c[1]), "=f"(c[2]), "=f"(c[3])
      : "r"(fbits(a[0])), "r"(fbits(a[1])), "r"(fbits(a[2])), "r"(fbits(a[3])), "r"(fbits(b[0])), "r"(fbits(b[1])), "f"(0.f));
}

// what tf32 leaves of a pair of values
__device__ __forceinline__ void rest2(const float* x, float* lo) {
  const f2 v = pack2(x[0], x[1]);
  const float2 l = unpack2(fsub2(v, v & 0xffffe000ffffe000ull));
  lo[0] = l.x;
  lo[1] = l.y;
}
// the nearest tf32 value of a finite one (the carry makes a zero of 0x7fffffff, the NaN that arithmetic leaves)
__device__ __forceinline__ float nearest(float x) { return __uint_as_float((__float_as_uint(x) + 0x1000u) & 0xffffe000u); }

__device__ __forceinline__ void add_pair(float* s, float x, float y) {
  const float2 v = unpack2(fadd2(pack2(s[0], s[1]), pack2(x, y)));
  s[0] = v.x;
  s[1] = v.y;
}

// The A operand of a step and its rest below tf32 (fp32 values only)
template <bool EXACT>
struct FragA {
  float x[4], lo[EXACT ? 1 : 4];
};
// N values that a lane has read, and their rests
template <int N, bool EXACT>
struct Vals {
  float x[N], lo[EXACT ? 1 : N];
  __device__ __forceinline__ void rest() {
    if constexpr (!EXACT) {
#pragma unroll
      for (int i = 0; i < N; i += 2) rest2(x + i, lo + i);
    }
  }
  __device__ __forceinline__ void put(FragA<EXACT>& f, int slot, int i) const {
    f.x[slot] = x[i];
    if constexpr (!EXACT) f.lo[slot] = lo[i];
  }
};
// Sums of one tile.  b: NB = 1 {k, k + 4} of (hi | lo); NB = 2 {hi, hi, lo, lo}
template <int NB, bool EXACT>
struct Acc {
  float s[4];                                        // leading terms, two steps at a time in round-to-nearest
  __device__ __forceinline__ void zero() {
#pragma unroll
    for (int i = 0; i < 4; ++i) s[i] = 0.f;
  }
  __device__ __forceinline__ void two(const FragA<EXACT>& a0, const FragA<EXACT>& a1, const float* b0, const float* b1) {
    float q[4];
    if constexpr (EXACT) {
      if constexpr (NB == 2) {
        mma8_first(q, a0.x, b0 + 2);
        mma8(q, a1.x, b1 + 2);
        mma8(q, a0.x, b0);
      } else {
        mma8_first(q, a0.x, b0);
      }
    } else {
      mma8_first(q, a0.lo, b0);
      mma8(q, a1.lo, b1);
      if constexpr (NB == 2) {
        mma8(q, a0.x, b0 + 2);
        mma8(q, a1.x, b1 + 2);
      }
      mma8(q, a0.x, b0);
    }
    mma8(q, a1.x, b1);
    add_pair(s, q[0], q[1]);
    add_pair(s + 2, q[2], q[3]);
  }
};

// One entry of the B operand of the columns: lane group g is the column.  The rounding of a leading term carries a NaN over into a
// zero.  V keeps its rest as it is, a NaN with it: what the unit cuts off averages out over the columns.  Omega (few steps are as
// ill-conditioned as the first) and U_prev have theirs rounded too, which loses a NaN as well, but not in the difference: x - (x - hi) is
// hi again, or NaN where x is NaN or infinite.  What of U_prev would round to infinity leaves more to the rest instead
enum Operand { kV, kOmega, kFactor };
template <int NB, Operand WHAT>
__device__ __forceinline__ void set_b(float* b, int half, int g, float x) {
  float hi = nearest(x);
  if constexpr (WHAT == kFactor) {
    const float top = __uint_as_float(0x7f7fe000u);
    hi = fmaxf(fminf(hi, top), -top);
  }
  float lo = x - hi;
  if constexpr (WHAT != kV) {
    hi = x - lo;
    lo = nearest(lo);
  }
  if constexpr (NB == 1) b[half] = g < 4 ? hi : lo;
  else {
    b[half] = hi;
    b[2 + half] = lo;
  }
}

// N neighbouring values of shared memory
__device__ __forceinline__ void ld_vals(const float* p, float (&x)[4]) {
  const float4 v = *reinterpret_cast<const float4*>(p);
  x[0] = v.x; x[1] = v.y; x[2] = v.z; x[3] = v.w;
}
__device__ __forceinline__ void widen(uint32_t w, float* x) {
  x[0] = __uint_as_float(w << 16);
  x[1] = __uint_as_float(w & 0xffff0000u);
}
__device__ __forceinline__ void ld_vals(const __nv_bfloat16* p, float (&x)[4]) {
  const uint2 v = *reinterpret_cast<const uint2*>(p);
  widen(v.x, x); widen(v.y, x + 2);
}
__device__ __forceinline__ void ld_vals(const __nv_bfloat16* p, float (&x)[8]) {
  const uint4 v = *reinterpret_cast<const uint4*>(p);
  widen(v.x, x); widen(v.y, x + 2); widen(v.z, x + 4); widen(v.w, x + 6);
}

__device__ __forceinline__ void mbar_init(uint64_t* bar) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(s_addr(bar)) : "memory");
}
__device__ __forceinline__ void mbar_expect(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(s_addr(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(s_addr(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
// gives up after `limit` cycles
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, long long limit) {
  if (mbar_try(bar, parity)) return true;
  const long long t0 = clock64();
  for (uint32_t it = 0; it < (1u << 28); ++it) {
    if (mbar_try(bar, parity)) return true;
    if ((it & 255u) == 255u && clock64() - t0 > limit) return false;
  }
  return false;
}
// about a second; with the test hook, whose producer arms its barrier and issues no copy, about a millisecond
__device__ __forceinline__ long long wait_limit(int stall) { return stall ? 2000000ll : 2000000000ll; }
__device__ __forceinline__ void tma_box(void* dst, const CUtensorMap* map, int x, int y, int z, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(
          s_addr(dst)),
      "l"(map), "r"(x), "r"(y), "r"(z), "r"(s_addr(bar))
      : "memory");
}
__device__ __forceinline__ void bulk_copy(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(s_addr(dst)),
               "l"(src), "r"(bytes), "r"(s_addr(bar))
               : "memory");
}
// one fp32 value, or a zero when `on` is false (the source is not read)
__device__ __forceinline__ void cp_one(uint32_t dst, const float* src, bool on) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src), "r"(on ? 4 : 0) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_wait1() { asm volatile("cp.async.wait_group 1;" ::: "memory"); }
__device__ __forceinline__ void bar_team(int id, int n) { asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory"); }


constexpr int kMfThreads = 192;

}  // namespace

// ---------------------------------------------------------------------------------------------
// k_mfiber.  A team of T warps takes the same columns; warp w of it owns the rows [16 RT w, 16 RT (w + 1)) and fills and
// empties its own two buffers of them, [CB blocks][16 RT rows][128 bytes], each block 8 EPL columns wide with its 16-byte
// units swizzled by the row (TMA's 128-byte pattern).  The warps of a team meet once a tile, for the sum of their shares
// of V.  GIVEN (a cold start, P = A_m Omega): V is Omega, [Q][r] in memory, and comes with the tile.
// ---------------------------------------------------------------------------------------------
template <int RT, int NB, int CB, int LD, bool GIVEN, typename TX>
__global__ void __launch_bounds__(kMfThreads, 2)
    k_mfiber(const __grid_constant__ Fiber2Args p, const __grid_constant__ CUtensorMap map) {
  constexpr bool EX = sizeof(TX) == 2;
  constexpr int EPL = 16 / (int)sizeof(TX), NMT = EPL / 2, TCB = 8 * EPL, TC = CB * TCB, ROWS = 16 * RT;
  constexpr int NV = 4 * NB, VP = TC + 4;            // columns of a factor, row pitch of V
  constexpr uint32_t BLK = (uint32_t)ROWS * 128u, STAGE = CB * BLK;
  extern __shared__ __align__(1024) unsigned char mf_smem[];
  pass_begin(p.clear, p.first);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = blockDim.x >> 5;
  const int g = lane >> 2, c4 = lane & 3;
  const int T = p.team, G = nw / T, team = warp / T, tw = warp - team * T;
  unsigned char* buf = mf_smem + (size_t)warp * 2 * STAGE;
  float* Vt = reinterpret_cast<float*>(mf_smem + (size_t)nw * 2 * STAGE) + (size_t)team * 2 * T * NV * VP;   // [2][T][NV][VP]
  uint64_t* bars = reinterpret_cast<uint64_t*>(mf_smem + (size_t)nw * 2 * STAGE + (size_t)nw * 2 * NV * VP * 4) + 2 * warp;
  if (LD == 0 && lane < 2) {
    mbar_init(bars + lane);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncwarp();
  const TX* __restrict__ X = static_cast<const TX*>(p.X);
  const int a = p.a, r = p.r, row0 = tw * ROWS;
  const int nti = (int)((p.I + TC - 1) / TC), total = (int)p.n_tiles, stride = (int)gridDim.x * G;
  const int d_o = stride / nti, d_i = stride - d_o * nti;
  int t_ld = (int)blockIdx.x * G + team;
  int o_ld = t_ld / nti, i_ld = t_ld - o_ld * nti;
  auto fill = [&](int st) {
    if (t_ld < total) {
      unsigned char* dst = buf + st * STAGE;
      if constexpr (LD == 0) {
        if (lane == 0) {
          mbar_expect(bars + st, STAGE);
#pragma unroll
          for (int cb = 0; cb < CB; ++cb)
            if (!p.stall) tma_box(dst + cb * BLK, &map, i_ld * TC + cb * TCB, row0, o_ld, bars + st);
        }
      } else {
#pragma unroll 1
        for (int cb = 0; cb < CB; ++cb) {
          const int64_t col = (int64_t)i_ld * TC + cb * TCB + lane;
          const bool on = col < p.I;
          const float* src = reinterpret_cast<const float*>(X) + ((int64_t)o_ld * a + row0) * p.I + (on ? col : 0);
          const uint32_t d = s_addr(dst + cb * BLK) + 4 * (lane & 3);
          const int last = a - 1 - row0;               // rows beyond the tensor are zeros; their address stays inside
#pragma unroll 8
          for (int k = 0; k < ROWS; ++k)
            cp_one(d + k * 128 + (((lane >> 2) ^ (k & 7)) << 4), src + (int64_t)(k <= last ? k : (last < 0 ? -row0 : last)) * p.I,
                   on && k <= last);
        }
      }
    }
    if constexpr (GIVEN) {                           // the team's warps share the copy of V
      if (t_ld < total) {
        const int64_t i0 = (int64_t)i_ld * TC;
        const float* src = p.U + ((int64_t)o_ld * p.I + i0) * r;
        const uint32_t d = s_addr(Vt + st * T * (NV * VP));
        const int n = (int)(p.I - i0 < TC ? p.I - i0 : TC) * r;
        for (int e = 32 * tw + lane; e < TC * r; e += 32 * T) {
          const int q = e / r, j = e - q * r;
          cp_one(d + 4 * (j * VP + q), src + (e < n ? e : 0), e < n);
        }
      }
    }
    if constexpr (LD == 1 || GIVEN) cp_commit();
    t_ld += stride;
    o_ld += d_o;
    i_ld += d_i;
    if (i_ld >= nti) { i_ld -= nti; ++o_ld; }
  };
  const int t_first = t_ld;
  if constexpr (GIVEN) {
    for (int e = lane; e < 2 * NV * VP; e += 32) Vt[tw * 2 * NV * VP + e] = 0.f;   // columns past r
    if (T > 1) bar_team(1 + team, 32 * T);
    else __syncwarp();
  }
  fill(0);
  fill(1);
  // the factor: step s, slots c4 and c4 + 4 are rows 8 s + 2 c4 and the next one
  float ub[2 * RT][2 * NB];
#pragma unroll
  for (int s = 0; s < 2 * RT && !GIVEN; ++s)
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int k = row0 + 8 * s + 2 * c4 + h, j = NB == 1 ? (g & 3) : g;
      set_b<NB, kFactor>(ub[s], h, g, (k < a && j < r) ? __ldg(p.U + (int64_t)k * p.ldu + j) : 0.f);
    }
  Acc<NB, EX> P[RT];
#pragma unroll
  for (int m = 0; m < RT; ++m) P[m].zero();
  // byte offsets of this lane's units: column owner (rows 2 c4 and 2 c4 + 1, unit g), row owner (row perm(g), units c4, c4 + 4)
  const uint32_t offc0 = (2 * c4) * 128 + ((g ^ (2 * c4)) << 4), offc1 = (2 * c4 + 1) * 128 + ((g ^ (2 * c4 + 1)) << 4);
  const int pr = (g >> 1) + 4 * (g & 1);
  const uint32_t offr0 = pr * 128 + ((c4 ^ pr) << 4), offr1 = pr * 128 + (((c4 + 4) ^ pr) << 4);

  int st = 0, vb = 0;
  uint32_t phase = 0;
  bool failed = false;
#pragma unroll 1
  for (int t = t_first; t < total; t += stride) {
    if constexpr (LD == 0) {
      const long long limit = wait_limit(p.stall);
      if (!failed && !mbar_wait(bars + st, (phase >> st) & 1u, limit)) {
        failed = true;                               // the team's barriers go on; what follows is not used
        atomicMax(p.status, (int)ASI_ERR_TIMEOUT);
        mbar_wait(bars + st, (phase >> st) & 1u, limit);   // the copies in flight get the limit once more
        if (t + stride < total) mbar_wait(bars + (st ^ 1), (phase >> (st ^ 1)) & 1u, limit);
      }
      phase ^= 1u << st;
    }
    if constexpr (LD == 1 || GIVEN) cp_wait1();
    __syncwarp();
    const unsigned char* xs = buf + st * STAGE;
    float* Vw = Vt + (vb * T + tw) * (NV * VP);
    // ---- V of this warp's rows
#pragma unroll
    for (int cb = 0; cb < CB && !GIVEN; ++cb) {
      Acc<NB, EX> v2[NMT];
#pragma unroll
      for (int m = 0; m < NMT; ++m) v2[m].zero();
#pragma unroll
      for (int s2 = 0; s2 < RT; ++s2) {
        Vals<EPL, EX> xa[2], xb[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const unsigned char* xr = xs + cb * BLK + (2 * s2 + h) * 1024;
          ld_vals(reinterpret_cast<const TX*>(xr + offc0), xa[h].x);
          ld_vals(reinterpret_cast<const TX*>(xr + offc1), xb[h].x);
          xa[h].rest();
          xb[h].rest();
        }
#pragma unroll
        for (int m = 0; m < NMT; ++m) {
          FragA<EX> f[2];
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            xa[h].put(f[h], 0, 2 * m); xa[h].put(f[h], 1, 2 * m + 1);
            xb[h].put(f[h], 2, 2 * m); xb[h].put(f[h], 3, 2 * m + 1);
          }
          v2[m].two(f[0], f[1], ub[2 * s2], ub[2 * s2 + 1]);
        }
      }
      // column 4 g + e (bf16: 8 g + e) sits in tile e / 2, rows g (e even) and g + 8 (e odd)
      float v[NMT][4];
#pragma unroll
      for (int m = 0; m < NMT; ++m)
#pragma unroll
        for (int i = 0; i < 4; ++i) v[m][i] = v2[m].s[i];
      if constexpr (NB == 1) {
#pragma unroll
        for (int m = 0; m < NMT; ++m)
#pragma unroll
          for (int i = 0; i < 4; ++i) v[m][i] += __shfl_xor_sync(0xffffffffu, v[m][i], 2);
        const bool odd = c4 & 2;
        float* d = Vw + (2 * (c4 & 1) + (odd ? 1 : 0)) * VP + cb * TCB + g * EPL;
#pragma unroll
        for (int m = 0; m < NMT; m += 2)
          *reinterpret_cast<float4*>(d + 2 * m) = odd ? make_float4(v[m][1], v[m][3], v[m + 1][1], v[m + 1][3])
                                                      : make_float4(v[m][0], v[m][2], v[m + 1][0], v[m + 1][2]);
      } else {
        float* d = Vw + (2 * c4) * VP + cb * TCB + g * EPL;
#pragma unroll
        for (int m = 0; m < NMT; m += 2) {
          *reinterpret_cast<float4*>(d + 2 * m) = make_float4(v[m][0], v[m][2], v[m + 1][0], v[m + 1][2]);
          *reinterpret_cast<float4*>(d + VP + 2 * m) = make_float4(v[m][1], v[m][3], v[m + 1][1], v[m + 1][3]);
        }
      }
    }
    if (T > 1) bar_team(1 + team, 32 * T);
    else __syncwarp();
    const float* Vr = Vt + vb * T * (NV * VP);
    {
      // ---- P of this warp's rows
#pragma unroll
      for (int cb = 0; cb < CB; ++cb) {
        float b[EPL][2 * NB];
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
          for (int u = 0; u < EPL; u += 4) {
            const float* src = Vr + (NB == 1 ? (g & 3) : g) * VP + cb * TCB + h * (TCB / 2) + c4 * EPL + u;
            float x[4];
            ld_vals(src, x);
            for (int w = 1; w < T && !GIVEN; ++w) {
              float y[4];
              ld_vals(src + w * (NV * VP), y);
#pragma unroll
              for (int i = 0; i < 4; ++i) x[i] += y[i];
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) set_b<NB, GIVEN ? kOmega : kV>(b[u + i], h, g, x[i]);
          }
#pragma unroll
        for (int m = 0; m < RT; ++m) {
          Vals<EPL, EX> x00, x10, x01, x11;
          const unsigned char* xr = xs + cb * BLK + m * 2048;
          ld_vals(reinterpret_cast<const TX*>(xr + offr0), x00.x);
          ld_vals(reinterpret_cast<const TX*>(xr + 1024 + offr0), x10.x);
          ld_vals(reinterpret_cast<const TX*>(xr + offr1), x01.x);
          ld_vals(reinterpret_cast<const TX*>(xr + 1024 + offr1), x11.x);
          x00.rest(); x10.rest(); x01.rest(); x11.rest();
#pragma unroll
          for (int e = 0; e < EPL; e += 2) {
            FragA<EX> f[2];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              x00.put(f[h], 0, e + h); x10.put(f[h], 1, e + h);
              x01.put(f[h], 2, e + h); x11.put(f[h], 3, e + h);
            }
            P[m].two(f[0], f[1], b[e], b[e + 1]);
          }
        }
      }
    }
    // the stage has been read by all lanes (its V by the team)
    if (GIVEN && T > 1) bar_team(1 + team, 32 * T);
    else __syncwarp();
    if (!failed) fill(st);
    else { t_ld += stride; if constexpr (LD == 1 || GIVEN) cp_commit(); }
    st ^= 1;
    vb ^= 1;
    if (T == 1) __syncwarp();
  }
  if (tid == 0) pdl_wait();
  // ---- one partial of P per CTA: the teams' sums meet in team order
  if (__syncthreads_or(failed)) return;              // else every copy has landed, and the buffers serve again
  float* red = reinterpret_cast<float*>(mf_smem) + (size_t)warp * (ROWS * NV);     // [nw][ROWS][NV]
#pragma unroll
  for (int m = 0; m < RT; ++m) {
    float v[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      v[i] = P[m].s[i];
      if constexpr (NB == 1) v[i] += __shfl_xor_sync(0xffffffffu, v[i], 2);
    }
    if (NB == 2 || c4 < 2) {
      float* d = red + (16 * m + pr) * NV + 2 * c4;
      *reinterpret_cast<float2*>(d) = make_float2(v[0], v[1]);
      *reinterpret_cast<float2*>(d + 8 * NV) = make_float2(v[2], v[3]);
    }
  }
  __syncthreads();
  const float* all = reinterpret_cast<const float*>(mf_smem);
  for (int e = tid; e < a * r; e += blockDim.x) {
    const int k = e / r, j = e - k * r;
    float s = 0.f;
    for (int q = 0; q < G; ++q) s += all[((size_t)q * T * ROWS + k) * NV + j];
    p.Pp[(int64_t)blockIdx.x * a * r + e] = s;
  }
}

namespace {
typedef CUresult (*EncodeFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                             const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                             CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
EncodeFn encode_fn() {
  static EncodeFn fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* q = nullptr;
    cudaDriverEntryPointQueryResult res;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &q, cudaEnableDefault, &res) == cudaSuccess &&
        res == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeFn>(q);
  });
  return fn;
}

// Rows a warp and warps a team: at most 64 rows a warp.  A CTA has as many teams as keep it near 96 KB, so that two share an SM.
struct MfShape {
  int rt, team, cb, nw;
  size_t smem;
};
MfShape mf_shape(int a, int r, bool bf16) {
  MfShape s;
  const int most = bf16 && r > 4 ? 32 : 64;          // rows of a warp (bf16, ranks above 4: 216 bytes of spills at 64)
  s.team = (a + most - 1) / most;
  s.rt = (a + 16 * s.team - 1) / (16 * s.team);
  s.cb = s.rt == 1 ? 4 : (s.rt == 2 ? 2 : 1);
  const int nv = r <= 4 ? 4 : 8, vp = s.cb * (bf16 ? 64 : 32) + 4;
  const size_t warp = (size_t)2 * s.cb * s.rt * 2048 + (size_t)2 * nv * vp * 4 + 16;
  int g = (int)((104 * 1024) / (warp * s.team));
  g = g < 1 ? 1 : g;
  while (g > 1 && g * s.team > kMfThreads / 32) --g;
  s.nw = g * s.team;
  s.smem = warp * s.nw;
  return s;
}
}  // namespace

// Modes of up to 384 entries (six warps of 64 rows; bf16 128, what k_wfiber takes where an address is odd) and ranks up to 8; rows of
// at least 32 columns.  bf16 needs rows on 16 bytes; fp32 rows of any length come by four-byte copies.
bool mfiber_supported(int64_t O, int64_t a, int64_t I, int r, bool bf16) {
  return a >= 2 && a <= (bf16 ? 128 : 384) && r <= 8 && I >= 32 && (!bf16 || I % 8 == 0) && O * ((I + 31) / 32) < (1ll << 30) &&
         O < (1ll << 31) && I < (1ll << 31) && a * I < (1ll << 37);
}
int mfiber_grid(int64_t O, int64_t a, int64_t I, int r, bool bf16, bool share_sm) {
  const MfShape s = mf_shape((int)a, r, bf16);
  const int64_t tc = s.cb * (bf16 ? 64 : 32), tiles = O * ((I + tc - 1) / tc), g = s.nw / s.team;
  const int per_sm = share_sm || s.smem > 112 * 1024 ? 1 : 2;
  return (int)std::min<int64_t>((tiles + g - 1) / g, 148 * per_sm);
}

template <int RT, int NB, int CB, int LD, bool GIVEN, typename TX>
static cudaError_t launch_mfiber_tg(const Fiber2Args& p, const CUtensorMap& map, const MfShape& s, int grid, cudaStream_t st) {
  const cudaError_t e = opt_in_smem(reinterpret_cast<const void*>(k_mfiber<RT, NB, CB, LD, GIVEN, TX>), s.smem);
  if (e != cudaSuccess) return e;
  return launch_pdl(k_mfiber<RT, NB, CB, LD, GIVEN, TX>, dim3(grid), dim3(32 * s.nw), s.smem, st, p, map);
}

template <int RT, int NB, int CB, int LD, typename TX>
static cudaError_t launch_mfiber_t(const Fiber2Args& p, const CUtensorMap& map, const MfShape& s, int grid, cudaStream_t st) {
  return p.given ? launch_mfiber_tg<RT, NB, CB, LD, true, TX>(p, map, s, grid, st)
                 : launch_mfiber_tg<RT, NB, CB, LD, false, TX>(p, map, s, grid, st);
}

cudaError_t launch_mfiber(const Fiber2Args& p0, int grid, bool bf16, cudaStream_t st) {
  Fiber2Args p = p0;
  const MfShape s = mf_shape(p.a, p.r, bf16);
  const int64_t tc = s.cb * (bf16 ? 64 : 32);
  p.team = s.team;
  p.n_tiles = p.O * ((p.I + tc - 1) / tc);
  const int eb = bf16 ? 2 : 4;
  const bool rows16 = (p.I * eb) % 16 == 0 && (reinterpret_cast<uintptr_t>(p.X) & 15u) == 0;
  CUtensorMap map;
  std::memset(&map, 0, sizeof(map));
  if (rows16) {
    const EncodeFn enc = encode_fn();
    if (!enc) return cudaErrorNotSupported;
    const cuuint64_t dims[3] = {(cuuint64_t)p.I, (cuuint64_t)p.a, (cuuint64_t)p.O};
    const cuuint64_t strides[2] = {(cuuint64_t)(p.I * eb), (cuuint64_t)(p.I * p.a * eb)};
    const cuuint32_t box[3] = {(cuuint32_t)(128 / eb), (cuuint32_t)(16 * s.rt), 1}, one[3] = {1, 1, 1};
    if (enc(&map, bf16 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, const_cast<void*>(p.X), dims,
            strides, box, one, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
      return cudaErrorInvalidValue;
  } else if (bf16) {
    return cudaErrorInvalidValue;                    // the caller takes another kernel
  }
  ProfScope prof(ASI_K_EXPAND, st, (double)p.O * p.a * p.I * eb);
#define ASI_MF(RT_, CB_, NB16_)  /* NB16: of bf16 above rank four, which has at most two row tiles a warp */                \
  if (bf16) return p.r <= 4 ? launch_mfiber_t<RT_, 1, CB_, 0, __nv_bfloat16>(p, map, s, grid, st)                      \
                            : launch_mfiber_t<RT_, NB16_, CB_, 0, __nv_bfloat16>(p, map, s, grid, st);                 \
  if (rows16) return p.r <= 4 ? launch_mfiber_t<RT_, 1, CB_, 0, float>(p, map, s, grid, st)                            \
                              : launch_mfiber_t<RT_, 2, CB_, 0, float>(p, map, s, grid, st);                           \
  return p.r <= 4 ? launch_mfiber_t<RT_, 1, CB_, 1, float>(p, map, s, grid, st)                                        \
                  : launch_mfiber_t<RT_, 2, CB_, 1, float>(p, map, s, grid, st)
  if (bf16 && p.r > 4 && s.rt > 2) return cudaErrorInvalidValue;   // not built: mf_shape
  switch (s.rt) {
    case 1: ASI_MF(1, 4, 2);
    case 2: ASI_MF(2, 2, 2);
    case 3: ASI_MF(3, 1, 1);
    default: ASI_MF(4, 1, 1);
  }
#undef ASI_MF
}

// ---------------------------------------------------------------------------------------------
// k_mplane.  A warp owns whole planes and two buffers for them.  Per plane:
//   1 columns  V3[w][j] = sum_h X[h][w] U3[h][j]
//   2 rows     V4[h][j] = sum_w X[h][w] U4[w][j] and P3[h][j] += sum_w X[h][w] V3[w][j], on the same fragments
//   3 columns  P4[w][j] += sum_h X[h][w] V4[h][j]
// The factors and the sums P3, P4 stay in registers.  Rows beyond the plane are zeros of the buffer; columns beyond a row are
// its neighbour's values and meet a zero of the factor, or make sums nobody reads.  GIVEN (a cold start): V3 and V4 are the
// planes' rows of Omega_3 and Omega_4 and come with the plane.
// ---------------------------------------------------------------------------------------------
constexpr int kMpThreads = 192;

template <int NB, int LD, bool GIVEN, typename TX>
__global__ void __launch_bounds__(kMpThreads, 2) k_mplane(const __grid_constant__ PlaneArgs p) {
  constexpr bool EX = sizeof(TX) == 2;
  constexpr int NV = 4 * NB, VP = 36;                // row pitch of V3 and V4: 32 and four
  extern __shared__ __align__(128) unsigned char mp_smem[];
  pass_begin(p.clear, p.first);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = blockDim.x >> 5;
  const int g = lane >> 2, c4 = lane & 3, H = p.H, W = p.W, hw = H * W;
  const int jb = NB == 1 ? (g & 3) : g;
  const int pb = p.pitch;                            // bytes of a buffer
  unsigned char* buf = mp_smem + (size_t)warp * (2 * pb);
  float* V3 = reinterpret_cast<float*>(mp_smem + (size_t)nw * 2 * pb) + warp * (4 * NV * VP);     // [2][NV][VP] (GIVEN: per buffer)
  float* V4 = V3 + 2 * NV * VP;                                                                   // [2][NV][VP]
  uint64_t* bars = reinterpret_cast<uint64_t*>(mp_smem + (size_t)nw * 2 * pb + (size_t)nw * 4 * NV * VP * 4) + 2 * warp;
  for (int e = lane; e < 2 * pb / 16; e += 32) reinterpret_cast<uint4*>(buf)[e] = make_uint4(0, 0, 0, 0);
  for (int e = lane; e < 4 * NV * VP; e += 32) V3[e] = 0.f;
  if (LD == 0 && lane < 2) {
    mbar_init(bars + lane);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // the zeros are older than the copies
  __syncwarp();
  const TX* __restrict__ X = static_cast<const TX*>(p.X);
  const int64_t stride = (int64_t)gridDim.x * nw;
  int64_t t_ld = (int64_t)blockIdx.x * nw + warp;
  auto fill = [&](int st) {
    if (t_ld < p.n_planes) {
      if constexpr (LD == 0) {
        if (lane == 0) {
          mbar_expect(bars + st, (uint32_t)(hw * sizeof(TX)));
          if (!p.stall) bulk_copy(buf + st * pb, X + t_ld * hw, (uint32_t)(hw * sizeof(TX)), bars + st);
        }
      } else {
        const float* src = reinterpret_cast<const float*>(X) + t_ld * hw;
        const uint32_t d = s_addr(buf + st * pb);
#pragma unroll 8
        for (int e = lane; e < hw; e += 32) cp_one(d + 4 * e, src + e, true);
      }
      if constexpr (GIVEN) {
        const uint32_t d3 = s_addr(V3 + st * NV * VP), d4 = s_addr(V4 + st * NV * VP);
        const float *s3 = p.U3 + t_ld * W * p.r3, *s4 = p.U4 + t_ld * H * p.r4;
        for (int e = lane; e < W * p.r3; e += 32) cp_one(d3 + 4 * ((e % p.r3) * VP + e / p.r3), s3 + e, true);
        for (int e = lane; e < H * p.r4; e += 32) cp_one(d4 + 4 * ((e % p.r4) * VP + e / p.r4), s4 + e, true);
      }
    }
    if constexpr (LD == 1 || GIVEN) cp_commit();
    t_ld += stride;
  };
  const int64_t t_first = t_ld;
  fill(0);
  fill(1);
  // orders that keep the four rows of a column owner and the two of a row owner on different banks: W = 8 (mod 16) wants
  // neighbouring rows and rows two apart, W = 4 (mod 8) rows two and four apart
  const bool dbl = (W & 7) == 4;
  const int kr0 = dbl ? 2 * c4 : c4, kr1 = dbl ? 2 * c4 + 1 : c4 + 4;
  const int pr = dbl ? (g >> 1) + 4 * (g & 1) : (g & 4) + ((g >> 1) & 1) + 2 * (g & 1);
  // columns of a lane's four values: column owner; row owner, half h
  auto wcol = [&](int e) { return LD == 0 ? 4 * g + e : 8 * e + g; };
  auto wrow = [&](int h, int e) { return LD == 0 ? 16 * h + 4 * c4 + e : 8 * e + 4 * h + c4; };
  float u3[4][2 * NB], u4[4][2 * NB];
#pragma unroll
  for (int s = 0; s < 4 && !GIVEN; ++s)
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int k = 8 * s + (h ? kr1 : kr0), w = wrow(h, s);
      set_b<NB, kFactor>(u3[s], h, g, (k < H && jb < p.r3) ? __ldg(p.U3 + k * p.r3 + jb) : 0.f);
      set_b<NB, kFactor>(u4[s], h, g, (w < W && jb < p.r4) ? __ldg(p.U4 + w * p.r4 + jb) : 0.f);
    }
  Acc<NB, EX> P3[2], P4[2];
#pragma unroll
  for (int m = 0; m < 2; ++m) {
    P3[m].zero();
    P4[m].zero();
  }
  auto ld4 = [&](const TX* s, Vals<4, EX>& v) {
    if constexpr (LD == 0) ld_vals(s, v.x);
    else {
#pragma unroll
      for (int e = 0; e < 4; ++e) v.x[e] = s[8 * e];
    }
    v.rest();
  };
  // steps 2 s2 and 2 s2 + 1 down the columns: rows 16 s2 .. 16 s2 + 15
  auto col_steps = [&](const TX* xs, int s2, const float* b0, const float* b1, Acc<NB, EX> (&sum)[2]) {
    Vals<4, EX> xa[2], xb[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      ld4(xs + (8 * (2 * s2 + h) + kr0) * W + wcol(0), xa[h]);
      ld4(xs + (8 * (2 * s2 + h) + kr1) * W + wcol(0), xb[h]);
    }
#pragma unroll
    for (int m = 0; m < 2; ++m) {
      FragA<EX> f[2];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        xa[h].put(f[h], 0, 2 * m); xa[h].put(f[h], 1, 2 * m + 1);
        xb[h].put(f[h], 2, 2 * m); xb[h].put(f[h], 3, 2 * m + 1);
      }
      sum[m].two(f[0], f[1], b0, b1);
    }
  };
  const int nkh = (H + 15) / 16;                     // pairs of k-steps, row tiles

  int st = 0;
  uint32_t phase = 0;
  bool failed = false;
#pragma unroll 1
  for (int64_t t = t_first; t < p.n_planes; t += stride) {
    if constexpr (LD == 0) {
      const long long limit = wait_limit(p.stall);
      if (!failed && !mbar_wait(bars + st, (phase >> st) & 1u, limit)) {
        failed = true;
        atomicMax(p.status, (int)ASI_ERR_TIMEOUT);
        mbar_wait(bars + st, (phase >> st) & 1u, limit);   // the copies in flight get the limit once more
        if (t + stride < p.n_planes) mbar_wait(bars + (st ^ 1), (phase >> (st ^ 1)) & 1u, limit);
      }
      phase ^= 1u << st;
    }
    if constexpr (LD == 1 || GIVEN) cp_wait1();
    __syncwarp();
    const TX* xs = reinterpret_cast<const TX*>(buf + st * pb);
    const float *W3 = V3 + (GIVEN ? st * NV * VP : 0), *W4 = V4 + (GIVEN ? st * NV * VP : 0);
    // ---- 1: V3
    if constexpr (!GIVEN) {
      Acc<NB, EX> v2[2];
      v2[0].zero();
      v2[1].zero();
#pragma unroll
      for (int s2 = 0; s2 < 2; ++s2) {
        if (s2 >= nkh) break;
        col_steps(xs, s2, u3[2 * s2], u3[2 * s2 + 1], v2);
      }
      float v[2][4];
#pragma unroll
      for (int m = 0; m < 2; ++m)
#pragma unroll
        for (int i = 0; i < 4; ++i) v[m][i] = v2[m].s[i];
      auto put = [&](int j, float x0, float x1, float x2, float x3) {
        float* d = V3 + j * VP + wcol(0);
        if constexpr (LD == 0) *reinterpret_cast<float4*>(d) = make_float4(x0, x1, x2, x3);
        else {
          d[0] = x0; d[8] = x1; d[16] = x2; d[24] = x3;
        }
      };
      if constexpr (NB == 1) {
#pragma unroll
        for (int m = 0; m < 2; ++m)
#pragma unroll
          for (int i = 0; i < 4; ++i) v[m][i] += __shfl_xor_sync(0xffffffffu, v[m][i], 2);
        if (c4 & 2) put(2 * (c4 & 1) + 1, v[0][1], v[0][3], v[1][1], v[1][3]);
        else put(2 * (c4 & 1), v[0][0], v[0][2], v[1][0], v[1][2]);
      } else {
        put(2 * c4, v[0][0], v[0][2], v[1][0], v[1][2]);
        put(2 * c4 + 1, v[0][1], v[0][3], v[1][1], v[1][3]);
      }
    }
    __syncwarp();
    // ---- 2: V4 and P3
    {
      float b3[4][2 * NB];
#pragma unroll
      for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int e = 0; e < 4; ++e) set_b<NB, GIVEN ? kOmega : kV>(b3[e], h, g, wrow(h, e) < W ? W3[jb * VP + wrow(h, e)] : 0.f);
#pragma unroll
      for (int m = 0; m < 2; ++m) {
        if (m >= nkh) break;
        Acc<NB, EX> v2;
        v2.zero();
        const int ra = 16 * m + pr, rb = ra + 8;
        Vals<4, EX> x00, x10, x01, x11;
        ld4(xs + ra * W + wrow(0, 0), x00);
        ld4(xs + rb * W + wrow(0, 0), x10);
        ld4(xs + ra * W + wrow(1, 0), x01);
        ld4(xs + rb * W + wrow(1, 0), x11);
#pragma unroll
        for (int e = 0; e < 4; e += 2) {
          FragA<EX> f[2];
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            x00.put(f[h], 0, e + h); x10.put(f[h], 1, e + h);
            x01.put(f[h], 2, e + h); x11.put(f[h], 3, e + h);
          }
          if constexpr (!GIVEN) v2.two(f[0], f[1], u4[e], u4[e + 1]);
          P3[m].two(f[0], f[1], b3[e], b3[e + 1]);
        }
        if constexpr (!GIVEN) {
          float v[4];
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            v[i] = v2.s[i];
            if constexpr (NB == 1) v[i] += __shfl_xor_sync(0xffffffffu, v[i], 2);
          }
          if constexpr (NB == 1) {
            float* d = V4 + (2 * (c4 & 1) + (c4 >> 1)) * VP;
            d[ra] = (c4 & 2) ? v[1] : v[0];
            d[rb] = (c4 & 2) ? v[3] : v[2];
          } else {
            float* d = V4 + 2 * c4 * VP;
            d[ra] = v[0]; d[VP + ra] = v[1];
            d[rb] = v[2]; d[VP + rb] = v[3];
          }
        }
      }
    }
    __syncwarp();
    // ---- 3: P4
#pragma unroll
    for (int s2 = 0; s2 < 2; ++s2) {
      if (s2 >= nkh) break;
      float b4[2][2 * NB];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        set_b<NB, GIVEN ? kOmega : kV>(b4[h], 0, g, W4[jb * VP + 8 * (2 * s2 + h) + kr0]);
        set_b<NB, GIVEN ? kOmega : kV>(b4[h], 1, g, W4[jb * VP + 8 * (2 * s2 + h) + kr1]);
      }
      col_steps(xs, s2, b4[0], b4[1], P4);
    }
    __syncwarp();                                    // the buffer has been read by all lanes
    if (!failed) fill(st);
    else { t_ld += stride; if constexpr (LD == 1 || GIVEN) cp_commit(); }
    st ^= 1;
  }
  if (tid == 0) pdl_wait();
  // ---- one partial of P3 and P4 per CTA: the warps' sums meet in warp order
  if (__syncthreads_or(failed)) return;              // else every copy has landed, and the buffers serve again
  float* red = reinterpret_cast<float*>(mp_smem) + (size_t)warp * (2 * 32 * NV);   // [nw][2][32][NV]
#pragma unroll
  for (int m = 0; m < 2; ++m) {
    float s3[4], s4[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      s3[i] = P3[m].s[i];
      s4[i] = P4[m].s[i];
      if constexpr (NB == 1) {
        s3[i] += __shfl_xor_sync(0xffffffffu, s3[i], 2);
        s4[i] += __shfl_xor_sync(0xffffffffu, s4[i], 2);
      }
    }
    if (NB == 2 || c4 < 2) {
      float* d = red + (16 * m + pr) * NV + 2 * c4;
      *reinterpret_cast<float2*>(d) = make_float2(s3[0], s3[1]);
      *reinterpret_cast<float2*>(d + 8 * NV) = make_float2(s3[2], s3[3]);
      d = red + 32 * NV + 2 * c4;                    // tile m: columns e = 2 m and the next
      *reinterpret_cast<float2*>(d + wcol(2 * m) * NV) = make_float2(s4[0], s4[1]);
      *reinterpret_cast<float2*>(d + wcol(2 * m + 1) * NV) = make_float2(s4[2], s4[3]);
    }
  }
  __syncthreads();
  const float* all = reinterpret_cast<const float*>(mp_smem);
  const int n3 = H * p.r3, n4 = W * p.r4;
  for (int e = tid; e < n3 + n4; e += blockDim.x) {
    const bool four = e >= n3;
    const int x = four ? e - n3 : e, r = four ? p.r4 : p.r3, k = x / r, j = x - k * r;
    const float* src = all + (four ? 32 * NV : 0) + k * NV + j;
    float s = 0.f;
    for (int w = 0; w < nw; ++w) s += src[(size_t)w * (2 * 32 * NV)];
    if (four) p.Pp4[(int64_t)blockIdx.x * n4 + x] = s;
    else p.Pp3[(int64_t)blockIdx.x * n3 + x] = s;
  }
}

namespace {
struct MpShape {
  int nw, pb;
  size_t smem;
};
MpShape mp_shape(int H, int W, int r, bool bf16) {
  MpShape s;
  const int nv = r <= 4 ? 4 : 8;
  s.pb = ((((H + 15) / 16 * 16) * W + 32) * (bf16 ? 2 : 4) + 127) / 128 * 128;
  const size_t warp = std::max((size_t)2 * s.pb + (size_t)4 * nv * 36 * 4 + 16, (size_t)2 * 32 * nv * 4);   // the epilogue reuses the buffers
  s.nw = std::min((int)((112 * 1024) / warp), kMpThreads / 32);
  s.smem = warp * s.nw;
  return s;
}
}  // namespace

// Maps of 12 to 32 rows and columns (smaller ones leave the tiles empty, larger ones keep too few warps on an SM: 56 x 56
// takes 51 us here, 43 with k_plane2).
// bf16 needs rows of four and planes on 16 bytes; fp32 planes of any size come by four-byte copies
bool mplane_supported(int64_t n_planes, int64_t H, int64_t W, int r3, int r4, bool bf16) {
  return H >= 12 && W >= 12 && H <= 32 && W <= 32 && r3 <= 8 && r4 <= 8 && n_planes < (1ll << 31) &&
         (!bf16 || (W % 4 == 0 && (H * W) % 8 == 0));
}
int mplane_grid(int64_t n_planes, int H, int W, int r, bool bf16, bool share_sm) {
  const MpShape s = mp_shape(H, W, r, bf16);
  return (int)std::min<int64_t>((n_planes + s.nw - 1) / s.nw, 148 * (share_sm ? 1 : 2));
}

template <int NB, int LD, bool GIVEN, typename TX>
static cudaError_t launch_mplane_tg(const PlaneArgs& p, const MpShape& s, int grid, cudaStream_t st) {
  const cudaError_t e = opt_in_smem(reinterpret_cast<const void*>(k_mplane<NB, LD, GIVEN, TX>), s.smem);
  if (e != cudaSuccess) return e;
  return launch_pdl(k_mplane<NB, LD, GIVEN, TX>, dim3(grid), dim3(32 * s.nw), s.smem, st, p);
}

template <int NB, int LD, typename TX>
static cudaError_t launch_mplane_t(const PlaneArgs& p, const MpShape& s, int grid, cudaStream_t st) {
  return p.given ? launch_mplane_tg<NB, LD, true, TX>(p, s, grid, st) : launch_mplane_tg<NB, LD, false, TX>(p, s, grid, st);
}

cudaError_t launch_mplane(const PlaneArgs& p0, int grid, bool bf16, cudaStream_t st) {
  PlaneArgs p = p0;
  const int r = std::max(p.r3, p.r4);
  const MpShape s = mp_shape(p.H, p.W, r, bf16);
  p.pitch = s.pb;
  const bool quads = p.W % 4 == 0 && ((int64_t)p.H * p.W * (bf16 ? 2 : 4)) % 16 == 0 && (reinterpret_cast<uintptr_t>(p.X) & 15u) == 0;
  if (bf16 && !quads) return cudaErrorInvalidValue;  // the caller takes another kernel
  ProfScope prof(ASI_K_EXPAND, st, (double)p.n_planes * p.H * p.W * (bf16 ? 2 : 4));
#define ASI_MP(NB_)                                                        \
  if (bf16) return launch_mplane_t<NB_, 0, __nv_bfloat16>(p, s, grid, st);   \
  if (quads) return launch_mplane_t<NB_, 0, float>(p, s, grid, st);          \
  return launch_mplane_t<NB_, 1, float>(p, s, grid, st)
  if (r <= 4) { ASI_MP(1); }
  ASI_MP(2);
#undef ASI_MP
}

}  // namespace asi
