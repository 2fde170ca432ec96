// Tensor-core kernels (sm_100a: tcgen05.mma, TMEM accumulator, TMA operand staging) for the steps of the
// path that are plain dense contractions: products of a bf16 tensor with a wide fp32 factor (16..64
// columns) in Algorithm 1 on token layers (B x N x D activations),
//   kTcLast         Y[q][j]     = sum_k X[q][k] U[k][j]          V_3 = A_(3)^T U_3, first core product
//   kTcLastExpand   P[k][j]     = sum_q X[q][k] V[q][j]          P_3 = A_(3) V_3 (split-K partials)
//   kTcToken        V[o][i][j]  = sum_k X[o][k][i] U[k][j]       V_2 = A_(2)^T U_2, dY x_2 U_2^T
//   kTcTokenExpand  P[k][j]     = sum_{o,i} X[o][k][i] V[o][i][j]  P_2 = A_(2) V_2 (split-K partials)
// X is exact in bf16; the fp32 factor (U or V) is split into three bf16 terms (24 mantissa bits), so one
// MMA of width 3 n per k-step (the three terms stacked as operand rows) yields three partial products in
// TMEM whose sum reproduces the fp32 product to fp32 rounding.
//
// The stacked operand [3 n][K] (bf16, K contiguous: hi rows, then mid, then lo) of a factor U is written by
// k_tc_split (one launch for all factors of a call; k_orth_apply writes that of a new factor itself); that of
// V_m is written by the projection's own epilogue, so V_m exists only in the form its expansion reads.
//
// k_tc_group runs up to three products in one launch (a CTA finds its product in a table).  One CTA owns a
// 128-row tile of Y and a share of K in chunks of 64, its warps in three roles that meet only through mbarriers:
//   * a producer thread keeps the stages full, each the X tile [128 x 64] and the operand tile
//     [3 n x 64] (cp.async.bulk.tensor, 128-byte swizzle);
//   * an issuer thread launches 4 k-steps of tcgen05.mma (M = 128, N = 3 n, K = 16) per chunk and commits
//     them to the mbarrier that frees the stage;
//   * eight warps read the three accumulator groups with tcgen05.ld (lane = row) and add them to registers after every
//     four chunks, because the unit's own sums truncate (a contraction of 2400 left in TMEM had eight times the error: 1.0e-6
//     against 1.2e-7); two accumulators where they fit, so that the next chunks do not wait.  A CTA of a product with
//     many tiles takes several, and the stages fill with the next one's chunks meanwhile.
// A launch uses clusters of 1, 2 or 4 CTAs: the CTAs of a cluster share one tile of a product whose contraction
// is long (each takes a quarter of K, the partial tiles meet in distributed shared memory in rank order) or own
// different tiles.  Stage count and TMEM columns follow n so that two CTAs share an SM: what bounds these products
// is latency -- few tiles, a prologue and an epilogue per tile, bytes in flight -- not the tensor pipe.
// Every wait has a time limit; on expiry the kernel records ASI_ERR_TIMEOUT in the workspace's status word, gives the copies and
// products in flight the limit once more, frees its TMEM and returns.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <mutex>

#include "asi_internal.h"

namespace asi {

namespace {

constexpr int kTcWorkers = 8;       // epilogue warps
constexpr int kTcThreads = (kTcWorkers + 2) * 32;   // + the MMA issuer warp and the TMA producer warp
constexpr int kTcM = 128;          // rows of Y per CTA (= TMEM lanes)
constexpr int kTcKC = 64;          // k per chunk: 64 bf16 = one 128-byte swizzle row
constexpr int kTcMaxStages = 4;
constexpr int kTcSeg = 4;          // chunks that add up in TMEM before their sum goes to registers
constexpr int kTcNMax = 64;
constexpr uint32_t kTileA = kTcM * kTcKC * 2;       // 16 KB

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
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
// waits for the phase with the given parity; gives up after 2e9 cycles (a second or so; a millisecond with the test hook, whose
// producer arms its barriers and issues no copy).  The limit is on the SM's own clock: a read of %globaltimer costs over 600
// cycles, and every chunk that was not there yet paid one
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, int stall) {
  if (mbar_try_wait(bar, parity)) return true;
  const long long t0 = clock64();
  for (uint32_t it = 0; it < (1u << 28); ++it) {
    if (mbar_try_wait(bar, parity)) return true;
    if ((it & 1023u) == 1023u && clock64() - t0 > (stall ? 2000000ll : 2000000000ll)) return false;
  }
  return false;
}
__device__ __forceinline__ void tma_load_2d(void* dst, const CUtensorMap* map, int x, int y, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(
          smem_u32(dst)),
      "l"(map), "r"(x), "r"(y), "r"(smem_u32(bar))
      : "memory");
}
__device__ __forceinline__ void tma_load_3d(void* dst, const CUtensorMap* map, int x, int y, int z, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(
          smem_u32(dst)),
      "l"(map), "r"(x), "r"(y), "r"(z), "r"(smem_u32(bar))
      : "memory");
}
// shared-memory matrix descriptor of a 128-byte-swizzled operand (start address, leading and stride byte
// offsets in 16-byte units; descriptor version 1).  K-major: rows of 128 bytes along K, groups of 8 rows
// 1024 bytes apart (stride offset), the leading offset is unused.  MN-major: rows of 128 bytes along M/N
// (64 bf16), one row per K index, groups of 8 K-rows 1024 bytes apart (stride offset), the next 64 M/N
// elements `lbo` bytes further (leading offset).
__device__ __forceinline__ uint64_t smem_desc_sw128(uint32_t addr, uint32_t lbo_bytes = 16) {
  uint64_t d = 0;
  d |= (uint64_t)((addr >> 4) & 0x3FFF);
  d |= (uint64_t)((lbo_bytes >> 4) & 0x3FFF) << 16;
  d |= (uint64_t)(1024 >> 4) << 32;       // stride byte offset
  d |= (uint64_t)1 << 46;                 // version
  d |= (uint64_t)2 << 61;                 // 128-byte swizzle
  return d;
}
// instruction descriptor of kind::f16: fp32 accumulator, bf16 x bf16, B K-major, A K-major or MN-major
__device__ __forceinline__ uint32_t instr_desc_bf16(int M, int N, bool a_mn_major) {
  return (1u << 4) | (1u << 7) | (1u << 10) | (a_mn_major ? (1u << 15) : 0u) | ((uint32_t)(N >> 3) << 17) |
         ((uint32_t)(M >> 4) << 24);
}
__device__ __forceinline__ void umma_bf16(uint32_t tmem_d, uint64_t da, uint64_t db, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, {%5, %5, %5, %5}, p;\n\t}" ::"r"(tmem_d),
      "l"(da), "l"(db), "r"(idesc), "r"(acc), "r"(0u)    // no output lane disabled
      : "memory");
}
__device__ __forceinline__ void umma_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
               : "memory");
}
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t (&v)[8]) {   // 8 columns of this thread's lane
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
               : "r"(taddr)
               : "memory");
}
// Bt[(t*n + j) * ldb + k] = t-th bf16 term of U[k][j] (hi, mid, lo: U = hi + mid + lo to 24 bits), for every factor
// of the call in one launch
__global__ void __launch_bounds__(256) k_tc_split(const __grid_constant__ TcSplitArgs p) {
  __shared__ float tile[32][33];
  pdl_wait();                                        // often the first kernel of a call: its dependents start behind all older work
  pdl_launch_dependents();
  if (p.clear && blockIdx.x == 0) p.clear[threadIdx.x] = 0;
  int q = 0;
  while (q + 1 < p.n && (int)blockIdx.x >= p.m[q + 1].first) ++q;
  const TcSplitMat& m = p.m[q];
  const int t = (int)blockIdx.x - m.first, nk = (m.K + 31) / 32;
  const int k0 = (t % nk) * 32, j0 = (t / nk) * 32;
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  float v[4];
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const int k = k0 + ty + 8 * r, j = j0 + tx;
    v[r] = __ldg(m.U + ((k < m.K && j < m.nv) ? (int64_t)k * m.nv + j : 0));
  }
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const int k = k0 + ty + 8 * r, j = j0 + tx;
    tile[ty + 8 * r][tx] = (k < m.K && j < m.nv) ? v[r] : 0.f;           // columns nv..N-1 of the operand are zero
  }
  __syncthreads();
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const int j = j0 + ty + 8 * r, k = k0 + tx;
    if (j < m.N && k < m.K) tc_store_terms(m.Bt, m.N, m.ldb, j, k, tile[tx][ty + 8 * r]);
  }
}

// How the X operand of D[m][n] = sum_k A(m, k) B[n][k] is laid out in memory:
//   kTcLast        X[m][k], k contiguous: one box [128 m x 64 k] (K-major);            CTA (mt, split of K)
//   kTcLastExpand  X[k][m], m contiguous: two boxes [64 k x 64 m] (MN-major);          CTA (mt, split of K)
//   kTcToken       X[o][k][m], m contiguous, one o per CTA row: two boxes (MN-major);  CTA (mt, o)
//   kTcTokenExpand X[o][m][i], i contiguous, K = (o, i) flattened: one box (K-major);  CTA (mt, split of K)
// Rows of a box that fall outside the tensor are zero-filled by TMA.
enum TcMode { kTcLast = 0, kTcLastExpand = 1, kTcToken = 2, kTcTokenExpand = 3 };

struct TcProb {
  CUtensorMap mapX, mapB;
  float* Y;            // fp32 result [M][ldy] of outer index / split s at Y + s * y_split (null: Bt instead)
  __nv_bfloat16* Bt;   // the result as a stacked operand: row m of outer index o is k = o * M + m
  int64_t y_split, ldb;
  int mode, M, N, nv, K, ldy;
  int k_per_split;     // multiple of 64; second tile index s contracts [s * k_per_split, min(K, (s + 1) * k_per_split))
  int inner;           // kTcTokenExpand: K enumerates (o, i) with i < inner (a multiple of 64)
  int mt;              // 128-row tiles
  int ksp;             // CTAs that share a tile (1 or the cluster size)
  int first;           // first CTA of the product in the launch (a multiple of the cluster size)
  int n_cta;
  int tpc;             // tiles a CTA takes one after another (1 where CTAs share a tile)
  int tiles;
  int nbuf;            // accumulators in TMEM: two where two CTAs' pairs fit an SM
  int nst;             // stages: as many as its operand width leaves room for beside a second CTA
};
struct TcGroup {
  TcProb p[3];
  int* status;         // status word of the caller's workspace (may be null): ASI_ERR_TIMEOUT when a wait expires
  int np, tmem_cols, cs;
  int stall;           // test hook: no copies, short waits
};

__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ float4 ld_cluster4(uint32_t local_addr, uint32_t rank) {
  uint32_t ra;
  float4 v;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(local_addr), "r"(rank));
  asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
               : "r"(ra)
               : "memory");
  return v;
}

// four columns col.. of result row m (outer index or split s)
__device__ __forceinline__ void tc_store4(const TcProb& p, int s, int m, int col, float4 v) {
  if (m >= p.M || col >= p.N) return;
  if (p.Y) {
    if (col < p.nv) *reinterpret_cast<float4*>(p.Y + (int64_t)s * p.y_split + (int64_t)m * p.ldy + col) = v;
  } else {
    const int64_t k = (int64_t)s * p.M + m;          // columns nv.. are exact zeros (their factor columns are)
    tc_store_terms(p.Bt, p.N, p.ldb, col, k, v.x);
    tc_store_terms(p.Bt, p.N, p.ldb, col + 1, k, v.y);
    tc_store_terms(p.Bt, p.N, p.ldb, col + 2, k, v.z);
    tc_store_terms(p.Bt, p.N, p.ldb, col + 3, k, v.w);
  }
}

__global__ void __launch_bounds__(kTcThreads, 2) k_tc_group(const __grid_constant__ TcGroup g) {
  extern __shared__ __align__(1024) uint8_t tc_smem[];
  int q = 0;
  while (q + 1 < g.np && (int)blockIdx.x >= g.p[q + 1].first) ++q;
  const TcProb& p = g.p[q];
  const int nst = p.nst, N = p.N, nbuf = p.nbuf;
  const uint32_t tile_b = (uint32_t)(3 * N) * 128u;     // operand tile: 3 N rows of 64 bf16
  const uint32_t stage = kTileA + tile_b;               // 1024-byte multiples: N is a multiple of 16
  // carve-up: stages, then barriers
  uint8_t* base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(tc_smem) + 1023) & ~(uintptr_t)1023);
  __shared__ __align__(8) uint64_t full[kTcMaxStages], s_free[kTcMaxStages], done[2], acc_free[2], drained[1];
  __shared__ uint32_t tmem_slot[1];

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const bool a_mn = p.mode == kTcLastExpand || p.mode == kTcToken;
  const int cta = (int)blockIdx.x - p.first;
  const bool live = cta < p.n_cta;                      // padding CTAs of the last cluster only take the barriers
  const int rank = p.ksp > 1 ? (int)cluster_rank() : 0;
  // the tiles of this CTA: the first one and how many (one that is shared, or up to tpc neighbours)
  const int tile0 = p.ksp > 1 ? cta / p.ksp : cta * p.tpc;
  const int ntile = !live ? 0 : (p.ksp > 1 ? 1 : (p.tiles - tile0 < p.tpc ? p.tiles - tile0 : p.tpc));
  struct Tile { int row0, s, k_begin, nchunk; };
  auto tile_of = [&](int t) {
    Tile x;
    x.row0 = ((tile0 + t) % p.mt) * kTcM;
    x.s = (tile0 + t) / p.mt;                           // outer index (kTcToken) or split of K
    x.k_begin = p.mode == kTcToken ? 0 : x.s * p.k_per_split;
    int k_end = (p.mode == kTcToken || p.K - x.k_begin < p.k_per_split) ? p.K : x.k_begin + p.k_per_split;
    if (k_end < x.k_begin) k_end = x.k_begin;
    x.nchunk = (k_end - x.k_begin + kTcKC - 1) / kTcKC; // a ragged last chunk is zero-filled by TMA
    if (p.ksp > 1) {
      const int per = (x.nchunk + p.ksp - 1) / p.ksp;
      x.k_begin += rank * per * kTcKC;
      x.nchunk = x.nchunk - rank * per < per ? x.nchunk - rank * per : per;
      if (x.nchunk < 0) x.nchunk = 0;
    }
    return x;
  };

  if (tid == 0) {
    for (int i = 0; i < nst; ++i) { mbar_init(full + i, 1); mbar_init(s_free + i, 1); }
    for (int i = 0; i < 2; ++i) { mbar_init(done + i, 1); mbar_init(acc_free + i, kTcWorkers); }
    mbar_init(drained, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {                                      // TMEM: fp32 columns x 128 lanes (3 N are used)
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(g.tmem_cols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem_d = *tmem_slot;
  pdl_wait();

  // The three bf16 terms of the factor are stacked along the operand's rows: one MMA of width 3 N per
  // k-step reads the X tile once and leaves the three partial products in three column groups of TMEM.
  bool ok = true;                                       // this thread's waits so far
  int loads = 0;                                        // chunks that this thread has brought (the producer)
  const int PN = N + 4;                                 // pitch of the exchanged tile: rows four banks apart
  float* xch = reinterpret_cast<float*>(base);          // [128][PN], over the stages of a tile that is shared
  if (warp == kTcWorkers) {
    // ---- MMA issuer (one thread): 4 k-steps per chunk, then the commit that frees the stage
    if (lane == 0) {
      const uint32_t idesc = instr_desc_bf16(kTcM, 3 * N, a_mn);
      const uint32_t a_base = smem_u32(base);
      const uint64_t a_step = a_mn ? 128 : 2;           // a k-step is 16 bf16: 32 bytes inside the swizzle row of a
      int st = 0, seg = 0;                              // K-major tile, 16 rows (2048 bytes) of an MN-major tile
      uint32_t ph = 0;                                  // (start-address field in 16-byte units)
#pragma unroll 1
      for (int t = 0; t < ntile && ok; ++t) {
        const int nchunk = tile_of(t).nchunk;
#pragma unroll 1
        for (int c0 = 0; c0 < nchunk && ok; c0 += kTcSeg, ++seg) {
          const int buf = nbuf == 2 ? seg & 1 : 0, turn = nbuf == 2 ? seg >> 1 : seg;
          if (turn > 0) {                               // the workers have read what the buffer held
            ok = mbar_wait(acc_free + buf, (uint32_t)(turn + 1) & 1u, g.stall);
            if (!ok) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          }
          const int c1 = c0 + kTcSeg < nchunk ? c0 + kTcSeg : nchunk;
#pragma unroll 1
          for (int c = c0; c < c1; ++c) {
            ok = mbar_wait(full + st, ph, g.stall);
            if (!ok) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint64_t da0 = smem_desc_sw128(a_base + st * stage, a_mn ? kTileA / 2 : 16);
            const uint64_t db0 = smem_desc_sw128(a_base + st * stage + kTileA);
#pragma unroll
            for (int ks = 0; ks < kTcKC / 16; ++ks)
              umma_bf16(tmem_d + (uint32_t)(buf * 3 * N), da0 + (uint64_t)ks * a_step, db0 + (uint64_t)(ks * 2), idesc,
                        ((c - c0) | ks) ? 1u : 0u);
            umma_commit(s_free + st);
            if (++st == nst) { st = 0; ph ^= 1u; }
          }
          if (ok) umma_commit(done + buf);
        }
      }
    }
  } else if (warp == kTcWorkers + 1) {
    // ---- TMA producer (one thread): keeps the stages full, across tiles
    if (lane == 0) {
      int st = 0;
      uint32_t ph = 1;
#pragma unroll 1
      for (int t = 0; t < ntile && ok; ++t) {
        const Tile x = tile_of(t);
#pragma unroll 1
        for (int c = 0; c < x.nchunk && ok; ++c, ++loads) {
          if (loads >= nst) ok = mbar_wait(s_free + st, ph, g.stall);
          if (!ok) break;
          uint8_t* As = base + st * stage;
          mbar_expect_tx(full + st, stage);
          if (g.stall) {
            if (++st == nst) { st = 0; ph ^= 1u; }
            continue;
          }
          const int kc = x.k_begin + c * kTcKC;
          if (p.mode == kTcLastExpand) {
            tma_load_2d(As, &p.mapX, x.row0, kc, full + st);
            tma_load_2d(As + kTileA / 2, &p.mapX, x.row0 + 64, kc, full + st);
          } else if (p.mode == kTcToken) {
            tma_load_3d(As, &p.mapX, x.row0, kc, x.s, full + st);
            tma_load_3d(As + kTileA / 2, &p.mapX, x.row0 + 64, kc, x.s, full + st);
          } else if (p.mode == kTcTokenExpand) {
            const int o = kc / p.inner;
            tma_load_3d(As, &p.mapX, kc - o * p.inner, x.row0, o, full + st);
          } else {
            tma_load_2d(As, &p.mapX, kc, x.row0, full + st);
          }
          tma_load_2d(As + kTileA, &p.mapB, kc, 0, full + st);
          if (++st == nst) { st = 0; ph ^= 1u; }
        }
      }
    }
  } else {
    // ---- workers: thread = row: warp w reads lanes 32 (w % 4) ..., warps 0-3 the columns [0, N/2), warps 4-7 the rest;
    // the loads of the next tile are under way meanwhile
    const int half = N >> 1;                            // 8, 16, 24 or 32 columns per warp
    const int col0 = (warp >> 2) * half;
    const int r = (warp & 3) * 32 + lane;
    const uint32_t taddr = tmem_d + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)col0;
    int seg = 0;
#pragma unroll 1
    for (int t = 0; t < ntile && ok; ++t) {
      const Tile x = tile_of(t);
      float sum[kTcNMax / 2];                           // an empty share of K adds nothing
#pragma unroll
      for (int i = 0; i < kTcNMax / 2; ++i) sum[i] = 0.f;
#pragma unroll 1
      for (int c0 = 0; c0 < x.nchunk; c0 += kTcSeg, ++seg) {
        const int buf = nbuf == 2 ? seg & 1 : 0, turn = nbuf == 2 ? seg >> 1 : seg;
        ok = mbar_wait(done + buf, (uint32_t)turn & 1u, g.stall);   // every reader of TMEM observes the completed phase
        if (__any_sync(0xffffffffu, ok ? 0 : 1)) ok = false;
        if (!ok) break;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
        for (int cc = 0; cc < kTcNMax / 2; cc += 8)
          if (cc < half) {
            uint32_t h[8], m[8], l[8];
            const uint32_t at = taddr + (uint32_t)(buf * 3 * N + cc);
            tmem_ld8(at, h);
            tmem_ld8(at + (uint32_t)N, m);
            tmem_ld8(at + (uint32_t)(2 * N), l);
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
            for (int i = 0; i < 8; ++i)                 // small terms first
              sum[cc + i] += (__uint_as_float(l[i]) + __uint_as_float(m[i])) + __uint_as_float(h[i]);
          }
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncwarp();
        if (lane == 0) mbar_arrive(acc_free + buf);     // all read: the buffer is free
      }
      if (!ok) break;
#pragma unroll
      for (int cc = 0; cc < kTcNMax / 2; cc += 8)
        if (cc < half) {
          const float4 v0 = make_float4(sum[cc], sum[cc + 1], sum[cc + 2], sum[cc + 3]);
          const float4 v1 = make_float4(sum[cc + 4], sum[cc + 5], sum[cc + 6], sum[cc + 7]);
          if (p.ksp > 1) {
            *reinterpret_cast<float4*>(xch + r * PN + col0 + cc) = v0;
            *reinterpret_cast<float4*>(xch + r * PN + col0 + cc + 4) = v1;
          } else {
            tc_store4(p, x.s, x.row0 + r, col0 + cc, v0);
            tc_store4(p, x.s, x.row0 + r, col0 + cc + 4, v1);
          }
        }
    }
  }
  const bool fail = __syncthreads_or(ok ? 0 : 1) != 0;
  pdl_launch_dependents();
  if (fail) {                                           // what is in flight gets the limit once more
    if (tid == 0 && g.status) atomicMax(g.status, (int)ASI_ERR_TIMEOUT);
    if (warp == kTcWorkers && lane == 0) {
      umma_commit(drained);
      mbar_wait(drained, 0, g.stall);
    } else if (warp == kTcWorkers + 1 && lane == 0) {
      for (int i = 0; i < nst; ++i)
        if (loads > i) mbar_wait(full + i, (uint32_t)((loads - 1 - i) / nst) & 1u, g.stall);   // the stage's last chunk
    }
    __syncwarp();
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_d), "r"(g.tmem_cols) : "memory");
  if (p.ksp > 1) {                                      // uniform in a cluster: its CTAs belong to one product
    // the shares of a tile meet: CTA `rank` adds the rows [rank * 128 / ksp, ..) in rank order
    cluster_sync_all();
    // at most four items a thread (128 N / (4 ksp) <= 1024); the CTA tells its peers that it is done with their tiles
    // before it stores, so that the barrier does not wait for the stores as well
    const int rows = kTcM / p.ksp, r0 = rank * rows, items = rows * (N / 4);
    const Tile x = tile_of(0);
    const bool meet = live && !fail;
    float4 sum[4];
    if (meet) {
      const uint32_t xa = smem_u32(xch);
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int e = tid + u * kTcThreads, ec = e < items ? e : 0;
        const int r = r0 + ec % rows, c4 = ec / rows;   // lanes = neighbouring rows: coalesced operand stores
        const uint32_t a = xa + (uint32_t)(r * PN + 4 * c4) * 4u;
        sum[u] = ld_cluster4(a, 0);
#pragma unroll
        for (int t = 1; t < 4; ++t)
          if (t < p.ksp) {
            const float4 v = ld_cluster4(a, (uint32_t)t);
            sum[u].x += v.x; sum[u].y += v.y; sum[u].z += v.z; sum[u].w += v.w;
          }
      }
    }
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    if (meet) {
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int e = tid + u * kTcThreads;
        if (e < items) tc_store4(p, x.s, x.row0 + r0 + e % rows, 4 * (e / rows), sum[u]);
      }
    }
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");   // no CTA leaves while its tile is being read
  }
}

using EncodeFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                              const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                              CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeFn encode_fn() {
  static EncodeFn fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeFn>(p);
  });
  return fn;
}


bool encode_bf16_map(CUtensorMap* map, const void* base, int rank, const cuuint64_t* dims, const cuuint64_t* strides,
                     const cuuint32_t* box) {
  EncodeFn enc = encode_fn();
  if (!enc) return false;
  const cuuint32_t estr[3] = {1, 1, 1};
  return enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, (cuuint32_t)rank, const_cast<void*>(base), dims, strides, box,
             estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

int pad16(int n) { return (n + 15) / 16 * 16; }
int64_t pad64(int64_t k) { return (k + 63) / 64 * 64; }

bool operand_map(CUtensorMap* map, const __nv_bfloat16* Bt, int64_t K, int N) {
  const cuuint64_t dims[2] = {(cuuint64_t)K, (cuuint64_t)(3 * N)};
  const cuuint64_t strides[1] = {(cuuint64_t)pad64(K) * 2};
  const cuuint32_t box[2] = {(cuuint32_t)kTcKC, (cuuint32_t)(3 * N)};
  return encode_bf16_map(map, Bt, 2, dims, strides, box);
}
}  // namespace

// bytes of the stacked operand of a [K x n] factor
size_t tc_operand_bytes(int64_t K, int n) { return (size_t)3 * pad16(n) * pad64(K) * 2; }
int64_t tc_operand_ld(int64_t K) { return pad64(K); }
int tc_operand_n(int n) { return pad16(n); }

// Which products of mode (O, a, I) with n columns run here: 0 none, 1 the last mode, 2 a mode with inner extent
int tc_kind(int64_t O, int64_t a, int64_t I, int n) {
  // the kernel counts columns in 32 bits up to the end of the last split: 2^24 is more than a split of such a tensor that
  // fits the device
  constexpr int64_t most = (1ll << 31) - (1ll << 24);
  if (n % 4 != 0 || n < 16 || n > kTcNMax || a >= most || O * I >= most) return 0;
  if (I == 1) return a % 64 == 0 && O >= kTcM ? 1 : 0;
  return I % 64 == 0 && O < 65536 ? 2 : 0;
}

void tc_add_split(TcSplitArgs* p, const float* U, int64_t K, int n, void* Bt) {
  TcSplitMat& m = p->m[p->n++];
  m.U = U;
  m.Bt = static_cast<__nv_bfloat16*>(Bt);
  m.K = (int)K;
  m.nv = n;
  m.N = pad16(n);
  m.ldb = pad64(K);
}

cudaError_t launch_tc_split(TcSplitArgs& p, cudaStream_t st) {
  int first = 0;
  for (int q = 0; q < p.n; ++q) {
    p.m[q].first = first;
    first += ((p.m[q].K + 31) / 32) * ((p.m[q].N + 31) / 32);
  }
  return launch_pdl(k_tc_split, dim3((unsigned)first), dim3(256), 0, st, p);
}

// One launch over the products of `c` (all with operands already split).  cudaErrorNotSupported: a tensor map could
// not be made (nothing was launched).
cudaError_t launch_tc_group(const TcCall* c, int n, int* status, int stall, cudaStream_t st) {
  if (n < 1 || n > 3) return cudaErrorInvalidValue;
  TcGroup g;
  g.np = n;
  g.status = status;
  g.stall = stall;
  double bytes = 0.0;
  int64_t tiles[3];
  int chunks[3];
  for (int q = 0; q < n; ++q) {
    const TcCall& k = c[q];
    TcProb& p = g.p[q];
    p.N = pad16(k.n);
    p.nv = k.n;
    p.inner = (int)k.I;
    p.ldb = k.out_ld;
    p.Bt = static_cast<__nv_bfloat16*>(k.out_bt);
    p.Y = k.Y;
    p.ldy = k.n;
    const int64_t Q = k.O * k.I;
    bool ok;
    int64_t second = 1;
    if (k.expand) {
      p.mode = k.I == 1 ? kTcLastExpand : kTcTokenExpand;
      p.M = (int)k.a;
      p.K = (int)Q;
      p.k_per_split = (int)k.q_per_split;
      p.y_split = k.a * k.n;
      second = k.nsplit;
      chunks[q] = (int)((std::min<int64_t>(k.q_per_split, Q) + kTcKC - 1) / kTcKC);
    } else {
      p.mode = k.I == 1 ? kTcLast : kTcToken;
      p.M = (int)(k.I == 1 ? Q : k.I);
      p.K = (int)k.a;
      p.k_per_split = (int)pad64(k.a);
      p.y_split = k.I * k.n;
      second = k.I == 1 ? 1 : k.O;
      chunks[q] = (int)((k.a + kTcKC - 1) / kTcKC);
    }
    if (k.I == 1) {
      const cuuint64_t dims[2] = {(cuuint64_t)k.a, (cuuint64_t)Q};
      const cuuint64_t strides[1] = {(cuuint64_t)k.a * 2};
      const cuuint32_t box[2] = {64, (cuuint32_t)(k.expand ? 64 : kTcM)};
      ok = encode_bf16_map(&p.mapX, k.X, 2, dims, strides, box);
    } else {
      const cuuint64_t dims[3] = {(cuuint64_t)k.I, (cuuint64_t)k.a, (cuuint64_t)k.O};
      const cuuint64_t strides[2] = {(cuuint64_t)k.I * 2, (cuuint64_t)k.a * k.I * 2};
      const cuuint32_t box[3] = {64, (cuuint32_t)(k.expand ? kTcM : 64), 1};
      ok = encode_bf16_map(&p.mapX, k.X, 3, dims, strides, box);
    }
    ok = ok && operand_map(&p.mapB, static_cast<const __nv_bfloat16*>(k.bt), p.K, p.N);
    if (!ok) return cudaErrorNotSupported;
    p.mt = (p.M + kTcM - 1) / kTcM;
    tiles[q] = p.mt * second;
    bytes += 2.0 * (double)k.a * Q;
  }
  // A product with few tiles and a long contraction shares each tile between the CTAs of a cluster.  Few: below 64, where it
  // leaves most SMs idle.  (At 200 a step's expansions of 64 + 64 tiles ran as 512 CTAs of four chunks, two waves of set-up and
  // exchange: ViT-Base MLP 245 us, LLM-shaped tokens 310; at 64, with sums of four chunks in registers, 227 and 283; without
  // clusters single layers lose 4 %.)
  constexpr int kFewTiles = 64;
  int cs = 1;
  for (int q = 0; q < n; ++q)
    while (cs < 4 && tiles[q] * cs < kFewTiles && chunks[q] >= 8 * cs) cs *= 2;
  auto shares = [&](int q) { return cs > 1 && tiles[q] < kFewTiles && chunks[q] >= 4 * cs; };
  // Tiles in turn where the launch has more than the machine holds at a time (two CTAs an SM), what the shared tiles leave of
  // it but 200 at least: the next tile's loads run under this one's epilogue, and the set-up (4 k of 12 k cycles) is paid
  // once (ViT-Base MLP 3 % against a count per product)
  int64_t shared = 0, plain = 0;
  for (int q = 0; q < n; ++q) (shares(q) ? shared : plain) += tiles[q] * (shares(q) ? cs : 1);
  const int64_t room = std::max<int64_t>(200, 296 - shared);
  int first = 0;
  for (int q = 0; q < n; ++q) {
    TcProb& p = g.p[q];
    p.ksp = shares(q) ? cs : 1;
    p.first = first;
    p.tiles = (int)tiles[q];
    p.tpc = p.ksp > 1 ? 1 : (int)std::min<int64_t>(8, (plain + room - 1) / room);
    p.n_cta = p.ksp > 1 ? (int)tiles[q] * p.ksp : (p.tiles + p.tpc - 1) / p.tpc;
    first += (p.n_cta + cs - 1) / cs * cs;
  }
  g.cs = cs;
  int cols = 0;
  for (int q = 0; q < n; ++q) {
    g.p[q].nbuf = 6 * g.p[q].N <= 256 ? 2 : 1;
    cols = std::max(cols, g.p[q].nbuf * 3 * g.p[q].N);
  }
  g.tmem_cols = cols <= 64 ? 64 : (cols <= 128 ? 128 : 256);
  // every product its own stage count: with those of the widest one (two at 64 columns) the four chunks of a narrower
  // product's tile took one round trip more
  size_t smem = 0;
  for (int q = 0; q < n; ++q) {
    TcProb& p = g.p[q];
    p.nst = p.N <= 16 ? 4 : (p.N <= 48 ? 3 : 2);
    smem = std::max(smem, 1024 + (size_t)p.nst * (kTileA + 3 * p.N * 128));
    smem = std::max(smem, 1024 + (size_t)kTcM * (p.N + 4) * 4);
  }
  const cudaError_t e = opt_in_smem(reinterpret_cast<const void*>(k_tc_group), smem);
  if (e != cudaSuccess) return e;
  ProfScope prof(c[0].expand ? ASI_K_EXPAND : ASI_K_MODEPROD, st, bytes);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)first);
  cfg.blockDim = dim3(kTcThreads);
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
  return cudaLaunchKernelEx(&cfg, k_tc_group, g);
}

}  // namespace asi
