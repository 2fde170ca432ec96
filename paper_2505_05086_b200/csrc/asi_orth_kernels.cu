// Orthogonalize(P_m) for ranks up to 64: Cholesky-QR with the Gram matrix, the factorisation and the row
// products in fp64 (in exact arithmetic the Gram-Schmidt basis of the columns of P).  Two launches for all modes:
//
//   k_orth_factor : CTA (c, m) sums the split partials of its rows of P_m in fp64 in split order and forms its
//                   share of G = P^T P; the eight CTAs of a cluster add their shares through distributed shared
//                   memory, the last cluster of a mode adds the clusters' shares (both in index order) and factors
//                   G = R^T R once per mode, carrying the identity along so that Y = R^{-T} falls out of the same
//                   elimination.
//   k_orth_apply  : U = P R^{-1}, i.e. U[k][j] = sum_{i <= j} P[k][i] Y[j][i]: a plain product without a chain.
//
// What bounds it: latency.  The elimination is a serial chain of r pivots (a reciprocal square root and two dependent
// multiply-adds each, ~90 cycles); around it every step is a round trip to L2 (~1000 cycles under load).  So four
// columns share one step, the two pivot warps work on step p + 1 while the other eight still update the rows behind
// step p, shares meet inside a cluster instead of through memory, and the loads of a sum are issued in batches that
// fit the chunk's shape.  The code is kept small: most of it runs once per launch, and straight-line code costs an
// instruction fetch per 128 bytes.
// A pivot d_j with d_j <= 1e-12 * trace(G), i.e. a Gram-Schmidt residual below 1e-6 * ||P||_F, raises
// ASI_ERR_RANK_DEFICIENT in the status word.
#include <cooperative_groups.h>

#include <algorithm>

#include "asi_internal.h"

namespace asi {

namespace {

constexpr int kOT = 320;                 // threads per CTA: two pivot warps and eight update warps
constexpr int kPivot = 64;               // threads of the pivot warps
constexpr int kAT = 256;                 // threads of k_orth_apply
constexpr int kOrthMaxRows = 64;         // rows of P per share, at most
constexpr int kOrthCluster = 8;          // chunks whose shares meet in distributed shared memory
constexpr int kMaxPacked = 136 * 16;     // packed upper triangle of a 64 x 64 matrix, in 4 x 4 blocks

__device__ __forceinline__ void named_sync(int id, int n) { asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory"); }
__device__ __forceinline__ void named_arrive(int id, int n) { asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(n) : "memory"); }

// element (i, k), k >= i, of an upper triangle in 4 x 4 blocks, nb block rows: the blocks' elements of one place lie side by side, so
// that threads with neighbouring blocks write them without bank conflicts
__device__ __forceinline__ int packed_at(int i, int k, int nb) {
  const int bi = i >> 2, bk = k >> 2;
  return ((i & 3) * 4 + (k & 3)) * (nb * (nb + 1) / 2) + bi * nb - bi * (bi - 1) / 2 + bk - bi;
}

// G = R^T R and Y = R^{-T} by one elimination on an r x r array T (ranks up to 16 NX): entries k >= i start as G,
// the rest as zero; row i of Y takes the place of the entries k <= i.  Update thread (ti, tj) keeps
// T[ti + 16 x][tj + 16 y] in registers and hands the four pivot rows of the next step over in Prow [4][64]; pivot
// thread k solves column k of them and hands rows of R and Y back in W[step & 1] [4][64].  Y goes to Yg (row-major,
// zero above the diagonal).
template <int NX>
__device__ __forceinline__ void eliminate(const double* Gq, double* Prow, double* W, double floor_d, int r,
                                          double* __restrict__ Yg, int* status) {
  const int tid = threadIdx.x, nb = (r + 3) >> 2;
  if (tid < kPivot) {
    bool bad = false;
#pragma unroll 1
    for (int p0 = 0; p0 < r; p0 += 4) {
      named_sync(1, kOT);                            // Prow holds the rows p0 .. p0 + 3
      double D[4][4], w[4];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int k = i; k < 4; ++k) D[i][k] = Prow[i * kQRMaxRank + p0 + k];
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        w[c] = Prow[c * kQRMaxRank + tid];
        if (tid >= p0 && tid < p0 + 4) w[c] = (tid == p0 + c) ? 1.0 : 0.0;     // the identity's columns p0 .. p0 + 3
        if (p0 + c >= r) D[c][c] = 1.0;              // rows past the end: identity
      }
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        double d = D[c][c];
        const bool low = p0 + c < r && !(d > floor_d);
        bad |= low;
        if (low) d = floor_d > 0.0 ? floor_d : 1.0;
        const double inv = rsqrt(d);
        w[c] *= inv;
#pragma unroll
        for (int k = c + 1; k < 4; ++k) D[c][k] *= inv;
#pragma unroll
        for (int i = c + 1; i < 4; ++i) {
          w[i] = fma(-D[c][i], w[c], w[i]);
#pragma unroll
          for (int k = i; k < 4; ++k) D[i][k] = fma(-D[c][i], D[c][k], D[i][k]);
        }
      }
      double* Wp = W + ((p0 >> 2) & 1) * (4 * kQRMaxRank) + tid;
#pragma unroll
      for (int c = 0; c < 4; ++c) Wp[c * kQRMaxRank] = w[c];
      named_arrive(2, kOT);                          // W of this step is there
      if (tid < r) {                                 // rows p0 .. p0 + 3 of Y are final
#pragma unroll
        for (int c = 0; c < 4; ++c)
          if (p0 + c < r) Yg[(int64_t)(p0 + c) * r + tid] = (tid <= p0 + c) ? w[c] : 0.0;
      }
    }
    if (bad && tid == 0) atomicMax(status, (int)ASI_ERR_RANK_DEFICIENT);
  } else {
    const int ut = tid - kPivot, ti = ut >> 4, tj = ut & 15;
    double T[NX][NX];
#pragma unroll
    for (int x = 0; x < NX; ++x)
#pragma unroll
      for (int y = 0; y < NX; ++y) {
        const int i = ti + 16 * x, k = tj + 16 * y;
        T[x][y] = (k >= i && k < r) ? Gq[packed_at(i, k, nb)] : 0.0;
      }
    if (ti < 4) {
#pragma unroll
      for (int y = 0; y < NX; ++y) Prow[ti * kQRMaxRank + tj + 16 * y] = T[0][y];
    }
    named_arrive(1, kOT);
#pragma unroll 1
    for (int p0 = 0; p0 < r; p0 += 4) {
      named_sync(2, kOT);
      const int b = p0 + 4;
      if (b >= r) break;
      // rows i >= b: T[i][k] -= sum_c W[i][c] W[k][c] for the columns of Y done so far (k < b) and of G (k >= i);
      // the four rows of the next step first
      const double* Ws = W + ((p0 >> 2) & 1) * (4 * kQRMaxRank);
      const bool mine = ((b ^ ti) & 12) == 0;        // this thread owns one of the rows b .. b + 3
      const int bx = b >> 4;
      double cw[NX][4];                              // read once for all of the thread's rows
#pragma unroll
      for (int y = 0; y < NX; ++y)
#pragma unroll
        for (int c = 0; c < 4; ++c) cw[y][c] = Ws[c * kQRMaxRank + tj + 16 * y];
#pragma unroll
      for (int pass = 0; pass < 2; ++pass) {
        if (pass == 1 || mine) {
#pragma unroll
          for (int x = 0; x < NX; ++x) {
            const int i = ti + 16 * x;
            const bool next = mine && x == bx;
            if (i >= b && (pass == 0) == next) {
              double a[4];
#pragma unroll
              for (int c = 0; c < 4; ++c) a[c] = Ws[c * kQRMaxRank + i];
#pragma unroll
              for (int y = 0; y < NX; ++y) {
                const int k = tj + 16 * y;
                double v = T[x][y];
#pragma unroll
                for (int c = 0; c < 4; ++c) v = fma(-a[c], cw[y][c], v);
                T[x][y] = (k < b || k >= i) ? v : 0.0;
                if (pass == 0) Prow[(i - b) * kQRMaxRank + k] = T[x][y];
              }
            }
          }
        }
        if (pass == 0) named_arrive(1, kOT);
      }
    }
  }
}

// dst[e] = sum over n of src[s * step + e] in order of s, e < len, with EB x SB loads in flight per thread.  Every
// load is issued from a clamped address: a condition next to a load makes the others wait for it.
template <int EB, int SB, typename TS, typename F>
__device__ __forceinline__ void sum_strided(const TS* __restrict__ src, int n, int64_t step, int len, int e0, int estep, int s0,
                                            int sstep, F&& put) {
#pragma unroll 1
  for (int eb = e0; eb < len; eb += EB * estep) {
    double acc[EB];
#pragma unroll
    for (int q = 0; q < EB; ++q) acc[q] = 0.0;
#pragma unroll 1
    for (int s = s0; s < n; s += SB * sstep) {
      TS t[EB][SB];
#pragma unroll
      for (int q = 0; q < EB; ++q)
#pragma unroll
        for (int u = 0; u < SB; ++u) {
          const int e = eb + q * estep, ss = s + u * sstep;
          t[q][u] = __ldcg(src + (int64_t)(ss < n ? ss : s) * step + (e < len ? e : eb));
        }
#pragma unroll
      for (int q = 0; q < EB; ++q)
#pragma unroll
        for (int u = 0; u < SB; ++u) acc[q] += (s + u * sstep < n) ? (double)t[q][u] : 0.0;
    }
#pragma unroll
    for (int q = 0; q < EB; ++q)
      if (eb + q * estep < len) put(eb + q * estep, acc[q]);
  }
}

}  // namespace

__global__ void __launch_bounds__(kOT) k_orth_factor(const __grid_constant__ QRArgs args) {
  const QRMode M = args.m[blockIdx.y];
  const int c = blockIdx.x, c8 = c & ~(kOrthCluster - 1), rank = c - c8;
  if (c8 >= M.nchunk || M.r > kQRMaxRank) return;    // the whole cluster; ranks above 64 take the k_qrb_* kernels
  pdl_wait();
  namespace cg = cooperative_groups;
  cg::cluster_group cluster = cg::this_cluster();
  extern __shared__ __align__(16) double orth_smem[];
  __shared__ int s_last;
  const int tid = threadIdx.x, r = M.r;
  const int nb = (r + 3) >> 2, nblk = nb * (nb + 1) / 2, len = nblk * 16, RP = 4 * nb;
  double* Ps = orth_smem;                            // this chunk's rows of P, [rows][2][nb][2]: pairs (4 b, 4 b + 1), then (4 b + 2, 4 b + 3)
  double* share = Ps + kOrthMaxRows * kQRMaxRank;    // [len]: this CTA's share of G
  double* red = share + kMaxPacked;                  // scratch: partial sums over splits / over row groups
  const int row0 = c * M.rows;
  const int nrows = c < M.nchunk ? min(M.rows, M.a - row0) : 0;
  const int nval = nrows * r;                        // the chunk is one contiguous run of P
  const int64_t base = (int64_t)row0 * r, sstride = (int64_t)M.a * r;
  // ---- sum of the split partials: a short chunk leaves threads over, which take every SG-th split
  auto place = [&](int e, double v) {
    const int k = e / r, j = e - k * r;
    Ps[k * RP + ((j & 2) ? RP / 2 : 0) + (j >> 2) * 2 + (j & 1)] = v;
    M.Pred[base + e] = v;
  };
  if (nrows > 0) {
    if (RP != r)
      for (int e = tid; e < nrows * RP; e += kOT) Ps[e] = 0.0;   // columns past r
    const int SG = nval >= kOT ? 1 : min(kOT / nval, min(M.nsplit, 8));
    if (RP != r) __syncthreads();
    if (SG > 1) {
      const int sg = tid / nval;
      if (sg < SG)
        sum_strided<1, 16>(M.Pp + base, M.nsplit, sstride, nval, tid - sg * nval, nval, sg, SG,
                           [&](int e, double v) { red[sg * nval + e] = v; });
      __syncthreads();
      for (int e = tid; e < nval; e += kOT) {
        double v = red[e];
        for (int q = 1; q < SG; ++q) v += red[q * nval + e];
        place(e, v);
      }
    } else if (nval <= 4 * kOT) {
      sum_strided<4, 8>(M.Pp + base, M.nsplit, sstride, nval, tid, kOT, 0, 1, place);
    } else {
      sum_strided<7, 4>(M.Pp + base, M.nsplit, sstride, nval, tid, kOT, 0, 1, place);
    }
  }
  __syncthreads();
  // ---- share of G in packed 4 x 4 blocks of the upper triangle: thread (block, row group), row groups in order
  {
    const int RG = min(kOT / nblk, 8);
    const int rg = tid / nblk, t = tid - rg * nblk;
    if (rg < RG) {
      int bi = 0, left = t;
      while (left >= nb - bi) { left -= nb - bi; ++bi; }
      const int bj = bi + left;
      double g[4][4];
#pragma unroll
      for (int x = 0; x < 4; ++x)
#pragma unroll
        for (int y = 0; y < 4; ++y) g[x][y] = 0.0;
#pragma unroll 1
      for (int rl = rg; rl < nrows; rl += RG) {
        const double* prow = Ps + rl * RP;
        const double2 a0 = *reinterpret_cast<const double2*>(prow + 2 * bi), a1 = *reinterpret_cast<const double2*>(prow + RP / 2 + 2 * bi);
        const double2 b0 = *reinterpret_cast<const double2*>(prow + 2 * bj), b1 = *reinterpret_cast<const double2*>(prow + RP / 2 + 2 * bj);
        const double a[4] = {a0.x, a0.y, a1.x, a1.y}, b[4] = {b0.x, b0.y, b1.x, b1.y};
#pragma unroll
        for (int x = 0; x < 4; ++x)
#pragma unroll
          for (int y = 0; y < 4; ++y) g[x][y] = fma(a[x], b[y], g[x][y]);
      }
      double* dst = (RG > 1 ? red + rg * len : share) + t;
#pragma unroll
      for (int x = 0; x < 4; ++x)
#pragma unroll
        for (int y = 0; y < 4; ++y) dst[(x * 4 + y) * nblk] = g[x][y];
    }
    if (RG > 1) {
      __syncthreads();
      for (int e = tid; e < len; e += kOT) {
        double v = red[e];
        for (int q = 1; q < RG; ++q) v += red[q * len + e];
        share[e] = v;
      }
    }
  }
  // ---- the cluster's shares meet: CTA `rank` adds the elements [rank * per, ..) of all of them, in chunk order
  cluster.sync();
  const int live = min(kOrthCluster, M.nchunk - c8), nclu = (M.nchunk + kOrthCluster - 1) / kOrthCluster;
  double* Gc = M.Gp + (int64_t)(c8 / kOrthCluster) * len;
  {
    const int per = (len + kOrthCluster - 1) / kOrthCluster, e1 = min(len, (rank + 1) * per);
    for (int e = rank * per + tid; e < e1; e += kOT) {
      double t[kOrthCluster], v = 0.0;
#pragma unroll
      for (int q = 0; q < kOrthCluster; ++q) t[q] = cluster.map_shared_rank(share, q < live ? q : 0)[e];
#pragma unroll
      for (int q = 0; q < kOrthCluster; ++q) v += q < live ? t[q] : 0.0;
      Gc[e] = v;
    }
  }
  __threadfence();
  cluster.sync();                                    // every share has been read and every part of Gc written
  if (rank != 0) return;
  if (tid == 0) {
    __threadfence();
    s_last = (atomicAdd(M.count, 1) == nclu - 1);
    if (s_last) *M.count = 0;
  }
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  double* Gq = Ps;                                   // [len]
  double* Prow = Gq + kMaxPacked;                    // [4][64]
  double* W = Prow + 4 * kQRMaxRank;                 // [2][4][64]
  sum_strided<7, 6>(M.Gp, nclu, len, len, tid, kOT, 0, 1, [&](int e, double v) { Gq[e] = v; });
  for (int e = tid; e < 2 * 4 * kQRMaxRank; e += kOT) W[e] = 0.0;
  for (int e = tid; e < 4 * kQRMaxRank; e += kOT) Prow[e] = 0.0;
  __syncthreads();
  double trace = 0.0;
  for (int b = 0, o = 0; b < nb; o += nb - b, ++b)   // entries past r are zero
    trace += (Gq[o] + Gq[5 * nblk + o]) + (Gq[10 * nblk + o] + Gq[15 * nblk + o]);
  double* Yg = M.Gp + (int64_t)nclu * len;           // R^{-T}, row-major
  if (r <= 16) eliminate<1>(Gq, Prow, W, 1e-12 * trace, r, Yg, args.status);
  else if (r <= 32) eliminate<2>(Gq, Prow, W, 1e-12 * trace, r, Yg, args.status);
  else eliminate<4>(Gq, Prow, W, 1e-12 * trace, r, Yg, args.status);
}

// CTA (c, m): 32 rows of U_m; thread (ti, tj) owns rows ti, ti + 16 and columns tj, tj + 16, ..
__global__ void __launch_bounds__(kAT) k_orth_apply(const __grid_constant__ QRArgs args) {
  const QRMode M = args.m[blockIdx.y];
  const int row0 = blockIdx.x * 32;
  if (row0 >= M.a || M.r > kQRMaxRank) return;
  pdl_wait();
  extern __shared__ __align__(16) double orth_smem[];
  const int tid = threadIdx.x, r = M.r, rr = r * r;
  const int PY = r | 1;                              // odd pitch: the lanes' rows of Y fall in distinct banks
  double* Ys = orth_smem;                            // [r][PY]
  double* Ps = Ys + r * PY;                          // [32][r]
  float* Us = reinterpret_cast<float*>(Ps + 32 * r); // [r][33]: the new rows, for the stacked operand
  const int nrows = min(32, M.a - row0);
  const int nb = (r + 3) >> 2;
  const double* Yg = M.Gp + (int64_t)((M.nchunk + kOrthCluster - 1) / kOrthCluster) * (nb * (nb + 1) * 8);
  // eight loads of P and eight of Y in flight per round
  for (int e0 = tid; e0 < rr; e0 += 8 * kAT) {
    double t[8], q[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int e = e0 + u * kAT;
      t[u] = __ldcg(Yg + (e < rr ? e : 0));
      q[u] = __ldcg(M.Pred + (int64_t)row0 * r + (e < nrows * r ? e : 0));
    }
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int e = e0 + u * kAT;
      if (e < rr) Ys[e / r * PY + e % r] = t[u];
      if (e < 32 * r) Ps[e] = (e < nrows * r) ? q[u] : 0.0;
    }
  }
  for (int e = rr + tid; e < 32 * r; e += kAT) Ps[e] = (e < nrows * r) ? __ldcg(M.Pred + (int64_t)row0 * r + e) : 0.0;
  __syncthreads();
  const int ti = tid >> 4, tj = tid & 15;
#pragma unroll 1
  for (int j = tj; j < r; j += 16) {
    const double* y = Ys + j * PY;
    double s0 = 0.0, s1 = 0.0, t0 = 0.0, t1 = 0.0;
    int i = 0;
#pragma unroll 4
    for (; i + 1 <= j; i += 2) {
      s0 = fma(Ps[ti * r + i], y[i], s0);
      t0 = fma(Ps[ti * r + i + 1], y[i + 1], t0);
      s1 = fma(Ps[(ti + 16) * r + i], y[i], s1);
      t1 = fma(Ps[(ti + 16) * r + i + 1], y[i + 1], t1);
    }
    if (i <= j) {
      s0 = fma(Ps[ti * r + i], y[i], s0);
      s1 = fma(Ps[(ti + 16) * r + i], y[i], s1);
    }
    const float u0 = (float)(s0 + t0), u1 = (float)(s1 + t1);
    if (row0 + ti < M.a) M.Uout[(int64_t)(row0 + ti) * r + j] = u0;
    if (row0 + ti + 16 < M.a) M.Uout[(int64_t)(row0 + ti + 16) * r + j] = u1;
    if (M.bt) {
      Us[j * 33 + ti] = u0;
      Us[j * 33 + ti + 16] = u1;
    }
  }
  if (!M.bt) return;
  // the stacked operand has k contiguous: lanes along k
  __syncthreads();
  for (int e = tid; e < 32 * r; e += kAT) {
    const int k = e & 31, j = e >> 5;
    if (row0 + k < M.a) tc_store_terms(M.bt, M.bt_n, M.bt_ld, j, row0 + k, Us[j * 33 + k]);
  }
}

// One row of one factor per thread: u = p R^{-1} with the Cholesky factor that k_sm_reduce left (ranks <= 8).
__global__ void __launch_bounds__(128) k_row_solve(const __grid_constant__ RowSolveArgs p) {
  pdl_launch_dependents();
  pdl_wait();
  __shared__ double Rs[ASI_MAX_MODES][kRfStride];
  for (int e = threadIdx.x; e < p.nd * kRfStride; e += 128) (&Rs[0][0])[e] = __ldcg(p.Rf + e);
  int row = blockIdx.x * 128 + threadIdx.x, m = 0;
  while (m + 1 < p.nd && row >= p.a[m]) row -= p.a[m++];
  const bool on = row < p.a[m];
  const int r = p.r[m];
  double q[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) q[j] = (on && j < r) ? __ldcg(p.Pred[m] + (int64_t)row * r + j) : 0.0;
  __syncthreads();
  if (!on) return;
  const double* R = Rs[m];
  float* dst = p.U[m] + (int64_t)row * r;
#pragma unroll
  for (int j = 0; j < 8; ++j)
    if (j < r) {
#pragma unroll
      for (int i = 0; i < 8; ++i)
        if (i < j) q[j] = fma(-q[i], R[i * 8 + j], q[j]);
      q[j] *= R[64 + j];
      dst[j] = (float)q[j];
    }
}

cudaError_t launch_row_solve(const RowSolveArgs& p, cudaStream_t st) {
  return launch_pdl(k_row_solve, dim3((unsigned)((p.total + 127) / 128)), dim3(128), 0, st, p);
}

// rows of P per CTA of k_orth_factor: about 64 partial loads per thread, so that many splits (the token mode: 40)
// mean short chunks and few splits (a long feature mode) few shares of G
int orth_rows(int64_t a, int r, int64_t nsplit) {
  int rows = kOrthMaxRows;
  while (rows > 8 && (int64_t)rows * r * nsplit > 16384) rows /= 2;
  while (rows < kOrthMaxRows && (a + rows - 1) / rows > 1024) rows *= 2;
  return rows;
}
size_t orth_gp_elems(int64_t nchunk, int r) {
  const size_t nb = (r + 3) / 4;
  return (size_t)((nchunk + kOrthCluster - 1) / kOrthCluster) * nb * (nb + 1) * 8 + (size_t)r * r;   // clusters' shares, R^{-T}
}

cudaError_t launch_orth(const QRArgs& p, int nd, cudaStream_t st) {
  int chunks = 1, amax = 1, rmax = 1;
  double bytes = 0.0;
  bool any = false, big = false;
  for (int m = 0; m < nd; ++m) {
    bytes += 4.0 * p.m[m].a * p.m[m].r * (p.m[m].nsplit + 1);
    if (p.m[m].r > kQRMaxRank) { big = true; continue; }
    any = true;
    chunks = std::max(chunks, p.m[m].nchunk);
    amax = std::max(amax, p.m[m].a);
    rmax = std::max(rmax, p.m[m].r);
  }
  ProfScope prof(ASI_K_QR, st, bytes);
  if (any) {
    const size_t s1 = (size_t)(kOrthMaxRows * kQRMaxRank + kMaxPacked + kOT * 16) * 8, s2 = ((size_t)rmax * (rmax | 1) + 32 * rmax) * 8 + 33 * 4 * (size_t)rmax;
    cudaError_t e = opt_in_smem(reinterpret_cast<const void*>(k_orth_factor), s1);
    if (e == cudaSuccess) e = opt_in_smem(reinterpret_cast<const void*>(k_orth_apply), s2);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)((chunks + kOrthCluster - 1) / kOrthCluster * kOrthCluster), (unsigned)nd);
    cfg.blockDim = dim3(kOT);
    cfg.dynamicSmemBytes = s1;
    cfg.stream = st;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = kOrthCluster;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 2;
    e = cudaLaunchKernelEx(&cfg, k_orth_factor, p);
    if (e != cudaSuccess) return e;
    e = launch_pdl(k_orth_apply, dim3((unsigned)((amax + 31) / 32), (unsigned)nd), dim3(kAT), s2, st, p);
    if (e != cudaSuccess) return e;
  }
  return big ? launch_qr_big(p, nd, st) : cudaSuccess;
}

}  // namespace asi
