// Orthogonalize(P_m) for ranks up to 64: Cholesky-QR with the Gram matrix, the factorisation and the row
// products in fp64 (in exact arithmetic the Gram-Schmidt basis of the columns of P).  Two launches for all modes:
//
//   k_orth_factor : CTA (c, m) sums the split partials of its rows of P_m in fp64 in split order and forms its
//                   share of G = P^T P; the last CTA of a group of shares adds the group, the last group adds the
//                   groups (both in index order) and factors G = R^T R once per mode, carrying the identity along
//                   so that Y = R^{-T} falls out of the same elimination.
//   k_orth_apply  : U = P R^{-1}, i.e. U[k][j] = sum_{i <= j} P[k][i] Y[j][i]: a plain product without a chain.
//
// What bounds it: the elimination is a serial chain of r pivots.  Four columns share one step (every thread
// factors the 4 x 4 pivot block for itself, so a step has two barriers and no broadcast), and only one CTA per
// mode walks the chain; the row solve that every CTA used to repeat is now the parallel second launch.
// A pivot d_j with d_j <= 1e-12 * trace(G), i.e. a Gram-Schmidt residual below 1e-6 * ||P||_F, raises
// ASI_ERR_RANK_DEFICIENT in the status word.
#include <algorithm>

#include "asi_internal.h"

namespace asi {

namespace {

constexpr int kOT = 256;                 // threads per CTA
constexpr int kOrthMaxRows = 64;         // rows of P per share, at most
constexpr int kMaxPacked = 136 * 16;     // packed upper triangle of a 64 x 64 matrix

// G = R^T R and Y = R^{-T} by one elimination on the r x r array T (ranks up to 16 NX): entries k >= i start as G,
// the rest as zero; row i of Y takes the place of the entries k <= i.  Thread (ti, tj) keeps T[ti + 16 x][tj + 16 y]
// in registers; shared memory carries what one step of four columns hands to the next: the four pivot rows
// (Prow [4][64]) and the finished rows of R and Y (W [64][4]).  Y goes to Yg (row-major, zero above the diagonal).
template <int NX>
__device__ void chol_with_inverse(double (&T)[NX][NX], double* Prow, double* W, double trace, int r,
                                  double* __restrict__ Yg, int* status) {
  const int tid = threadIdx.x, ti = tid >> 4, tj = tid & 15;
  const double floor_d = 1e-12 * trace;
  if (ti < 4) {
#pragma unroll
    for (int y = 0; y < NX; ++y) Prow[ti * kQRMaxRank + tj + 16 * y] = T[0][y];
  }
  __syncthreads();
#pragma unroll 1
  for (int p0 = 0; p0 < r; p0 += 4) {
    // column k of the four pivot rows; the pivot block itself is factored by every thread that needs it
    if (tid < r) {
      double D[4][4], inv[4], w[4];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int k = i; k < 4; ++k)
          D[i][k] = (p0 + k < r) ? Prow[i * kQRMaxRank + p0 + k] : (i == k ? 1.0 : 0.0);
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        w[c] = Prow[c * kQRMaxRank + tid];
        if (tid >= p0 && tid < p0 + 4) w[c] = (tid == p0 + c) ? 1.0 : 0.0;     // the identity's columns p0 .. p0 + 3
      }
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        double d = D[c][c];
        if (p0 + c < r && !(d > floor_d)) {
          if (tid == 0) atomicMax(status, (int)ASI_ERR_RANK_DEFICIENT);
          d = (floor_d > 0.0) ? floor_d : 1.0;
        }
        inv[c] = rsqrt(d);
        w[c] *= inv[c];
#pragma unroll
        for (int k = c + 1; k < 4; ++k) D[c][k] *= inv[c];
#pragma unroll
        for (int i = c + 1; i < 4; ++i) {
          w[i] = fma(-D[c][i], w[c], w[i]);
#pragma unroll
          for (int k = i; k < 4; ++k) D[i][k] = fma(-D[c][i], D[c][k], D[i][k]);
        }
      }
      *reinterpret_cast<double2*>(W + tid * 4) = make_double2(w[0], w[1]);
      *reinterpret_cast<double2*>(W + tid * 4 + 2) = make_double2(w[2], w[3]);
      // rows p0 .. p0 + 3 of Y are final
#pragma unroll
      for (int c = 0; c < 4; ++c)
        if (p0 + c < r) Yg[(int64_t)(p0 + c) * r + tid] = (tid <= p0 + c) ? w[c] : 0.0;
    }
    __syncthreads();
    // rows i >= b: T[i][k] -= sum_c W[i][c] W[k][c] for the columns of Y done so far (k < b) and of G (k >= i)
    const int b = p0 + 4;
    if (b >= r) break;
    double wk[NX][4];
#pragma unroll
    for (int y = 0; y < NX; ++y) {
      const double2 c0 = *reinterpret_cast<const double2*>(W + (tj + 16 * y) * 4);
      const double2 c1 = *reinterpret_cast<const double2*>(W + (tj + 16 * y) * 4 + 2);
      wk[y][0] = c0.x; wk[y][1] = c0.y; wk[y][2] = c1.x; wk[y][3] = c1.y;
    }
#pragma unroll
    for (int x = 0; x < NX; ++x) {
      const int i = ti + 16 * x;
      if (i >= b) {
        const double2 a0 = *reinterpret_cast<const double2*>(W + i * 4);
        const double2 a1 = *reinterpret_cast<const double2*>(W + i * 4 + 2);
#pragma unroll
        for (int y = 0; y < NX; ++y) {
          const int k = tj + 16 * y;
          double v = fma(-a0.x, wk[y][0], T[x][y]);
          v = fma(-a0.y, wk[y][1], v);
          v = fma(-a1.x, wk[y][2], v);
          v = fma(-a1.y, wk[y][3], v);
          T[x][y] = (k < b || k >= i) ? v : 0.0;
        }
        if (i < b + 4) {
#pragma unroll
          for (int y = 0; y < NX; ++y) Prow[(i - b) * kQRMaxRank + tj + 16 * y] = T[x][y];
        }
      }
    }
    __syncthreads();
  }
}

// Sum of n shares (each `len` doubles) at element e, for up to EB elements at once so that EB * 8 loads are in
// flight; the shares are added in index order.
template <int EB>
__device__ __forceinline__ void fold_shares(const double* __restrict__ src, int n, int len, int e0, double (&v)[EB]) {
#pragma unroll
  for (int q = 0; q < EB; ++q) v[q] = 0.0;
  for (int s = 0; s < n; s += 8) {
    double t[EB][8];
#pragma unroll
    for (int q = 0; q < EB; ++q)
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int e = e0 + q * kOT;
        t[q][u] = __ldcg(src + (int64_t)(s + u < n ? s + u : s) * len + (e < len ? e : 0));
      }
#pragma unroll
    for (int q = 0; q < EB; ++q)
#pragma unroll
      for (int u = 0; u < 8; ++u) v[q] += (s + u < n) ? t[q][u] : 0.0;
  }
}

// the r x r matrix from packed 4 x 4 blocks of its upper triangle (shared memory), then the elimination
template <int NX>
__device__ void factor_packed(const double* Gq, double* Prow, double* W, double trace, int r, double* Yg, int* status) {
  const int nb = (r + 3) >> 2, ti = threadIdx.x >> 4, tj = threadIdx.x & 15;
  double T[NX][NX];
#pragma unroll
  for (int x = 0; x < NX; ++x)
#pragma unroll
    for (int y = 0; y < NX; ++y) {
      const int i = ti + 16 * x, k = tj + 16 * y;
      const int bi = i >> 2, bk = k >> 2;
      T[x][y] = (k >= i && k < r) ? Gq[(bi * nb - bi * (bi - 1) / 2 + bk - bi) * 16 + (i & 3) * 4 + (k & 3)] : 0.0;
    }
  chol_with_inverse<NX>(T, Prow, W, trace, r, Yg, status);
}

}  // namespace

__global__ void __launch_bounds__(kOT) k_orth_factor(const __grid_constant__ QRArgs args) {
  const QRMode M = args.m[blockIdx.y];
  const int c = blockIdx.x;
  if (c >= M.nchunk || M.r > kQRMaxRank) return;     // ranks above 64 take the k_qrb_* kernels
  pdl_wait();
  extern __shared__ __align__(16) double orth_smem[];
  __shared__ int s_last;
  double* Ps = orth_smem;                            // this chunk's rows of P, pitch r
  const int tid = threadIdx.x, r = M.r;
  const int row0 = c * M.rows;
  const int nrows = min(M.rows, M.a - row0);
  const int nval = nrows * r;                        // the chunk is one contiguous run of P
  const int64_t base = (int64_t)row0 * r, sstride = (int64_t)M.a * r;
  // ---- sum of the split partials, in split order per lane group; eight loads in flight per element.  A short
  // chunk leaves threads over: they take every SG-th split and the SG sums meet in order.
  int SG = 1;
  while (SG < 8 && nval * SG * 2 <= kOT) SG *= 2;
  const int lanes = kOT / SG;
  {
    const int e0 = tid % lanes, sg = tid / lanes;
    double* part = Ps + nval;                        // [SG][nval] (SG > 1 only: nval <= 128)
    constexpr int EB = 8, SB = 4;                    // elements x splits in flight per thread
    for (int eb = e0; eb < nval; eb += EB * lanes) {
      const float* src = M.Pp + base;
      double acc[EB];
#pragma unroll
      for (int q = 0; q < EB; ++q) acc[q] = 0.0;
      for (int s = sg; s < M.nsplit; s += SB * SG) {
        float t[EB][SB];
#pragma unroll
        for (int q = 0; q < EB; ++q)
#pragma unroll
          for (int u = 0; u < SB; ++u) {
            const int e = eb + q * lanes, ss = s + u * SG;
            // always a load, from a clamped address when off: a condition next to a load makes the others wait
            t[q][u] = __ldcg(src + (int64_t)(ss < M.nsplit ? ss : s) * sstride + (e < nval ? e : 0));
          }
#pragma unroll
        for (int q = 0; q < EB; ++q)
#pragma unroll
          for (int u = 0; u < SB; ++u) acc[q] += (s + u * SG < M.nsplit) ? (double)t[q][u] : 0.0;
      }
#pragma unroll
      for (int q = 0; q < EB; ++q) {
        const int e = eb + q * lanes;
        if (e >= nval) break;
        if (SG > 1) part[sg * nval + e] = acc[q];
        else {
          Ps[e] = acc[q];
          M.Pred[base + e] = acc[q];
        }
      }
    }
    if (SG > 1) {
      __syncthreads();
      for (int e = tid; e < nval; e += kOT) {
        double v = 0.0;
        for (int q = 0; q < SG; ++q) v += part[q * nval + e];
        Ps[e] = v;
        M.Pred[base + e] = v;
      }
    }
  }
  __syncthreads();
  // ---- share of G in packed 4 x 4 blocks of the upper triangle: thread (block, row group); the row groups of a
  // block (rows == rg mod RG) meet in order
  const int nb = (r + 3) >> 2, nblk = nb * (nb + 1) / 2, len = nblk * 16;
  double* Gc = M.Gp + (int64_t)c * len;
  {
    int RG = kOT / nblk;
    if (RG > 8) RG = 8;
    if (RG < 1) RG = 1;
    double* red = Ps + kOrthMaxRows * kQRMaxRank;    // [RG][len]
    const int rg = tid / nblk, t = tid - rg * nblk;
    if (rg < RG) {
      int bi = 0, left = t;
      while (left >= nb - bi) { left -= nb - bi; ++bi; }
      const int i0 = 4 * bi, j0 = 4 * (bi + left);
      double g[4][4];
      int ii[4], jj[4];
#pragma unroll
      for (int x = 0; x < 4; ++x) {
        ii[x] = i0 + x < r ? i0 + x : r - 1;
        jj[x] = j0 + x < r ? j0 + x : r - 1;
#pragma unroll
        for (int y = 0; y < 4; ++y) g[x][y] = 0.0;
      }
#pragma unroll 2
      for (int rl = rg; rl < nrows; rl += RG) {
        const double* prow = Ps + rl * r;
        double a[4], b[4];
#pragma unroll
        for (int x = 0; x < 4; ++x) { a[x] = prow[ii[x]]; b[x] = prow[jj[x]]; }
#pragma unroll
        for (int x = 0; x < 4; ++x)
#pragma unroll
          for (int y = 0; y < 4; ++y) g[x][y] = fma(a[x], b[y], g[x][y]);
      }
      double* dst = (RG > 1 ? red + rg * len : Gc) + t * 16;
#pragma unroll
      for (int x = 0; x < 4; ++x)
#pragma unroll
        for (int y = 0; y < 4; y += 2) *reinterpret_cast<double2*>(dst + x * 4 + y) = make_double2(g[x][y], g[x][y + 1]);
    }
    if (RG > 1) {
      __syncthreads();
      for (int e = tid; e < len; e += kOT) {
        double v = red[e];
        for (int q = 1; q < RG; ++q) v += red[q * len + e];
        Gc[e] = v;
      }
    }
  }
  // ---- shares -> groups -> G, each level by its last CTA, in index order
  const int grp = c / M.gs, ngroups = (M.nchunk + M.gs - 1) / M.gs;
  const int gfirst = grp * M.gs, gsize = min(M.gs, M.nchunk - gfirst);
  double* Gg = M.Gp + (int64_t)M.nchunk * len;       // [ngroups][len]
  double* Yg = Gg + (int64_t)ngroups * len;          // R^{-T}, row-major
  __threadfence();
  __syncthreads();
  if (tid == 0) s_last = (atomicAdd(M.gcount + grp, 1) == gsize - 1);
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  constexpr int EB = 5;
  double v[EB];
  if (ngroups > 1) {
    for (int e0 = tid; e0 < len; e0 += EB * kOT) {
      fold_shares<EB>(M.Gp + (int64_t)gfirst * len, gsize, len, e0, v);
#pragma unroll
      for (int q = 0; q < EB; ++q)
        if (e0 + q * kOT < len) Gg[(int64_t)grp * len + e0 + q * kOT] = v[q];
    }
    __threadfence();
    __syncthreads();
    if (tid == 0) {
      M.gcount[grp] = 0;
      s_last = (atomicAdd(M.count, 1) == ngroups - 1);
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    if (tid == 0) *M.count = 0;
  } else if (tid == 0) {
    M.gcount[grp] = 0;
  }
  const double* src = ngroups > 1 ? Gg : M.Gp;
  const int nsum = ngroups > 1 ? ngroups : gsize;
  double* Gq = orth_smem;                            // [len]
  double* Prow = Gq + kMaxPacked;                    // [4][64]
  double* W = Prow + 4 * kQRMaxRank;                 // [64][4]
  for (int e0 = tid; e0 < len; e0 += EB * kOT) {
    fold_shares<EB>(src, nsum, len, e0, v);
#pragma unroll
    for (int q = 0; q < EB; ++q)
      if (e0 + q * kOT < len) Gq[e0 + q * kOT] = v[q];
  }
  W[tid] = 0.0;                                      // columns past r multiply zeros
  __syncthreads();
  double trace = 0.0;
  for (int b = 0, o = 0; b < nb; o += nb - b, ++b)
#pragma unroll
    for (int x = 0; x < 4; ++x)
      if (4 * b + x < r) trace += Gq[o * 16 + x * 5];
  if (r <= 16) factor_packed<1>(Gq, Prow, W, trace, r, Yg, args.status);
  else if (r <= 32) factor_packed<2>(Gq, Prow, W, trace, r, Yg, args.status);
  else factor_packed<4>(Gq, Prow, W, trace, r, Yg, args.status);
}

// CTA (c, m): 32 rows of U_m; thread (ti, tj) owns rows ti, ti + 16 and columns tj, tj + 16, ..
__global__ void __launch_bounds__(kOT) k_orth_apply(const __grid_constant__ QRArgs args) {
  const QRMode M = args.m[blockIdx.y];
  const int row0 = blockIdx.x * 32;
  if (row0 >= M.a || M.r > kQRMaxRank) return;
  pdl_wait();
  extern __shared__ __align__(16) double orth_smem[];
  const int tid = threadIdx.x, r = M.r, rr = r * r;
  const int PY = r | 1;                              // odd pitch: the lanes' rows of Y fall in distinct banks
  double* Ys = orth_smem;                            // [r][PY]
  double* Ps = Ys + r * PY;                          // [32][r]
  const int nrows = min(32, M.a - row0);
  const int nb = (r + 3) >> 2;
  const double* Yg = M.Gp + (int64_t)(M.nchunk + (M.nchunk + M.gs - 1) / M.gs) * (nb * (nb + 1) * 8);
  // eight loads of P and eight of Y in flight per round
  for (int e0 = tid; e0 < rr; e0 += 8 * kOT) {
    double t[8], q[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int e = e0 + u * kOT;
      t[u] = __ldcg(Yg + (e < rr ? e : 0));
      q[u] = __ldcg(M.Pred + (int64_t)row0 * r + (e < nrows * r ? e : 0));
    }
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int e = e0 + u * kOT;
      if (e < rr) Ys[e / r * PY + e % r] = t[u];
      if (e < 32 * r) Ps[e] = (e < nrows * r) ? q[u] : 0.0;
    }
  }
  for (int e = rr + tid; e < 32 * r; e += kOT) Ps[e] = (e < nrows * r) ? __ldcg(M.Pred + (int64_t)row0 * r + e) : 0.0;
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
    if (row0 + ti < M.a) {
      M.Uout[(int64_t)(row0 + ti) * r + j] = u0;
      if (M.bt) tc_store_terms(M.bt, M.bt_n, M.bt_ld, j, row0 + ti, u0);
    }
    if (row0 + ti + 16 < M.a) {
      M.Uout[(int64_t)(row0 + ti + 16) * r + j] = u1;
      if (M.bt) tc_store_terms(M.bt, M.bt_n, M.bt_ld, j, row0 + ti + 16, u1);
    }
  }
}

// One row of one factor per thread: u = p R^{-1} with the Cholesky factor k_sm_reduce left (ranks <= 8).
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
// shares per group: one group up to 16 shares, else 8 each, at most kOrthGroups groups per mode (their counters sit in the status block)
int orth_group(int64_t nchunk) {
  int gs = nchunk <= 16 ? 16 : 8;
  while ((nchunk + gs - 1) / gs > kOrthGroups) gs *= 2;
  return gs;
}
size_t orth_gp_elems(int64_t nchunk, int r) {
  const int gs = orth_group(nchunk);
  const size_t nb = (r + 3) / 4;
  return (size_t)(nchunk + (nchunk + gs - 1) / gs) * nb * (nb + 1) * 8 + (size_t)r * r;   // packed shares and groups, R^{-T}
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
    const size_t s1 = (size_t)2 * kOrthMaxRows * kQRMaxRank * 8, s2 = ((size_t)rmax * (rmax | 1) + 32 * rmax) * 8;
    cudaError_t e = opt_in_smem(reinterpret_cast<const void*>(k_orth_factor), s1);
    if (e == cudaSuccess) e = opt_in_smem(reinterpret_cast<const void*>(k_orth_apply), s2);
    if (e != cudaSuccess) return e;
    e = launch_pdl(k_orth_factor, dim3((unsigned)chunks, (unsigned)nd), dim3(kOT), s1, st, p);
    if (e != cudaSuccess) return e;
    e = launch_pdl(k_orth_apply, dim3((unsigned)((amax + 31) / 32), (unsigned)nd), dim3(kOT), s2, st, p);
    if (e != cudaSuccess) return e;
  }
  return big ? launch_qr_big(p, nd, st) : cudaSuccess;
}

}  // namespace asi
