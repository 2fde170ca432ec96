// Internal declarations shared by the translation units of the ASI library.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include "asi.h"

struct asi_plan;

namespace asi {

// Mode-m view of a contiguous tensor: element (o, k, i) at o*a*I + k*I + i.
// Fibers of the mode are indexed by the flat column q = o*I + i.
struct ModeView {
  int64_t O, a, I, Q;   // Q = O*I = b_m
  int r;
};

static inline size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

constexpr int kStatusBytes = 1024;    // status word (int 0), completion counters (ints 16..255)
constexpr int kQRMaxRank = 64;       // ranks k_orth_* cover (above: k_qrb_*)

// Y(o, j, i) = sum_k X(o, k, i) * B(k, j): the small-mode contraction that serves the
// projection V = A_m^T U, the core products, Z1, Z3, and the final expansions.
struct ModeProdArgs {
  const void* X;
  const float* B;          // [a][n_out]
  float* Y;
  int64_t O, a, I, Q;
  int n_out;
  int64_t so, sj, si;      // Y(o, j, i) = Y[o*so + j*sj + i*si]
};

// One mode's P = A_m (A_m^T U) in a single pass (k_fiber); Pp: [grid][a][r] partials.
struct FiberArgs {
  const void* X;
  const float* U;
  float* Pp;
  int64_t O, a, I, n_tiles;
  int r, vec4;
  int* clear;          // as in PlaneArgs
};

// Modes 3 and 4 of a conv activation in one pass over whole planes (k_wplane; k_plane2 for S x S maps).
struct PlaneArgs {
  const void* X;
  const float* U3;
  const float* U4;
  float* Pp3;          // [grid][S][r3]
  float* Pp4;          // [grid][S][r4]
  int64_t n_planes;
  int S, H, W, r3, r4;
  int np, pitch, nsc, nsr;   // planes per tile, row pitch, lanes per column pair and row (set by the launcher)
  int first = 0;           // the first kernel of a call
  int given = 0;           // k_mplane: U3 and U4 are Omega_3 [planes W][r3] and Omega_4 [planes H][r4], and P_m = A_m Omega_m
  int* clear = nullptr;    // not null: CTA 0 zeroes the 256 ints of the workspace's status block
  int* status = nullptr;   // status word of the workspace (an expired wait on a bulk copy)
  int stall = 0;           // test hook (k_mplane, k_plane2): the barriers are armed and no copy is issued, so the waits expire
};

// One mode with strided fibers, a <= 128, r <= 4 (k_fiber2): both products in one pass, or with
// project_only the mode product Y[o][j][i] = sum_k X[o][k][i] U[k][j] alone.
struct Fiber2Args {
  const void* X;
  const float* U;      // U[k * ldu + j]
  float* Pp;           // [grid][a][r] partials of P (not project_only)
  float* Y;            // project_only: Y[o * y_so + j * y_sj + i]
  int64_t y_so, y_sj;
  int64_t O, I, n_tiles;
  int ldu, a, r, project_only, nstage;
  int given;           // k_mfiber: U is Omega [O I][r], and P = A Omega
  int team;            // k_mfiber: warps that share the rows of a tile (set by the launcher)
  int* status;         // status word of the workspace (k_mfiber: an expired wait on a copy)
  int stall;           // test hook (k_mfiber), as in PlaneArgs
  int first;           // the first kernel of a call
  int* clear;          // as in PlaneArgs (first kernels only)
};

struct QRMode {
  const float* Pp;     // [nsplit][a][r]
  double* Pred;        // [a][r]
  double* Gp;          // packed shares of G, one per eight chunks, then R^{-T} (orth_gp_elems doubles)
  float* Uout;         // [a][r]
  int* count;          // one counter, zero on entry and on exit
  int a, r, nsplit, nchunk;
  int rows;            // rows of P per chunk
  __nv_bfloat16* bt;   // not null: U_m also as the stacked operand [3 bt_n][bt_ld] of the tensor-core products
  int64_t bt_ld;
  int bt_n;
};
struct QRArgs {
  QRMode m[ASI_MAX_MODES];
  int* status;
};
// U_m = P_m R_m^{-1} for ranks <= 8, one row per thread, from what k_sm_reduce left (P_m and the Cholesky factor)
struct RowSolveArgs {
  const double* Pred[ASI_MAX_MODES];   // [a][r]
  const double* Rf;                    // [modes][kRfStride]
  float* U[ASI_MAX_MODES];
  int a[ASI_MAX_MODES], r[ASI_MAX_MODES];
  int nd, total;                       // total = sum of a
};
// Z4[c', j, kh, kw] = sum_{i,h',w'} Z1[i,c',h',w'] Z3pad[i,j,h's+kh-p,w's+kw-p], then
// dW[c', cl, kh, kw] = sum_j Z4[c', j, kh, kw] U2[(g*cg + cl), j].
struct ConvTailArgs {
  const float* Z1;     // [r1][Cout][Ho][Wo]
  const float* Z3;     // [r1][r2][H][W]
  const float* U2;     // [C][r2]
  float* dW;           // [Cout][C/groups][kh][kw]
  int r1, r2, C, Cout, H, W, Ho, Wo, kh, kw, sh, sw, ph, pw, groups;
};

// Fused small-map conv kernels (asi_smallmap_kernels.cu)
constexpr int kRedRows = 8;          // rows of P per CTA in the partial-reduction kernel
struct SmTile1Args {            // k_sm_tile1
  const void* act;
  const float* U_prev;
  float* Pp[ASI_MAX_MODES];     // per-mode partials [nsplit][a_m][r_m]
  int* status;                  // status word (int 0) and completion counters (ints 16..255) of the workspace
  int64_t u_off[ASI_MAX_MODES];
  int r[ASI_MAX_MODES];
  int B, C, n_tiles_b;
  int aligned;                  // act starts on 16 bytes (bf16: 8); else it is read one value at a time (never batched)
  unsigned long long wait_ns;   // limit of the bounded wait on the bulk-copy barrier
  int stall_copy;               // test hook: the producer arms the barrier but issues no copy (the wait must expire)
};
struct SmPass1Args {            // k_sm_pass1
  const void* act;
  const float* U_prev;
  float* Pp[ASI_MAX_MODES];     // per-mode partials [nsplit][a_m][r_m]
  int* status;                  // status word (int 0) and completion counters (ints 16..255) of the workspace
  int64_t u_off[ASI_MAX_MODES];
  int r[ASI_MAX_MODES];
  int B, C, H, W, n_tiles_b;    // n_tiles_b: role-B CTAs (column tiles of all samples)
  int cs, cc, pitch, off_u2;    // role C: CTAs per sample, channels per CTA, floats per channel, start of U_2 in shared memory
  int cl;                       // cluster size of the launch, a multiple of cs
  int vec4;                     // columns come in whole groups of four (C H W % 4 == 0)
  int aligned;                  // act starts on 16 bytes (bf16: 8); else a group is read value by value (never batched)
  int bulk;                     // role C's tile comes by bulk copies (fp32, vec4, aligned)
  unsigned long long wait_ns;   // limit of the bounded wait on the bulk-copy barrier
  int stall_copy;               // test hook: the producer arms the barrier but issues no copy (the wait must expire)
};
// Fixed-order fp64 reduction of the per-tile partials of every P_m, plus per-chunk shares of
// G_m = P_m^T P_m.
struct SmReduceMode {
  const float* Pp;     // [nsplit][a][r], or [nsplit][a][a] Gram matrices A_m A_m^T when gram != 0
  double* Pred;        // [a][r], or [a][a] (the summed Gram matrix) when gram != 0
  double* Gp;          // [nchunk][r][r]
  double* Pg;          // gram != 0 and factor != 0: [a][r], P_m = G_m U_m^prev
  const float* U_prev; // gram != 0 and factor != 0: U_m^prev [a][r]
  float* U;            // large: U_m [a][r] is written here
  int a, r, nsplit, nchunk, gram;
};
// Rows a mode up to which k_sm_reduce_large, which solves for them too, takes a layer.  A conv layer: a row a thread.  Token layers: what
// k_mfiber takes, whose partials are many
constexpr int kSolveRows = 512, kSolveRowsTokens = 384;
constexpr int kRfStride = 80;   // doubles per mode in Rf: rows of R_m at pitch 8, then 1 / diag(R_m) at [64..72)
struct SmReduceArgs {
  SmReduceMode m[ASI_MAX_MODES];
  int large;           // != 0: k_sm_reduce_large (gram == 0, factor != 0, at most kSolveRows rows a mode)
  int factor;          // != 0: the last CTA of each mode factors G_m = R_m^T R_m into Rf (ranks <= 8)
  double* Rf;          // [modes][kRfStride]
  int* counter;        // one per mode, zero on entry, zero again on exit
  int* status;
};
// Finishes Orthogonalize (U_m = P_m R_m^{-1}, rows it needs) in its prologue, then the core.
struct SmCoreArgs {
  const void* act;
  const double* Pred[ASI_MAX_MODES];   // P_m [a][r] in fp64
  const double* Rf;                    // [4][kRfStride]: the Cholesky factors written by the reduction kernel
  float* U_new;
  float* Tp;                    // [C][r1 r3 r4]: the activation contracted over all modes but the channels
  float* Tg;                    // [ceil(n_tiles / gs)][core_elems] per-group partial cores
  float* core;
  int* status;
  int* counter;                 // zero on entry, zero again on exit
  int* gcount;                  // one counter per group of gs tiles, same convention
  int gs;
  int64_t u_off[ASI_MAX_MODES];
  int r[ASI_MAX_MODES];
  int B, C, H, W, tile_c, n_tiles;   // tile_c: channels per tile
  int vec4;                     // columns may be read four at a time (whole groups, aligned)
  int staged;                   // the tile whole in shared memory (set by the launcher)
};
struct SmWgradArgs {
  const float* core;
  const float* U;
  const void* dY;
  float* dW;
  int* status;
  int64_t u_off[ASI_MAX_MODES];
  int r[ASI_MAX_MODES];
  int B, C, Cout, H, W, Ho, Wo, kh, kw, sh, sw, ph, pw, groups, cpb;
  int vec4;                     // columns of dY may be read four at a time
  int nt;                       // threads per CTA: 256 or 512 (the staged form has 512 and splits its sums as nt would)
  int ncl;                      // output channels expanded per round of term 5 (divides cpb)
  int nbuf;                     // staging blocks of term 5: two, or one
  int bulk_store;               // 1: dW row blocks leave through the bulk-copy engine (16-byte sized and aligned)
};
size_t sm_tile1_smem(int S, int R, int B, int C);
int sm_tile1_role_c_ctas(int S, int B);
cudaError_t launch_sm_tile1(const SmTile1Args& p, int S, int R, bool bf16, cudaStream_t st);
cudaError_t launch_sm_tile1_batched(const SmTile1Args* a, int n, int S, int R, bool bf16, cudaStream_t st);
size_t sm_pass1_smem(const SmPass1Args& p, int kind, int R);
int sm_pass1_pitch(int HW);
void sm_pass1_split(int HW, int C, int B, int* cs, int* cc);
int sm_pass1_off_u2(int R, int cc, int pitch);
int sm_pass1_tiles_b(int64_t chw, bool vec4);
int sm_core_tile_c(int HW, int C);
size_t sm_core_smem(const SmCoreArgs& p, int R, bool bf16);
size_t sm_wgrad_smem(const SmWgradArgs& p, int R, bool staged, bool bf16);
cudaError_t launch_sm_pass1(const SmPass1Args& p, int kind, int R, bool bf16, cudaStream_t st);
// Tensor-core products of bf16 tensors (asi_tc_kernels.cu).  A factor enters as its stacked operand (three bf16 terms).
size_t tc_operand_bytes(int64_t K, int n);
int64_t tc_operand_ld(int64_t K);
int tc_operand_n(int n);
int tc_kind(int64_t O, int64_t a, int64_t I, int n);
struct TcSplitMat {
  const float* U;          // [K][nv]
  __nv_bfloat16* Bt;       // [3 N][ldb]
  int64_t ldb;
  int K, nv, N, first;
};
struct TcSplitArgs {
  TcSplitMat m[3];
  int* clear;              // not null: the first CTA zeroes the workspace's status block
  int n;
};
void tc_add_split(TcSplitArgs* p, const float* U, int64_t K, int n, void* Bt);
cudaError_t launch_tc_split(TcSplitArgs& p, cudaStream_t st);
struct TcCall {
  const void* X;           // bf16 [O][a][I]
  const void* bt;          // stacked operand of U [a][n] (projection) or of V [O I][n] (expansion)
  float* Y;                // projection: [O][I][n]; expansion: [nsplit][a][n]
  void* out_bt;            // projection with Y == null: the result as the stacked operand of an [O I][n] factor
  int64_t out_ld;
  int64_t O, a, I, q_per_split;
  int n, nsplit, expand;
};
cudaError_t launch_tc_group(const TcCall* c, int n, int* status, int stall, cudaStream_t st);
cudaError_t launch_sm_reduce(const SmReduceArgs& p, int nd, int max_chunks, cudaStream_t st);
cudaError_t launch_sm_core(const SmCoreArgs& p, int R, bool bf16, int beside, cudaStream_t st);
cudaError_t launch_sm_wgrad(const SmWgradArgs& p, int R, bool bf16, int beside, cudaStream_t st);
// the same kernels over several layers of one variant in one launch each (n <= sm_max_batch())
int sm_max_batch();
cudaError_t launch_sm_pass1_batched(const SmPass1Args* a, int n, int kind, int R, bool bf16, cudaStream_t st);
cudaError_t launch_sm_reduce_batched(const SmReduceArgs* a, const int* max_chunks, int n, cudaStream_t st);
cudaError_t launch_sm_core_batched(const SmCoreArgs* a, int n, int R, bool bf16, int beside, cudaStream_t st);
cudaError_t launch_sm_wgrad_batched(const SmWgradArgs* a, int n, int R, bool bf16, int beside, cudaStream_t st);

// Benchmark timing aid (asi_profile_begin / asi_profile_end).
struct ProfState {
  int id;
  cudaEvent_t* ev;
  int n_pairs, used;
  double bytes;
};
extern ProfState g_prof;
struct ProfScope {
  cudaStream_t st;
  int slot;
  ProfScope(int id, cudaStream_t s, double alg_bytes) : st(s), slot(-1) {
    if (g_prof.id == id) {
      g_prof.bytes += alg_bytes;
      if (g_prof.used < g_prof.n_pairs) {
        slot = g_prof.used;
        cudaEventRecord(g_prof.ev[2 * slot], st);
      }
      ++g_prof.used;
    }
  }
  ~ProfScope() {
    if (slot >= 0) cudaEventRecord(g_prof.ev[2 * slot + 1], st);
  }
};

#ifdef __CUDACC__
// Programmatic dependent launch.  Every kernel of the path may start (and do whatever does not depend on its predecessor in the
// stream) once every CTA of the predecessor has passed pdl_launch_dependents() or has exited; pdl_wait() then blocks until
// the predecessor has finished and its writes are visible.  The first kernel of a call is one too, whatever the caller had
// on the stream before: all its threads wait first, and only then does it let its dependents start, so that everything
// behind it finds all older work of the stream finished (its launch hides behind the kernel before: 1 to 2 us a call).
__device__ __forceinline__ void pdl_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Bt[(t N + j) ldb + k] = t-th bf16 term of v (hi, mid, lo: v = hi + mid + lo to 24 bits)
__device__ __forceinline__ void tc_store_terms(__nv_bfloat16* Bt, int N, int64_t ldb, int j, int64_t k, float v) {
  const __nv_bfloat16 h = __float2bfloat16_rn(v);
  const float r1 = v - __bfloat162float(h);
  const __nv_bfloat16 m = __float2bfloat16_rn(r1);
  Bt[(int64_t)j * ldb + k] = h;
  Bt[(int64_t)(N + j) * ldb + k] = m;
  Bt[(int64_t)(2 * N + j) * ldb + k] = __float2bfloat16_rn(r1 - __bfloat162float(m));
}

// A mode pass of Algorithm 1 depends on nothing the passes before it on the stream write.  The first kernel of a call waits
// for all that is older and (clear not null) zeroes the workspace's status block; the passes behind it run beside their
// predecessor and call pdl_wait() only before they end, so that the kernel behind the last pass sees all of them finished.
__device__ __forceinline__ void pass_begin(int* clear, bool first) {
  if (first) pdl_wait();
  pdl_launch_dependents();
  if (clear && blockIdx.x == 0)
    for (int e = threadIdx.x; e < 256; e += blockDim.x) clear[e] = 0;
}

template <typename... Params, typename... Args>
static inline cudaError_t launch_pdl(void (*kernel)(Params...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                                     const Args&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<Params>(args)...);
}
#endif

// Opt-in to more than 48 KB of dynamic shared memory.  The attribute belongs to a (device, kernel) pair,
// so the sizes already granted are remembered per device.
cudaError_t opt_in_smem(const void* kernel, size_t need);

// One product of a grouped launch (asi_gemm_kernels.cu): C[m][j] = sum_k A(m, k) B[k][j] per outer index o
struct GemmProb {
  const void* X;
  const float* B;          // [K][ldb], columns 0 .. n - 1
  float* Y;                // C(o, m, j) of split s at s * ysplit + o * so + m * si + j * sj
  int64_t sxo, ld, ysplit, so, sj, si;
  int64_t M, K, O;
  int64_t kin;             // k-major A: k per outer slab of X (K when there is one)
  int64_t kps;             // K in nsplit parts of kps (a multiple of 128 unless nsplit == 1)
  int ldb, n, nsplit;      // row pitch of B, columns
  int km, vec, bvec, yvec; // k-major A; rows of A / of B readable, rows of C writable four values at a time
};
// the same as the kernels take it, counted in 32 bits
struct GemmArg {
  const void* X;
  const float* B;
  float* Y;
  int64_t sxo, ld, ysplit, so, sj, si;
  int ldb, kin;
  int M, K, O, n;
  int nsplit, kps;
  int tiles_m, first;      // 32-row tiles; first CTA of the product in the launch
  int ksp, n_cta;          // CTAs that share a tile (1 or the cluster size), CTAs of the product (set by the launcher)
  int km, vec, bvec, yvec;
  int k0;                  // first k (a tile of a wide product)
};
constexpr int64_t kGemmMaxSpan = 1ll << 29;    // k of a split, where there are several
constexpr int64_t kGemmMaxGrid = 1ll << 30;
constexpr int kMaxGroup = 8;
struct GemmGroup {
  GemmProb p[kMaxGroup];
  int np;
  int* clear;              // not null: the first CTA zeroes the 256 ints of the workspace's status block
};
struct GemmArgs {
  GemmArg p[kMaxGroup];
  int np, nst;
  int* clear;
};
bool gemm_narrow(const GemmProb& p);
#ifdef __CUDACC__
__host__ __device__
#endif
GemmArg gemm_tile_arg(const GemmProb& p, int64_t t, int xbytes);
int gemm_expand_splits(int64_t a, int64_t Q);
// Y(o, j, i) = sum_k X[o][k][i] B[k][j] at Y + o * so + j * sj + i * si
void gemm_add(GemmGroup* g, const GemmProb& p);
GemmProb gemm_project(const void* X, const float* B, float* Y, int64_t O, int64_t a, int64_t I, int n, int64_t so, int64_t sj,
                      int64_t si, bool bf16);
// Pp[s][k][j] = sum over the columns (o, i) of split s of X[o][k][i] V[(o, i)][j]
GemmProb gemm_expand(const void* X, const float* V, float* Pp, int64_t O, int64_t a, int64_t I, int n, int nsplit, int64_t kps,
                     bool bf16);
cudaError_t launch_gemm_group(const GemmGroup& g, bool bf16, cudaStream_t st);

int orth_rows(int64_t a, int r, int64_t nsplit);
size_t orth_gp_elems(int64_t nchunk, int r);
cudaError_t launch_orth(const QRArgs& p, int nd, cudaStream_t st);
cudaError_t launch_qr_big(const QRArgs& p, int nd, cudaStream_t st);
cudaError_t launch_row_solve(const RowSolveArgs& p, cudaStream_t st);
cudaError_t launch_fiber(const FiberArgs& p, int grid, bool x_bf16, cudaStream_t st);
size_t fiber_smem(int a);
bool wfiber_supported(int64_t O, int64_t a, int64_t I, int r);
int64_t wfiber_tiles(int64_t O, int64_t a, int64_t I, bool bf16);
int wfiber_grid(int64_t O, int64_t a, int64_t I, int r);
cudaError_t launch_wfiber(const Fiber2Args& p, int grid, bool bf16, cudaStream_t st);
bool wplane_supported(int64_t n_planes, int64_t H, int64_t W, int r3, int r4);
int wplane_grid(int64_t n_planes, int H, int W, int r, bool bf16);
cudaError_t launch_wplane(const PlaneArgs& p, int grid, bool bf16, cudaStream_t st);
bool mfiber_supported(int64_t O, int64_t a, int64_t I, int r, bool bf16);
int mfiber_grid(int64_t O, int64_t a, int64_t I, int r, bool bf16, bool share_sm);
cudaError_t launch_mfiber(const Fiber2Args& p, int grid, bool bf16, cudaStream_t st);
bool mplane_supported(int64_t n_planes, int64_t H, int64_t W, int r3, int r4, bool bf16);
int mplane_grid(int64_t n_planes, int H, int W, int r, bool bf16, bool share_sm);
cudaError_t launch_mplane(const PlaneArgs& p, int grid, bool bf16, cudaStream_t st);
bool fiber2_supported(int64_t O, int64_t a, int64_t I, int r, bool bf16);
int64_t fiber2_tiles(int64_t O, int64_t I);
int fiber2_grid(int64_t O, int64_t a, int64_t I, int r, bool bf16, bool share_sm);
bool fiber_reg_supported(int64_t O, int64_t a, int64_t I, int r, bool bf16);
int fiber_reg_grid(int64_t O, int64_t a, int64_t I, int r, bool bf16);
cudaError_t launch_fiber_reg(const Fiber2Args& p, int grid, bool bf16, cudaStream_t st);
cudaError_t launch_fiber2(const Fiber2Args& p, int grid, bool bf16, cudaStream_t st);
// core = T x_2 U_2^T x_3 U_3^T x_4 U_4^T for T [r1][C][H][W] in one launch (k_core_tail)
struct CoreTailArgs {
  const float* T;
  const float *U2, *U3, *U4;
  float* part;         // [r1][chunks x splits][r2 r3 r4] partial cores
  float* core;
  int* counter;        // one per i < r1, zero on entry, zero again on exit
  int r1, r2, r3, r4, C, H, W, RH, cper;
};
bool core_tail_supported(int r2, int r3, int r4, int H, int W);
size_t core_tail_part_elems(int r1, int r2, int r3, int r4, int C, int H, int W);
cudaError_t launch_core_tail(const CoreTailArgs& p, cudaStream_t st);
cudaError_t launch_z3(const float* core, const float* U3, const float* U4, float* Z3, int r12, int r3, int r4,
                      int H, int W, cudaStream_t st);
// token path (asi_token_kernels.cu)
struct CoreTokArgs {
  const float* T;      // [B][N][r3]
  const float* U1;     // [B][r1], or null: B = r1 = 1 with coefficient one
  const float* U2;     // [N][r2]
  float* core;         // [r1][r2][r3]
  int B, N, r1, r2, r3;
};
cudaError_t launch_core_tok(const CoreTokArgs& p, cudaStream_t st);
struct LinMidArgs {
  const float* Y1;     // [B][Dout][r2]
  const float* U1;     // [B][r1], or null: B = r1 = 1 with coefficient one
  const float* core;   // [r1 r2][r3]
  float* Z4;           // [Dout][r3]
  int B, Dout, r1, r2, r3;
};
cudaError_t launch_lin_mid(const LinMidArgs& p, cudaStream_t st);
struct LinTailArgs {
  const float* Z4;     // [Dout][r]
  const float* U;      // [Din][r]
  float* dW;           // [Dout][Din]
  int Dout, Din, r, vec;
};
cudaError_t launch_lin_tail(const LinTailArgs& p, cudaStream_t st);
bool plane2_supported(int S, int64_t n_planes, int r3, int r4);
int plane2_grid(int S, int64_t n_planes, int max_ctas);
cudaError_t launch_plane2(const PlaneArgs& p, int grid, bool bf16, cudaStream_t st);
int64_t fiber_tiles(int64_t O, int64_t a, int64_t I);
cudaError_t launch_conv_tail(const ConvTailArgs& p, cudaStream_t st);
cudaError_t launch_conv_tail_split(const ConvTailArgs& p, float* Z4p, int nsp, cudaStream_t st);


}  // namespace asi

namespace asi {
// rank selection aids (asi_spectrum_kernels.cu)
size_t spectrum_ws_bytes(const struct ::asi_plan* pl);
cudaError_t launch_philox_words(uint64_t seed, uint32_t stream, int64_t n_groups, uint32_t* out, cudaStream_t st);
struct FillArgs {
  float* out[ASI_MAX_MODES];
  int64_t n[ASI_MAX_MODES];
  uint32_t stream[ASI_MAX_MODES];
  int* clear;          // not null: the first CTA zeroes the 256 ints of the workspace's status block
};
cudaError_t launch_fill_gaussian(uint64_t seed, const FillArgs& p, int count, cudaStream_t st);
cudaError_t launch_mode_spectrum(const struct ::asi_plan* pl, const void* act, double* eig, double* energy, char* w,
                                 cudaStream_t st);
cudaError_t launch_pick_ranks(const struct ::asi_plan* pl, const double* eig, const double* energy, double eps,
                              int r_max, int* ranks, cudaStream_t st);
size_t perplexity_ws_bytes();
cudaError_t launch_perplexity(const float* x, const float* y, int64_t n, double* out, double* part, cudaStream_t st);
}  // namespace asi

struct asi_plan {
  asi_layer_desc_t d;
  int nd;
  int64_t dims[ASI_MAX_MODES];
  int r[ASI_MAX_MODES];
  int64_t N;
  int64_t u_off[ASI_MAX_MODES], u_elems, core_elems;
  int64_t dy_elems, dw_elems, Ho, Wo;
  asi::ModeView mv[ASI_MAX_MODES];
  bool bf16;

  // compress workspace (byte offsets)
  size_t off_Pp[ASI_MAX_MODES], off_Pred[ASI_MAX_MODES], off_Gp[ASI_MAX_MODES], off_T[2];
  size_t off_Rf, off_Pg[ASI_MAX_MODES];
  size_t v_off[ASI_MAX_MODES];     // V_m of the modes without a one-pass kernel
  int tc_mode[ASI_MAX_MODES];      // 0: SIMT, 1: last-mode tensor-core products, 2: inner-extent (token) products
  size_t tcu_off[ASI_MAX_MODES], tcv_off[ASI_MAX_MODES];   // their stacked operands of U_m and V_m
  int nsplit[ASI_MAX_MODES], nchunk[ASI_MAX_MODES], qr_rows[ASI_MAX_MODES];
  int64_t q_per_split[ASI_MAX_MODES];
  int core_order[ASI_MAX_MODES];
  size_t compress_ws;

  // wgrad workspace (byte offsets)
  size_t off_Z[3], off_Z4p;
  int conv_nsp;                    // > 1: terms 4-5 in two launches with conv_nsp partial Z4 per channel
  bool lin_tc;                     // linear backward: dY x_2 U_2^T on the tensor cores
  size_t off_wtc;                  // bf16 operand scratch of that product
  bool core_tok;                   // token layer whose first core product contracts the last mode: the rest in one launch
  bool core_tail;                  // the core products after the first in one launch
  size_t off_ctp;                  // partial cores of that launch
  size_t wgrad_ws;

  int launches_compress, launches_wgrad;

  // fused small-map path
  bool fast_compress, fast_wgrad;
  bool fast_vec4, wgrad_vec4;      // columns of the activation / of dY come in whole groups of four
  bool small_rank;                 // every rank <= 8: partials are reduced by the parallel fp64 kernel
  bool fiber[ASI_MAX_MODES];       // mode handled by the single-pass fiber kernel
  int fiber_grid[ASI_MAX_MODES];
  bool plane;                      // modes 3 and 4 together by the whole-plane kernel
  int plane_grid;
  bool wfiber[ASI_MAX_MODES];      // ... by warps on their own (strided fibers)
  bool fiber2[ASI_MAX_MODES];      // ... by its register-tiled successor (ranks <= 4, 16-byte aligned rows)
  bool mfiber[ASI_MAX_MODES], mplane;   // ... with the factor on the tensor cores
  bool cfiber[ASI_MAX_MODES];      // ... in a cold start, where one product is all there is: modes of up to eight entries too
  int cgrid[ASI_MAX_MODES];        // ... and its CTAs there
  int long_cut;                    // sixteenths of its CTAs that k_mfiber goes without on modes of more than 128 entries
  bool plane2;                     // 56 x 56 planes, ranks <= 4
  bool rows16;                     // act has to start on 16 bytes
  int fast_kind;                   // 7, 14: modes 3 and 4 as Gram matrices of such square maps; 0: any map of at most 256 positions
  int tile_S;                      // != 0: the first pass is k_sm_tile1 for this map size, else k_sm_pass1
  int fast_R, n_tiles_b, fast_cs, fast_cc, core_tile_c, n_tiles_core, cpb, wgrad_ncl, wgrad_nt, fold_gs;
  int wgrad_nbuf;
};
