// C ABI of the ASI library: plan construction (host only) and the enqueue sequences.
#include <algorithm>
#include <cstdio>
#include <cstring>
#include <mutex>
#include <new>
#include <utility>
#include <vector>

#include "asi_internal.h"

using namespace asi;

namespace {

bool valid_ptr(const void* p) { return p != nullptr; }

size_t elem_bytes(const asi_plan* pl) { return pl->bf16 ? 2 : 4; }

void set_mode_views(asi_plan* pl) {
  for (int m = 0; m < pl->nd; ++m) {
    int64_t O = 1, I = 1;
    for (int j = 0; j < m; ++j) O *= pl->dims[j];
    for (int j = m + 1; j < pl->nd; ++j) I *= pl->dims[j];
    pl->mv[m] = ModeView{O, pl->dims[m], I, O * I, pl->r[m]};
  }
}

// dynamic shared memory a fused kernel may ask for: 227 KB per CTA minus up to ~17 KB of static arrays
constexpr size_t kSmemLimit = 208 * 1024;

void build_fused_pass1(const asi_plan* pl, const void* act, const float* U_prev, char* w, SmPass1Args* a);
void build_fused_core(const asi_plan* pl, const void* act, float* U_new, float* core, char* w, bool gram_modes, SmCoreArgs* c);

// Which fused kernels cover this layer (decided once, at plan creation).
void choose_kernels(asi_plan* pl) {
  pl->fast_compress = pl->fast_wgrad = false;
  pl->fast_kind = pl->fast_R = pl->n_tiles_b = pl->cpb = 0;
  if (pl->d.kind != ASI_CONV2D || (pl->d.flags & ASI_FLAG_GENERIC_ONLY)) return;
  int rmax = 0;
  for (int m = 0; m < 4; ++m) rmax = std::max(rmax, pl->r[m]);
  if (rmax > 8) return;
  const int R = rmax <= 4 ? 4 : 8;
  pl->fast_R = R;
  const int64_t B = pl->dims[0], C = pl->dims[1], H = pl->dims[2], W = pl->dims[3];
  // whole planes of at most 256 positions (a CTA's threads), rows and columns of at most 32 (a warp's lanes)
  if (H * W <= 256 && H <= 32 && W <= 32 && B <= 1024 && C <= 4096) {
    pl->fast_kind = (H == W && (H == 7 || H == 14)) ? (int)H : 0;
    pl->fast_vec4 = (C * H * W) % 4 == 0;
    sm_pass1_split((int)(H * W), (int)C, (int)B, &pl->fast_cs, &pl->fast_cc);
    pl->core_tile_c = sm_core_tile_c((int)(H * W), (int)C);
    pl->n_tiles_core = (int)((C + pl->core_tile_c - 1) / pl->core_tile_c);
    pl->n_tiles_b = sm_pass1_tiles_b(C * H * W, pl->fast_vec4);
    // whole batches and whole samples as tiles of 512 threads where two such CTAs share an SM (7 x 7 maps: batches up
    // to 64; at 128 the two kernels are level and the other one keeps all layers of a network in one launch)
    pl->tile_S = 0;
    if (H == W && (H == 7 || H == 14 || H == 16) && B % 8 == 0 && (H != 7 || (C % 4 == 0 && B <= 64)) &&
        sm_tile1_smem((int)H, R, (int)B, (int)C) <= 113 * 1024) {
      pl->tile_S = (int)H;
      pl->n_tiles_b = (int)(H == 7 ? C / 4 : C);
    }
    pl->fold_gs = 8;                                 // tiles per group of the core's two-level sum
    while ((pl->n_tiles_core + pl->fold_gs - 1) / pl->fold_gs > 192) pl->fold_gs *= 2;
    SmPass1Args a;
    SmCoreArgs c;
    build_fused_pass1(pl, nullptr, nullptr, nullptr, &a);
    build_fused_core(pl, nullptr, nullptr, nullptr, nullptr, true, &c);
    pl->fast_compress = sm_pass1_smem(a, pl->fast_kind, R) <= kSmemLimit && sm_core_smem(c, R, pl->bf16) <= kSmemLimit;
  }
  if (B <= 4096 && H <= 64 && W <= 64) {
    const int Cout = pl->d.cout;
    const int64_t HoWo = pl->Ho * pl->Wo;
    // channels per CTA: the smallest count of one, two, four that makes a row of the tile a multiple of four values
    int cpb = 1;
    for (int c = 1; c <= 4; c *= 2)
      if (Cout % c == 0 && (c * HoWo) % 4 == 0) { cpb = c; break; }
    pl->wgrad_vec4 = (cpb * HoWo) % 4 == 0 && (Cout * HoWo) % 4 == 0;
    SmWgradArgs a;
    std::memset(&a, 0, sizeof(a));
    for (int m = 0; m < 4; ++m) a.r[m] = pl->r[m];
    a.B = (int)B; a.C = (int)C; a.Cout = Cout; a.H = (int)H; a.W = (int)W;
    a.Ho = (int)pl->Ho; a.Wo = (int)pl->Wo; a.kh = pl->d.kh; a.kw = pl->d.kw; a.cpb = cpb;
    a.ph = pl->d.pad_h; a.pw = pl->d.pad_w; a.groups = pl->d.groups;
    a.vec4 = pl->wgrad_vec4 ? 1 : 0;
    a.nt = 256;
    // term 5 expands the channels in two rounds when the staging blocks fit, else one at a time
    // (one at a time, too, where two would keep the CTA from sharing its SM with three others)
    a.nbuf = 2;
    a.ncl = cpb >= 2 ? cpb / 2 : 1;
    if (sm_wgrad_smem(a, R, false, pl->bf16) > 56 * 1024) a.ncl = 1;
    // one staging block where two keep a fourth CTA off the SM (ResNet-18 tail at 64: 512 CTAs, three an SM took 29.8 us,
    // four take 24.9)
    if (sm_wgrad_smem(a, R, false, pl->bf16) > 56 * 1024) {
      a.nbuf = 1;
      if (sm_wgrad_smem(a, R, false, pl->bf16) > 56 * 1024) a.nbuf = 2;
    }
    // 256 threads where three such CTAs share an SM and the stream of dY is short (at 128 x 784 values a CTA 512
    // threads take 28 us against 36; at 128 x 196, 256 take 39 us against 46), else 512.  A CTA that needs an SM for itself pays on
    // small maps only: larger ones recompute Z3 in every CTA, and four launches are faster (28 x 28, B = 128, seven
    // layers: 118 us here against 28 us a layer beside other work)
    const size_t need = sm_wgrad_smem(a, R, false, pl->bf16);
    if (need > 75 * 1024 || B * cpb * HoWo > 32768) a.nt = 512;
    if (a.nt == 512 && sm_wgrad_smem(a, R, false, pl->bf16) > kSmemLimit) a.nt = 256;
    // A CTA with much to do gives way to the launches that split the reduction where there are few of these CTAs: Cout / cpb of at most
    // 128, and fewer where dY is below a million values, so that Z1 is a grouped product.  Much: the multiply-adds of term 4 and
    // 0.7 for each of dY's values, which told the two apart best over 159 layers (maps to 40 x 40); half as many
    // with ranks above four, whose loops are twice as wide.  One layer's weight gradient in us, a CTA a channel against the
    // split launches: 32 x 28 x 28 to 55 channels 5 x 5 52.7, 24.1; 128 x 28 x 28 to 64 28.9, 20.0; 64 x 28 x 28 to 128 23.9, 22.6;
    // 16 x 28 x 28 to 15 12.7, 15.1; 32 x 20 x 20 to 64 bf16 13.2, 19.1; 32 x 28 x 28 to 147 20.0, 23.8; 1 x 1 kernels lose (64 x 24 x 24 11.6, 14.5)
    // Long rows of dW, which the last of these launches writes with one CTA each, stay with the CTAs too (681 channels, 31 x 20 x 20 to 8,
    // 5 x 5 20.5, 32.8; 192 channels, 40 x 27 x 27 to 34, 5 x 5 48.5, 31.3)
    const int64_t ctas = Cout / cpb, dy = B * Cout * HoWo, kk = pl->d.kh * pl->d.kw;
    const int64_t work = cpb * HoWo * (10 * kk * pl->r[0] * pl->r[1] + 7 * B) / 10000;   // thousands
    const bool split = kk >= 9 && C / pl->d.groups * kk <= 6400 && work >= (R == 4 ? 68 : 30) && ctas <= 128 && (dy >= (1 << 20) || ctas <= (work >= 150 ? 64 : R == 4 ? 24 : 36));
    if (H * W <= 256 ? need <= kSmemLimit : need <= 113 * 1024 && !split) {
      pl->fast_wgrad = true;
      pl->cpb = cpb;
      pl->wgrad_ncl = a.ncl;
      pl->wgrad_nbuf = a.nbuf;
      pl->wgrad_nt = a.nt;
    }
  }
}

// The core of a conv layer, batch first: one streamed product that leaves t1 values, then k_core_tail, where the mode with the largest
// a_m / r_m first leaves fewer and takes two grouped products more.  The other side of each line, one layer's compress in us:
//   below a million values the batch product is a grouped one, good where it is short against the batch: ranks 3 or 4 16 x 64 x 28 x 28 41
//   against 33, 16 x 40 x 28 x 28 33 against 29; 33 x 19 x 18 x 18 27 against 32, 36 x 30 x 27 x 27 36 against 39
//   up to 128 channels their product is streamed too, so t1 must be small (ranks 8 4: 32 x 128 x 56 x 56 95 against 89; 32 x 128 x 28 x 28
//   51 against 54), and a large fp32 tensor with a long batch whose rank is above four has the channels first where these suit the
//   faster kernel (ranks 8 4: 128 x 128 x 28 x 28 88.6 against 83.2, 96 x 128 x 28 x 28 72.7 against 69.1; 96 x 64 x 28 x 28 52 and 52; 64 x 128 x 28 x 28 65
//   against 67; rows off 16 bytes 96 x 118 x 17 x 17 62 against 66)
//   beyond, the channels are a grouped product, and a large t1 costs only fp32 layers whose batch hardly shrinks (24 x 768 x 28 x 28
//   ranks 6 6: 151 against 136; 64 x 512 x 28 x 28 ranks 8 4 200 against 204; 32 x 512 x 28 x 28 bf16 118 against 122)
bool batch_first(const asi_plan* pl) {
  const int64_t B = pl->dims[0], C = pl->dims[1], chw = C * pl->dims[2] * pl->dims[3], r1 = pl->r[0], t1 = r1 * chw;
  if (B < 4 * r1) return false;
  if (pl->N < (1 << 20)) return chw <= 800 * B;
  if (!wfiber_supported(1, B, chw, pl->r[0])) return false;
  const bool channels = !pl->bf16 && B > 64 && r1 > 4 && pl->r[1] <= 4 && pl->N >= (6 << 20) &&
                        fiber2_supported(B, C, chw / C, pl->r[1], pl->bf16);
  if (C <= 128) return t1 <= (2 << 20) && !channels;
  return pl->bf16 || C < 512 || B >= 8 * r1 || t1 <= (int64_t)(r1 > 4 ? 7 : 9) << 18;
}

// ranks up to eight: the rows of the factors are solved for in a launch of their own
bool solves_wide(const asi_plan* pl) {
  int64_t most = 0;
  for (int m = 0; m < pl->nd; ++m) most = std::max(most, pl->dims[m]);
  return most > (pl->d.kind == ASI_CONV2D ? kSolveRows : kSolveRowsTokens);
}

// Workspace layouts.  Every region is 256-byte aligned; region 0 holds the status word (byte 0)
// and the completion counter of the core kernel (byte 64).
//   kSeparate  regions side by side, a V as large as the largest mode's among them
//   kShared    the core's intermediate tensors take the place of what the mode passes and Orthogonalize leave to one another
//   kPlain     regions side by side as without k_mfiber, k_mplane and the batch-first core
enum Layout { kSeparate, kShared, kPlain };
void layout_compress(asi_plan* pl, Layout how) {
  size_t off = kStatusBytes;
  int rmax = 0;
  for (int m = 0; m < pl->nd; ++m) rmax = std::max(rmax, pl->r[m]);
  pl->small_rank = !pl->fast_compress && rmax <= 8 && !(pl->d.flags & ASI_FLAG_GENERIC_ONLY);
  for (int m = 0; m < ASI_MAX_MODES; ++m) {
    pl->fiber[m] = false;
    pl->wfiber[m] = false;
    pl->fiber_grid[m] = 0;
  }
  pl->plane = false;
  pl->plane_grid = 0;
  if (!pl->fast_compress && !(pl->d.flags & ASI_FLAG_GENERIC_ONLY) && pl->d.kind == ASI_CONV2D &&
      wplane_supported(pl->dims[0] * pl->dims[1], pl->dims[2], pl->dims[3], pl->r[2], pl->r[3])) {
    pl->plane = true;
    pl->plane_grid = wplane_grid(pl->dims[0] * pl->dims[1], (int)pl->dims[2], (int)pl->dims[3],
                                 std::max(pl->r[2], pl->r[3]), pl->bf16);
  }
  // one-pass kernel for every mode with a rank <= 8 and a short fiber, whatever the other modes' ranks
  if (!pl->fast_compress && !(pl->d.flags & ASI_FLAG_GENERIC_ONLY))
    for (int m = 0; m < pl->nd; ++m) {
      if (pl->plane && m >= 2) continue;
      const ModeView& v = pl->mv[m];
      pl->wfiber[m] = wfiber_supported(v.O, v.a, v.I, pl->r[m]);
      if (pl->wfiber[m]) {
        pl->fiber[m] = true;
        pl->fiber_grid[m] = wfiber_grid(v.O, v.a, v.I, pl->r[m]);
      } else if (pl->r[m] <= 8 && v.a <= 128 && fiber_smem((int)v.a) <= kSmemLimit) {
        pl->fiber[m] = true;
        pl->fiber_grid[m] = (int)std::min<int64_t>(fiber_tiles(v.O, v.a, v.I), 296);
      }
    }
  // register-tiled successors where the shape fits them (one partial per CTA, fewer and larger CTAs)
  pl->plane2 = false;
  for (int m = 0; m < ASI_MAX_MODES; ++m) pl->fiber2[m] = false;
  if (pl->plane && pl->dims[2] == pl->dims[3] && plane2_supported((int)pl->dims[2], pl->dims[0] * pl->dims[1], pl->r[2], pl->r[3])) {
    pl->plane2 = true;
    pl->plane_grid = plane2_grid((int)pl->dims[2], pl->dims[0] * pl->dims[1],
                                 (pl->d.flags & ASI_FLAG_SHARE_SM) ? 148 : 296);
  }
  for (int m = 0; m < pl->nd; ++m)
    if (pl->fiber[m] && fiber2_supported(pl->mv[m].O, pl->mv[m].a, pl->mv[m].I, pl->r[m], pl->bf16)) {
      pl->fiber2[m] = true;
      pl->wfiber[m] = false;
      pl->fiber_grid[m] = fiber2_grid(pl->mv[m].O, pl->mv[m].a, pl->mv[m].I, pl->r[m], pl->bf16,
                                      (pl->d.flags & ASI_FLAG_SHARE_SM) != 0);
    }
  // these copy rows on 16 bytes, and so did the kernel that 28 x 28 planes had: such layers want the address on 16 bytes
  const int64_t planes = pl->dims[0] * (pl->nd > 1 ? pl->dims[1] : 1);
  const bool plane28 = pl->plane && pl->dims[2] == 28 && pl->dims[3] == 28 && pl->r[2] <= 4 && pl->r[3] <= 4 && planes % 8 == 0;
  if (plane28 && how == kPlain) pl->plane_grid = plane2_grid(28, planes, (pl->d.flags & ASI_FLAG_SHARE_SM) ? 148 : 296);
  pl->rows16 = pl->plane2 || plane28;
  for (int m = 0; m < pl->nd; ++m) pl->rows16 = pl->rows16 || pl->fiber2[m];
  // the factor on the tensor cores: the first two modes of conv layers and the batch of token layers, where they fill the tiles (a
  // mode of 8 leaves half of each empty: 8 x 512 x 5632 bf16, ranks 8, 36 us against 29 of k_fiber_reg; 32 x 197 x 3072 16 against 28;
  // compress of 8 x 700 x 56 x 56 161 us against 140, of 10 x 700 x 56 x 56 182 against 178, of 10 x 64 x 28 x 28 29 against 30).
  // Not the rows of a matrix: few columns average the operands' rounding less (82 x 958: 9.3e-8 against 5.1e-8)
  pl->mplane = false;
  for (int m = 0; m < ASI_MAX_MODES; ++m) pl->mfiber[m] = pl->cfiber[m] = false;
  const bool share = (pl->d.flags & ASI_FLAG_SHARE_SM) != 0;
  if (pl->plane && how != kPlain && mplane_supported(pl->dims[0] * pl->dims[1], pl->dims[2], pl->dims[3], pl->r[2], pl->r[3], pl->bf16)) {
    pl->mplane = true;
    pl->plane_grid = mplane_grid(pl->dims[0] * pl->dims[1], (int)pl->dims[2], (int)pl->dims[3], std::max(pl->r[2], pl->r[3]),
                                 pl->bf16, share);
  }
  if (!pl->fast_compress && !(pl->d.flags & ASI_FLAG_GENERIC_ONLY) && how != kPlain)
    for (int m = 0; m < (pl->d.kind == ASI_CONV2D ? 2 : 1); ++m) {
      const ModeView& v = pl->mv[m];
      if (pl->d.kind == ASI_LINEAR && (pl->nd != 3 || !pl->fiber[m] || v.a <= 8)) continue;
      if (!mfiber_supported(v.O, v.a, v.I, v.r, pl->bf16) || (pl->bf16 && !pl->wfiber[m] && !pl->fiber2[m])) continue;
      pl->cfiber[m] = v.a > 8 || pl->fiber[m];
      pl->cgrid[m] = mfiber_grid(v.O, v.a, v.I, v.r, pl->bf16, share);
      if (v.a <= 8) continue;
      pl->mfiber[m] = pl->fiber[m] = true;
      pl->fiber_grid[m] = mfiber_grid(v.O, v.a, v.I, v.r, pl->bf16, share);
      if (v.a > 128) pl->fiber_grid[m] -= pl->fiber_grid[m] * pl->long_cut / 16;
    }
  const size_t passes = off;                          // what the mode passes and Orthogonalize leave to one another: from here
  // V_m of the modes without a one-pass kernel, one region each (their products share launches); at least the
  // largest V of the layer
  if (!pl->fast_compress) {
    size_t used = 0, vmax = 0;
    for (int m = 0; m < pl->nd; ++m) {
      const size_t bytes = align_up((size_t)pl->mv[m].Q * pl->r[m] * 4, 256);
      pl->v_off[m] = off + used;
      vmax = std::max(vmax, bytes);
      if (!pl->fiber[m] && !(pl->plane && m >= 2)) used += bytes;
    }
    off += how == kShared ? used : std::max(used, vmax);
  }
  for (int m = 0; m < pl->nd; ++m) {
    const ModeView& v = pl->mv[m];
    int64_t ns = gemm_expand_splits(v.a, v.Q);
    int64_t qps = (v.Q + ns - 1) / ns;
    qps = (qps + 127) / 128 * 128;
    ns = (v.Q + qps - 1) / qps;
    if (pl->fast_compress) {                                             // one partial per column tile, per sample,
      ns = m == 0 ? pl->n_tiles_b : (m == 1 ? pl->dims[0] : pl->dims[0] * pl->fast_cs);   // per role-C CTA (k_sm_tile1: per
      if (pl->tile_S) ns = m == 1 ? sm_tile1_role_c_ctas(pl->tile_S, (int)pl->dims[0]) : pl->n_tiles_b;   // tile); the cold-start
      qps = ((v.Q + ns - 1) / ns + 127) / 128 * 128;                     // expansion splits the columns over at most as many
    }
    if (pl->fiber[m] || (pl->plane && m >= 2)) {                         // one partial per CTA of k_fiber /
      ns = pl->fiber[m] ? pl->fiber_grid[m] : pl->plane_grid;            // a plane kernel; the cold-start expansion
      qps = ((v.Q + ns - 1) / ns + 63) / 64 * 64;                        // uses the same count (empty splits
    }                                                                    // write 0)
    pl->nsplit[m] = (int)ns;
    pl->q_per_split[m] = qps;
    pl->qr_rows[m] = (pl->fast_compress || pl->small_rank) ? kRedRows : orth_rows(v.a, v.r, ns);
    pl->nchunk[m] = (int)((v.a + pl->qr_rows[m] - 1) / pl->qr_rows[m]);
    pl->off_Pp[m] = off;
    if (pl->mfiber[m]) pl->cgrid[m] = (int)ns;
    size_t pp_elems = (size_t)(pl->cfiber[m] ? std::max<int64_t>(ns, pl->cgrid[m]) : ns) * v.a * v.r;
    if (pl->fast_compress && pl->fast_kind && m >= 2) pp_elems = std::max(pp_elems, (size_t)ns * v.a * v.a);
    off = align_up(off + pp_elems * 4, 256);
    pl->off_Pred[m] = off;
    off = align_up(off + (size_t)v.a * std::max<int64_t>(v.r, (pl->fast_compress && m >= 2) ? v.a : 0) * 8, 256);
    pl->off_Gp[m] = off;
    const size_t shares = (pl->fast_compress || pl->small_rank) ? (size_t)pl->nchunk[m] * v.r * v.r : 0;   // k_sm_reduce's
    off = align_up(off + std::max(shares, orth_gp_elems(pl->nchunk[m], v.r)) * 8, 256);
  }
  // core chain: contract the mode with the largest a_m / r_m first, then the rest in order
  int order[ASI_MAX_MODES];
  for (int m = 0; m < pl->nd; ++m) order[m] = m;
  int best = 0;
  for (int m = 1; m < pl->nd; ++m)
    if ((double)pl->dims[m] / pl->r[m] > (double)pl->dims[best] / pl->r[best]) best = m;
  // linear layers: the feature mode first where that shrinks the tensor by four at least (k_core_tok does the rest)
  if (pl->d.kind == ASI_LINEAR && (pl->nd == 2 || pl->dims[pl->nd - 1] >= 4 * pl->r[pl->nd - 1])) best = pl->nd - 1;
  // conv layers whose core k_core_tail finishes: the batch first where that pays
  const bool tail = pl->d.kind == ASI_CONV2D && !pl->fast_compress && !(pl->d.flags & ASI_FLAG_GENERIC_ONLY) &&
                    core_tail_supported(pl->r[1], pl->r[2], pl->r[3], (int)pl->dims[2], (int)pl->dims[3]);
  if (tail && how != kPlain && batch_first(pl)) best = 0;
  std::swap(order[0], order[best]);
  std::sort(order + 1, order + pl->nd);
  std::memcpy(pl->core_order, order, sizeof(order));
  int64_t cd[ASI_MAX_MODES];
  for (int m = 0; m < pl->nd; ++m) cd[m] = pl->dims[m];
  int64_t tmax[2] = {0, 0};
  for (int s = 0; s + 1 < pl->nd; ++s) {
    cd[order[s]] = pl->r[order[s]];
    int64_t n = 1;
    for (int m = 0; m < pl->nd; ++m) n *= cd[m];
    tmax[s & 1] = std::max(tmax[s & 1], n);
  }
  if (pl->fast_compress) {
    tmax[0] = pl->dims[1] * (pl->core_elems / pl->r[1]);        // per-channel shares
    tmax[1] = (int64_t)((pl->n_tiles_core + pl->fold_gs - 1) / pl->fold_gs) * pl->core_elems;
  }
  size_t t_off = how == kShared && !pl->fast_compress ? passes : off;   // the first of them is written behind all of Orthogonalize
  for (int t = 0; t < 2; ++t) {
    pl->off_T[t] = t_off;
    t_off = align_up(t_off + (size_t)tmax[t] * 4, 256);
  }
  off = std::max(off, t_off);
  // Tensor-core products of bf16 tensors: a factor of 16..64 columns (a multiple of 4) over the last mode (a_m a
  // multiple of 64, at least 128 fibers) or over a mode whose inner extent is a multiple of 64
  for (int m = 0; m < pl->nd; ++m) {
    const ModeView& v = pl->mv[m];
    pl->tc_mode[m] = 0;
    if (pl->bf16 && pl->d.kind == ASI_LINEAR && !pl->fiber[m] && !(pl->d.flags & ASI_FLAG_GENERIC_ONLY))
      pl->tc_mode[m] = tc_kind(v.O, v.a, v.I, v.r);
    if (!pl->tc_mode[m]) continue;
    pl->tcu_off[m] = off;
    off = align_up(off + tc_operand_bytes(v.a, v.r), 256);
    pl->tcv_off[m] = off;
    off = align_up(off + tc_operand_bytes(v.Q, v.r), 256);
  }
  pl->off_Rf = off;                                   // Cholesky factors of the fused path
  off = align_up(off + (size_t)ASI_MAX_MODES * kRfStride * 8, 256);
  for (int m = 0; m < ASI_MAX_MODES; ++m) pl->off_Pg[m] = 0;
  if (pl->fast_compress)
    for (int m = 2; m < 4; ++m) {                     // P_m of a Gram mode
      pl->off_Pg[m] = off;
      off = align_up(off + (size_t)pl->dims[m] * pl->r[m] * 8, 256);
    }
  pl->core_tail = pl->core_tok = false;
  pl->off_ctp = off;
  if (tail && order[0] == 0) {                       // the others follow in order
    pl->core_tail = true;
    off = align_up(off + 4 * core_tail_part_elems(pl->r[0], pl->r[1], pl->r[2], pl->r[3], (int)pl->dims[1],
                                                  (int)pl->dims[2], (int)pl->dims[3]), 256);
  }
  pl->compress_ws = off;
  pl->launches_compress = 3;
  if (!pl->fast_compress) {
    pl->core_tok = pl->d.kind == ASI_LINEAR && (pl->nd == 2 || order[0] == 2);
    // the kernels of Orthogonalize (one for ranks up to eight where solves_wide does not say two), the core chain, one launch per one-pass mode (one for both
    // spatial modes), one projection and one expansion launch for all SIMT modes together
    pl->launches_compress = (pl->small_rank && !solves_wide(pl) ? 1 : 2) + ((pl->core_tail || pl->core_tok) ? 2 : pl->nd);
    bool simt = false, tc = false;
    for (int m = 0; m < pl->nd; ++m) {
      if (pl->plane && m >= 2) pl->launches_compress += (m == 2);
      else if (pl->fiber[m]) pl->launches_compress += 1;
      else if (pl->tc_mode[m]) tc = true;
      else simt = true;
    }
    if (tc) pl->launches_compress += 3;              // operand split, projections, expansions
    if (simt) pl->launches_compress += 2;
  }
}

// asi_compress_static_ws takes the layers whose workspace fits its 4 MiB with the mode passes of the fp32 pipe.  k_mfiber has a partial
// of P for each of up to 296 CTAs also on modes of 129 to 384 entries, where the grouped products keep a few, and a batch-first
// core larger intermediate tensors (three in a hundred of these layers grew past 4 MiB).  Such a layer shares its regions, and where that is
// not enough (one in five thousand) up to half of the CTAs of its long modes go: 148 for 296 cost 8 x 364 x 28 x 56 4 of
// 76 us, 9 x 230 x 36 x 36 2 of 63
void fit_compress(asi_plan* pl) {
  const auto fits = [&](Layout how) {
    layout_compress(pl, how);
    return pl->compress_ws <= (size_t)ASI_STATIC_WS_MAX_BYTES;
  };
  pl->long_cut = 0;
  if (fits(kSeparate)) return;
  if (fits(kPlain))
    for (; pl->long_cut <= 8; ++pl->long_cut)
      if (fits(kShared)) return;
  pl->long_cut = 0;
  layout_compress(pl, kSeparate);
}

void layout_wgrad(asi_plan* pl) {
  size_t off = kStatusBytes;
  int64_t z[3] = {0, 0, 0};
  if (pl->d.kind == ASI_CONV2D) {
    z[0] = (int64_t)pl->r[0] * pl->d.cout * pl->Ho * pl->Wo;          // Z1
    z[1] = (int64_t)pl->r[0] * pl->r[1] * pl->dims[2] * pl->dims[3];  // Z3
    pl->launches_wgrad = pl->fast_wgrad ? 1 : 3;
  } else {
    // dY x_2 U_2^T [B][Dout][r2] (two modes: dY x_1 U_1^T [Dout][r1]), then Z4 [Dout][r_last]
    z[0] = pl->nd == 3 ? pl->dims[0] * pl->d.cout * pl->r[1] : (int64_t)pl->d.cout * pl->r[0];
    z[1] = (int64_t)pl->r[pl->nd - 1] * pl->d.cout;
    pl->lin_tc = pl->nd == 3 && pl->bf16 && !(pl->d.flags & ASI_FLAG_GENERIC_ONLY) &&
                 tc_kind(pl->dims[0], pl->dims[1], pl->d.cout, pl->r[1]) == 2;
    pl->launches_wgrad = pl->lin_tc ? 4 : 3;
  }
  for (int t = 0; t < 3; ++t) {
    pl->off_Z[t] = off;
    off = align_up(off + (size_t)z[t] * 4, 256);
  }
  pl->off_wtc = off;
  if (pl->d.kind == ASI_LINEAR && pl->lin_tc) off = align_up(off + tc_operand_bytes(pl->dims[1], pl->r[1]), 256);
  pl->conv_nsp = 1;
  pl->off_Z4p = off;
  if (pl->d.kind == ASI_CONV2D && !pl->fast_wgrad && !(pl->d.flags & ASI_FLAG_GENERIC_ONLY) &&
      (int64_t)pl->r[0] * pl->Ho * pl->Wo >= 1024 && pl->d.cout < 296) {
    pl->conv_nsp = (int)std::min<int64_t>(16, std::max<int64_t>(2, 592 / pl->d.cout));
    pl->conv_nsp = (int)std::min<int64_t>(pl->conv_nsp, (int64_t)pl->r[0] * pl->Ho);
    off = align_up(off + (size_t)pl->conv_nsp * pl->d.cout * pl->r[1] * pl->d.kh * pl->d.kw * 4, 256);
    pl->launches_wgrad = 4;
  }
  pl->wgrad_ws = off;
}

// act and dY are read four values at a time where they start on 16 bytes (bf16: 8), else one at a time
bool four_aligned(const asi_plan* pl, const void* p) {
  return (reinterpret_cast<uintptr_t>(p) & (pl->bf16 ? 7u : 15u)) == 0;
}
bool element_aligned(const asi_plan* pl, const void* p) {
  return (reinterpret_cast<uintptr_t>(p) & (elem_bytes(pl) - 1)) == 0;
}

// asi_compress takes this address: any element's, but for the 16-byte rows of the large-map kernels' bulk copies
bool compress_takes(const asi_plan* pl, const void* act) {
  return element_aligned(pl, act) && (!pl->rows16 || (reinterpret_cast<uintptr_t>(act) & 15u) == 0);
}

int stalls(const asi_plan* pl) { return (pl->d.flags & ASI_FLAG_TEST_EXPIRE_WAIT) ? 1 : 0; }

asi_status_t check_ws(const void* ws, size_t have, size_t need) {
  if (!valid_ptr(ws)) return ASI_ERR_INVALID_ARG;
  if (have < need || (reinterpret_cast<uintptr_t>(ws) & 255u)) return ASI_ERR_WORKSPACE;
  return ASI_OK;
}

thread_local char g_cuda_err[256] = "";

#define ASI_CUDA(call)                                                        \
  do {                                                                        \
    cudaError_t e__ = (call);                                                 \
    if (e__ != cudaSuccess) {                                                 \
      snprintf(g_cuda_err, sizeof(g_cuda_err), "%s: %s", #call, cudaGetErrorString(e__)); \
      return ASI_ERR_CUDA;                                                    \
    }                                                                         \
  } while (0)

// Argument blocks of the fused small-map kernels for one layer (shared by the single-layer and the
// batched entry points).
void build_fused_pass1(const asi_plan* pl, const void* act, const float* U_prev, char* w, SmPass1Args* a) {
  a->act = act;
  a->U_prev = U_prev;
  for (int m = 0; m < 4; ++m) {
    a->Pp[m] = reinterpret_cast<float*>(w + pl->off_Pp[m]);
    a->u_off[m] = pl->u_off[m];
    a->r[m] = pl->r[m];
  }
  a->status = reinterpret_cast<int*>(w);     // cleared by the kernel itself
  a->B = (int)pl->dims[0];
  a->C = (int)pl->dims[1];
  a->H = (int)pl->dims[2];
  a->W = (int)pl->dims[3];
  a->n_tiles_b = pl->n_tiles_b;
  a->cs = pl->fast_cs;
  a->cl = pl->fast_cs;
  a->cc = pl->fast_cc;
  a->pitch = sm_pass1_pitch(a->H * a->W);
  a->off_u2 = sm_pass1_off_u2(pl->fast_R, a->cc, a->pitch);
  a->vec4 = pl->fast_vec4 ? 1 : 0;
  a->aligned = four_aligned(pl, act) ? 1 : 0;
  a->bulk = (!pl->bf16 && pl->fast_vec4 && a->aligned) ? 1 : 0;
  a->stall_copy = stalls(pl);
  a->wait_ns = a->stall_copy ? 1000000ull : 1000000000ull;      // 1 ms under the test hook, else 1 s
}

void build_tile1(const asi_plan* pl, const void* act, const float* U_prev, char* w, SmTile1Args* a) {
  a->act = act;
  a->U_prev = U_prev;
  for (int m = 0; m < 4; ++m) {
    a->Pp[m] = reinterpret_cast<float*>(w + pl->off_Pp[m]);
    a->u_off[m] = pl->u_off[m];
    a->r[m] = pl->r[m];
  }
  a->status = reinterpret_cast<int*>(w);
  a->B = (int)pl->dims[0];
  a->C = (int)pl->dims[1];
  a->n_tiles_b = pl->n_tiles_b;
  a->aligned = four_aligned(pl, act) ? 1 : 0;
  a->stall_copy = stalls(pl);
  a->wait_ns = a->stall_copy ? 1000000ull : 1000000000ull;
}

int build_fused_reduce(const asi_plan* pl, char* w, const float* gram_U_prev, SmReduceArgs* ra) {
  int max_chunks = 1;
  std::memset(ra, 0, sizeof(*ra));
  for (int m = 0; m < pl->nd; ++m) {
    ra->m[m].Pp = reinterpret_cast<const float*>(w + pl->off_Pp[m]);
    ra->m[m].Pred = reinterpret_cast<double*>(w + pl->off_Pred[m]);
    ra->m[m].Gp = reinterpret_cast<double*>(w + pl->off_Gp[m]);
    ra->m[m].a = (int)pl->dims[m];
    ra->m[m].r = pl->r[m];
    ra->m[m].nsplit = pl->nsplit[m];
    ra->m[m].nchunk = pl->nchunk[m];
    if (gram_U_prev && pl->fast_kind && m >= 2) {
      ra->m[m].gram = 1;
      ra->m[m].nchunk = (int)((pl->dims[m] * pl->dims[m] + 24) / 25);   // ~25 Gram elements per CTA
      ra->m[m].Pg = reinterpret_cast<double*>(w + pl->off_Pg[m]);
      ra->m[m].U_prev = gram_U_prev + pl->u_off[m];
    }
    max_chunks = std::max(max_chunks, ra->m[m].nchunk);
  }
  ra->factor = 1;
  ra->Rf = reinterpret_cast<double*>(w + pl->off_Rf);
  ra->counter = reinterpret_cast<int*>(w) + 20;
  ra->status = reinterpret_cast<int*>(w);
  return max_chunks;
}

void build_fused_core(const asi_plan* pl, const void* act, float* U_new, float* core, char* w, bool gram_modes,
                      SmCoreArgs* c) {
  c->act = act;
  c->U_new = U_new;
  c->Rf = reinterpret_cast<const double*>(w + pl->off_Rf);
  c->Tp = reinterpret_cast<float*>(w + pl->off_T[0]);
  c->core = core;
  c->status = reinterpret_cast<int*>(w);
  c->counter = reinterpret_cast<int*>(w) + 16;
  c->gcount = reinterpret_cast<int*>(w) + 64;
  c->gs = pl->fold_gs;
  c->Tg = reinterpret_cast<float*>(w + pl->off_T[1]);
  for (int m = 0; m < 4; ++m) {
    const bool gram = gram_modes && pl->fast_kind && m >= 2;
    c->Pred[m] = reinterpret_cast<const double*>(w + (gram ? pl->off_Pg[m] : pl->off_Pred[m]));
    c->u_off[m] = pl->u_off[m];
    c->r[m] = pl->r[m];
  }
  c->B = (int)pl->dims[0];
  c->C = (int)pl->dims[1];
  c->H = (int)pl->dims[2];
  c->W = (int)pl->dims[3];
  c->tile_c = pl->core_tile_c;
  c->n_tiles = pl->n_tiles_core;
  c->vec4 = (pl->fast_vec4 && (pl->core_tile_c * c->H * c->W) % 4 == 0 && four_aligned(pl, act)) ? 1 : 0;
  c->staged = 0;
}

void build_fused_wgrad(const asi_plan* pl, const float* core, const float* U, const void* dY, float* dW, char* w,
                       SmWgradArgs* g) {
  g->core = core; g->U = U; g->dY = dY; g->dW = dW;
  for (int m = 0; m < 4; ++m) {
    g->u_off[m] = pl->u_off[m];
    g->r[m] = pl->r[m];
  }
  g->B = (int)pl->dims[0]; g->C = (int)pl->dims[1]; g->Cout = pl->d.cout;
  g->H = (int)pl->dims[2]; g->W = (int)pl->dims[3]; g->Ho = (int)pl->Ho; g->Wo = (int)pl->Wo;
  g->kh = pl->d.kh; g->kw = pl->d.kw; g->sh = pl->d.stride_h; g->sw = pl->d.stride_w;
  g->ph = pl->d.pad_h; g->pw = pl->d.pad_w; g->groups = pl->d.groups; g->cpb = pl->cpb;
  g->ncl = pl->wgrad_ncl;
  g->vec4 = pl->wgrad_vec4 && four_aligned(pl, dY) ? 1 : 0;
  g->nt = pl->wgrad_nt;
  g->nbuf = pl->wgrad_nbuf;
  g->status = reinterpret_cast<int*>(w);
  g->bulk_store = (((pl->dims[1] / pl->d.groups) * pl->d.kh * pl->d.kw) % 4 == 0 &&
                   (reinterpret_cast<uintptr_t>(dW) & 15u) == 0) ? 1 : 0;
}

// U_m^{new} = Orthogonalize(P_m) for all modes given the split partials.
// gram_U_prev != nullptr: the partials of modes 3 and 4 of a 7x7 or 14x14 map are Gram matrices A_m A_m^T
// (written by the fused first pass) and P_m = G_m U_m^prev is formed during the reduction.
asi_status_t orthogonalize_all(const asi_plan* pl, float* U_new, char* w, const float* gram_U_prev,
                               bool first_core_tc, cudaStream_t st) {
  int max_chunks = 1;
  if (pl->fast_compress) {
    SmReduceArgs ra;
    max_chunks = build_fused_reduce(pl, w, gram_U_prev, &ra);
    ASI_CUDA(launch_sm_reduce(ra, pl->nd, max_chunks, st));
    return ASI_OK;      // the core kernel solves for the rows of U_m
  }
  if (pl->small_rank) {
    SmReduceArgs ra;
    max_chunks = build_fused_reduce(pl, w, nullptr, &ra);
    // Few rows: the CTA that factors a mode solves for them too.  Longer modes are products with few partials, which 512 threads
    // reduce no faster, and their rows take the machine: two launches (one layer's compress, one CTA against these:
    // 512 x 384 rank 4 42.7 us, 41.0; 512 x 1024 rank 8 43.0, 38.9; 128 x 4096 rank 8 88.3, 62.5; 128 x 14336 rank 8 213, 118).
    // Conv layers have the partials of the other modes: 32 x 512 x 20 x 20 ranks 3 74.9, 77.5; 8 x 1024 x 20 x 20 ranks 8 89, 85
    RowSolveArgs rs;
    std::memset(&rs, 0, sizeof(rs));
    const bool wide = solves_wide(pl);
    for (int m = 0; m < pl->nd; ++m) {
      float* const U = U_new + pl->u_off[m];
      if (!wide) ra.m[m].U = U;
      rs.Pred[m] = ra.m[m].Pred;
      rs.U[m] = U;
      rs.a[m] = (int)pl->dims[m];
      rs.r[m] = pl->r[m];
      rs.total += rs.a[m];
    }
    rs.Rf = ra.Rf;
    rs.nd = pl->nd;
    ra.large = !wide;
    ASI_CUDA(launch_sm_reduce(ra, pl->nd, max_chunks, st));
    if (wide) ASI_CUDA(launch_row_solve(rs, st));
    return ASI_OK;
  }
  QRArgs qa;
  std::memset(&qa, 0, sizeof(qa));
  for (int m = 0; m < pl->nd; ++m) {
    qa.m[m].Pp = reinterpret_cast<const float*>(w + pl->off_Pp[m]);
    qa.m[m].Pred = reinterpret_cast<double*>(w + pl->off_Pred[m]);
    qa.m[m].Gp = reinterpret_cast<double*>(w + pl->off_Gp[m]);
    qa.m[m].Uout = U_new + pl->u_off[m];
    qa.m[m].a = (int)pl->dims[m];
    qa.m[m].r = pl->r[m];
    qa.m[m].nsplit = pl->nsplit[m];
    qa.m[m].nchunk = pl->nchunk[m];
    qa.m[m].rows = pl->qr_rows[m];
    qa.m[m].count = reinterpret_cast<int*>(w) + 20 + m;
    if (first_core_tc && m == pl->core_order[0]) {   // the first core product reads U_m as a stacked operand
      qa.m[m].bt = reinterpret_cast<__nv_bfloat16*>(w + pl->tcu_off[m]);
      qa.m[m].bt_n = tc_operand_n(pl->r[m]);
      qa.m[m].bt_ld = tc_operand_ld(pl->dims[m]);
    }
  }
  qa.status = reinterpret_cast<int*>(w);
  ASI_CUDA(launch_orth(qa, pl->nd, st));
  return ASI_OK;
}

// A mode product: the register-tiled streaming kernel when a large tensor fits it (strided fibers, contiguous outputs
// per (o, j)), else the grouped SIMT product.
// first: the first kernel of a call.
cudaError_t stream_modeprod(const asi_plan* pl, const ModeProdArgs& a, bool x_bf16, bool first, cudaStream_t st) {
  const bool fits = !(pl->d.flags & ASI_FLAG_GENERIC_ONLY) && a.si == 1 && a.sj == a.I &&
                    a.so == (int64_t)a.n_out * a.I && a.Q * a.a >= (1 << 20) &&
                    a.I >= 32 && wfiber_supported(a.O, a.a, a.I, a.n_out);
  const bool f2 = fits && fiber2_supported(a.O, a.a, a.I, a.n_out, x_bf16) &&
                  (reinterpret_cast<uintptr_t>(a.X) & 15u) == 0 && (reinterpret_cast<uintptr_t>(a.Y) & 15u) == 0;
  if (!fits) {
    GemmGroup g;
    g.np = 0;
    g.clear = nullptr;
    gemm_add(&g, gemm_project(a.X, a.B, a.Y, a.O, a.a, a.I, a.n_out, a.so, a.sj, a.si, x_bf16));
    return launch_gemm_group(g, x_bf16, st);
  }
  Fiber2Args f;
  std::memset(&f, 0, sizeof(f));
  f.X = a.X;
  f.U = a.B;
  f.ldu = a.n_out;
  f.Y = a.Y;
  f.y_so = a.so;
  f.y_sj = a.sj;
  f.O = a.O; f.I = a.I; f.a = (int)a.a; f.r = a.n_out;
  f.n_tiles = fiber2_tiles(a.O, a.I);
  f.project_only = 1;
  f.first = first;
  if (!f2) return launch_wfiber(f, wfiber_grid(a.O, a.a, a.I, a.n_out), x_bf16, st);
  return launch_fiber2(f, fiber2_grid(a.O, a.a, a.I, a.n_out, x_bf16, (pl->d.flags & ASI_FLAG_SHARE_SM) != 0),
                       x_bf16, st);
}

// Orthogonalize, then core = A x_1 U_1^T ... x_n U_n^T (Algorithm 1, core update with U^T).
asi_status_t finish_compress(const asi_plan* pl, const void* act, float* U_new, float* core,
                             char* w, const float* gram_U_prev, bool tc_ready, int beside, cudaStream_t st) {
  // the first core product runs on the tensor cores when its mode does: after a warm step the operand's zero columns
  // are there from the split of U_prev and Orthogonalize fills in the rest, a cold start splits U_new here
  const int m0 = pl->core_order[0];
  const bool tc_core = pl->tc_mode[m0] == 1 && (reinterpret_cast<uintptr_t>(act) & 15u) == 0;
  asi_status_t qs = orthogonalize_all(pl, U_new, w, gram_U_prev, tc_core && tc_ready, st);
  if (qs != ASI_OK) return qs;
  if (tc_core && !tc_ready) {
    TcSplitArgs sp;
    sp.n = 0;
    sp.clear = nullptr;
    tc_add_split(&sp, U_new + pl->u_off[m0], pl->mv[m0].a, pl->r[m0], w + pl->tcu_off[m0]);
    ASI_CUDA(launch_tc_split(sp, st));
  }
  if (pl->fast_compress) {
    SmCoreArgs c;
    build_fused_core(pl, act, U_new, core, w, gram_U_prev != nullptr, &c);
    ASI_CUDA(launch_sm_core(c, pl->fast_R, pl->bf16, beside, st));
    return ASI_OK;
  }
  int64_t cd[ASI_MAX_MODES];
  for (int m = 0; m < pl->nd; ++m) cd[m] = pl->dims[m];
  const void* src = act;
  bool src_bf16 = pl->bf16;
  for (int s = 0; s < pl->nd; ++s) {
    const int m = pl->core_order[s];
    ModeProdArgs a;
    a.X = src;
    a.B = U_new + pl->u_off[m];
    a.O = 1;
    a.I = 1;
    for (int j = 0; j < m; ++j) a.O *= cd[j];
    for (int j = m + 1; j < pl->nd; ++j) a.I *= cd[j];
    a.a = cd[m];
    a.Q = a.O * a.I;
    a.n_out = pl->r[m];
    a.so = (int64_t)pl->r[m] * a.I;
    a.sj = a.I;
    a.si = 1;
    float* dst = (s == pl->nd - 1) ? core : reinterpret_cast<float*>(w + pl->off_T[s & 1]);
    a.Y = dst;
    if (s == 0 && tc_core) {
      const ModeView& v = pl->mv[m];
      const TcCall t = {act, w + pl->tcu_off[m], dst, nullptr, 0, v.O, v.a, v.I, 0, v.r, 1, 0};
      ASI_CUDA(launch_tc_group(&t, 1, reinterpret_cast<int*>(w), stalls(pl), st));
    } else {
      ASI_CUDA(stream_modeprod(pl, a, src_bf16, false, st));
    }
    if (s == 0 && pl->core_tok) {
      CoreTokArgs t;
      t.T = dst;
      t.core = core;
      t.r3 = pl->r[pl->nd - 1];
      if (pl->nd == 3) {
        t.U1 = U_new + pl->u_off[0]; t.U2 = U_new + pl->u_off[1];
        t.B = (int)pl->dims[0]; t.N = (int)pl->dims[1]; t.r1 = pl->r[0]; t.r2 = pl->r[1];
      } else {
        t.U1 = nullptr; t.U2 = U_new + pl->u_off[0];
        t.B = 1; t.N = (int)pl->dims[0]; t.r1 = 1; t.r2 = pl->r[0];
      }
      ASI_CUDA(launch_core_tok(t, st));
      break;
    }
    cd[m] = pl->r[m];
    src = dst;
    src_bf16 = false;
    if (s == 0 && pl->core_tail) {
      CoreTailArgs t;
      std::memset(&t, 0, sizeof(t));
      t.T = dst;
      t.U2 = U_new + pl->u_off[1]; t.U3 = U_new + pl->u_off[2]; t.U4 = U_new + pl->u_off[3];
      t.part = reinterpret_cast<float*>(w + pl->off_ctp);
      t.core = core;
      t.counter = reinterpret_cast<int*>(w) + 32;
      t.r1 = pl->r[0]; t.r2 = pl->r[1]; t.r3 = pl->r[2]; t.r4 = pl->r[3];
      t.C = (int)pl->dims[1]; t.H = (int)pl->dims[2]; t.W = (int)pl->dims[3];
      ASI_CUDA(launch_core_tail(t, st));
      break;
    }
  }
  return ASI_OK;
}

// Side streams of the batched entry points (and of asi_step_host's second copy): the layers of a step are independent, so their
// kernel chains run beside one another on up to kLanes streams that fork from and join the caller's stream by events.  A call borrows a set
// for the time it enqueues and hands it back (a set may serve the next call while its kernels still run: a stream
// only orders work).  At most kMaxSets sets exist; they are destroyed with the last plan.  No set -- or a caller that
// is capturing a graph, whose capture would otherwise keep the streams -- means one chain after another.
constexpr int kLanes = 8, kMaxSets = 8;
struct LaneSet {
  int device;
  cudaStream_t s[kLanes];
  cudaEvent_t fork, join[kLanes];
};
std::mutex g_lane_mu;
std::vector<LaneSet*> g_lane_idle;
int g_lane_sets = 0;                                 // idle and borrowed
long g_plans = 0;                                    // live plans (under g_lane_mu)

void destroy_lanes(LaneSet* l) {
  for (int i = 0; i < kLanes; ++i) {
    if (l->s[i]) cudaStreamDestroy(l->s[i]);
    if (l->join[i]) cudaEventDestroy(l->join[i]);
  }
  if (l->fork) cudaEventDestroy(l->fork);
  delete l;
}

LaneSet* borrow_lanes(cudaStream_t st) {
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  int dev = -1;
  if (cudaStreamIsCapturing(st, &cap) != cudaSuccess || cap != cudaStreamCaptureStatusNone ||
      cudaGetDevice(&dev) != cudaSuccess) {
    (void)cudaGetLastError();
    return nullptr;
  }
  std::lock_guard<std::mutex> lock(g_lane_mu);
  for (size_t i = 0; i < g_lane_idle.size(); ++i)
    if (g_lane_idle[i]->device == dev) {
      LaneSet* l = g_lane_idle[i];
      g_lane_idle.erase(g_lane_idle.begin() + i);
      return l;
    }
  if (g_lane_sets >= kMaxSets) return nullptr;
  g_lane_idle.reserve(kMaxSets);                     // handing a set back never allocates
  LaneSet* l = new (std::nothrow) LaneSet;
  if (!l) return nullptr;
  std::memset(l, 0, sizeof(*l));
  l->device = dev;
  bool ok = cudaEventCreateWithFlags(&l->fork, cudaEventDisableTiming) == cudaSuccess;
  for (int i = 0; ok && i < kLanes; ++i)
    ok = cudaStreamCreateWithFlags(&l->s[i], cudaStreamNonBlocking) == cudaSuccess &&
         cudaEventCreateWithFlags(&l->join[i], cudaEventDisableTiming) == cudaSuccess;
  if (!ok) {
    (void)cudaGetLastError();
    destroy_lanes(l);
    return nullptr;
  }
  ++g_lane_sets;
  return l;
}

void return_lanes(LaneSet* l) {
  std::lock_guard<std::mutex> lock(g_lane_mu);
  g_lane_idle.push_back(l);
}

// the batched entry points keep lists on the host: a failed allocation is an error code like any other
asi_status_t no_host_memory() {
  snprintf(g_cuda_err, sizeof(g_cuda_err), "out of host memory");
  return ASI_ERR_CUDA;
}

// What the layers of a batched call write, as address ranges.  Layers that write to the same memory (a workspace that
// two of them share) run one after another, each with launches of its own.
struct Written {
  std::vector<std::pair<uintptr_t, uintptr_t>> r;
  void add(const void* p, size_t bytes) {
    const uintptr_t at = reinterpret_cast<uintptr_t>(p);
    if (bytes) r.emplace_back(at, at + bytes);
  }
  bool apart() {
    std::sort(r.begin(), r.end());
    for (size_t i = 1; i < r.size(); ++i)
      if (r[i].first < r[i - 1].second) return false;
    return true;
  }
};

// Runs n_chains pieces of work, chain c on the caller's stream (c == 0, or all of them when they are not independent) or
// on a lane.
template <typename F>
asi_status_t run_chains(int n_chains, bool independent, cudaStream_t st, F&& chain) {
  LaneSet* l = n_chains > 1 && independent ? borrow_lanes(st) : nullptr;
  asi_status_t rc = ASI_OK;
  cudaError_t e = cudaSuccess;
  const int used = l ? std::min(n_chains - 1, kLanes) : 0;
  if (l) e = cudaEventRecord(l->fork, st);
  for (int i = 0; i < used && e == cudaSuccess; ++i) e = cudaStreamWaitEvent(l->s[i], l->fork, 0);
  for (int c = 0; c < n_chains && rc == ASI_OK && e == cudaSuccess; ++c) {
    try {
      rc = chain(c, (l && c > 0) ? l->s[(c - 1) % kLanes] : st);
    } catch (const std::bad_alloc&) {
      rc = no_host_memory();
    }
  }
  for (int i = 0; i < used; ++i) {                   // joined whatever happened: nothing of this call stays behind
    const cudaError_t e1 = cudaEventRecord(l->join[i], l->s[i]), e2 = cudaStreamWaitEvent(st, l->join[i], 0);
    if (e == cudaSuccess) e = e1 != cudaSuccess ? e1 : e2;
  }
  if (l) return_lanes(l);
  if (rc != ASI_OK) return rc;
  ASI_CUDA(e);
  return ASI_OK;
}

GemmProb simt_expand(const asi_plan* pl, int m, const void* act, const float* V, char* w) {
  const ModeView& v = pl->mv[m];
  return gemm_expand(act, V, reinterpret_cast<float*>(w + pl->off_Pp[m]), v.O, v.a, v.I, v.r, pl->nsplit[m],
                     pl->q_per_split[m], pl->bf16);
}

// The plan of a cold start: P_m = A_m Omega_m by one launch of SIMT products, one of tensor-core products, and the passes of the
// modes that a warm step has on k_mfiber and k_mplane, which take Omega as their V (64 x 128 x 28 x 28 fp32, ranks 4: 72.1 -> 55.7 us).
// These passes are launches of their own, so small tensors stay with the SIMT products (8 x 32 x 24 x 24 ranks 6 33 us with the passes,
// 26 without; 16 x 115 x 24 x 24, a million values, 31 and 35).  Where SIMT products remain for another mode all the same, the line
// lies at two million (15 x 70 x 32 x 33 51 and 46, 24 x 98 x 512 tokens 50 and 44; 49 x 40 x 40 x 40 52 and 56), but for batches of up
// to eight, which these products take badly (3 x 163 x 56 x 56 57 and 66).  The partials of P follow the kernel
asi_plan cold_plan(const asi_plan* pl, const void* act) {
  asi_plan c = *pl;
  const bool on16 = (reinterpret_cast<uintptr_t>(act) & 15u) == 0;
  bool all = true;
  for (int m = 0; m < c.nd; ++m) all = all && (c.cfiber[m] || (c.mplane && m >= 2));
  const bool early = all || (c.d.kind == ASI_CONV2D && c.dims[0] <= 8);
  const bool passes = (!c.bf16 || on16) && c.N >= (early ? 1 << 20 : 1 << 21);
  c.mplane = c.mplane && passes;
  for (int m = 0; m < c.nd; ++m) {
    c.cfiber[m] = c.cfiber[m] && passes;
    if (c.cfiber[m]) {
      c.nsplit[m] = c.cgrid[m];
    } else if (c.mfiber[m] && c.dims[m] > 128) {     // the grouped product of a long mode is not cut as small
      const int64_t Q = c.mv[m].Q, ns = std::min(gemm_expand_splits(c.dims[m], Q), c.nsplit[m]);
      c.q_per_split[m] = ((Q + ns - 1) / ns + 127) / 128 * 128;
      c.nsplit[m] = (int)((Q + c.q_per_split[m] - 1) / c.q_per_split[m]);
    }
  }
  return c;
}

// pl: of cold_plan.  first: nothing of this call is enqueued yet; the first launch here zeroes the status block
asi_status_t expand_modes(const asi_plan* pl, const void* act, const float* const* omega, char* w, bool first,
                          cudaStream_t st) {
  int* const status = reinterpret_cast<int*>(w);
  bool clear = first;
  const bool on16 = (reinterpret_cast<uintptr_t>(act) & 15u) == 0, planes = pl->mplane;
  GemmGroup g;
  g.np = 0;
  TcSplitArgs sp;
  sp.n = 0;
  TcCall t[3];
  for (int m = 0; m < pl->nd; ++m) {
    const ModeView& v = pl->mv[m];
    if (pl->cfiber[m] || (planes && m >= 2)) continue;
    if (pl->tc_mode[m] && on16) {
      t[sp.n] = {act, w + pl->tcv_off[m], reinterpret_cast<float*>(w + pl->off_Pp[m]), nullptr, 0, v.O, v.a, v.I,
                 pl->q_per_split[m], v.r, pl->nsplit[m], 1};
      tc_add_split(&sp, omega[m], v.Q, v.r, w + pl->tcv_off[m]);
    } else {
      gemm_add(&g, simt_expand(pl, m, act, omega[m], w));
    }
  }
  g.clear = clear ? status : nullptr;
  bool head = true;                                  // the first launch here waits for Omega; those behind it find it there
  if (g.np) {
    ASI_CUDA(launch_gemm_group(g, pl->bf16, st));
    clear = head = false;
  }
  if (planes) {
    PlaneArgs a{};
    a.X = act;
    a.U3 = omega[2];
    a.U4 = omega[3];
    a.Pp3 = reinterpret_cast<float*>(w + pl->off_Pp[2]);
    a.Pp4 = reinterpret_cast<float*>(w + pl->off_Pp[3]);
    a.n_planes = pl->dims[0] * pl->dims[1];
    a.H = (int)pl->dims[2];
    a.W = (int)pl->dims[3];
    a.r3 = pl->r[2];
    a.r4 = pl->r[3];
    a.status = status;
    a.stall = stalls(pl);
    a.given = 1;
    a.first = head;
    a.clear = clear ? status : nullptr;
    ASI_CUDA(launch_mplane(a, pl->plane_grid, pl->bf16, st));
    clear = head = false;
  }
  for (int m = 0; m < pl->nd; ++m) {
    if (!pl->cfiber[m]) continue;
    const ModeView& v = pl->mv[m];
    Fiber2Args f;
    std::memset(&f, 0, sizeof(f));
    f.X = act;
    f.U = omega[m];
    f.Pp = reinterpret_cast<float*>(w + pl->off_Pp[m]);
    f.O = v.O; f.I = v.I; f.a = (int)v.a; f.r = v.r;
    f.status = status;
    f.stall = stalls(pl);
    f.given = 1;
    f.first = head;
    f.clear = clear ? status : nullptr;
    ASI_CUDA(launch_mfiber(f, pl->nsplit[m], pl->bf16, st));
    clear = head = false;
  }
  if (sp.n) {
    sp.clear = clear ? status : nullptr;
    ASI_CUDA(launch_tc_split(sp, st));
    ASI_CUDA(launch_tc_group(t, sp.n, status, stalls(pl), st));
  }
  return ASI_OK;
}

}  // namespace

extern "C" {

const char* asi_status_string(asi_status_t s) {
  switch (s) {
    case ASI_OK: return "ok";
    case ASI_ERR_INVALID_ARG: return "invalid argument";
    case ASI_ERR_UNSUPPORTED: return "unsupported configuration";
    case ASI_ERR_RANK_RANGE: return "rank outside [1, min(a_m, b_m)]";
    case ASI_ERR_WORKSPACE: return "workspace too small or misaligned";
    case ASI_ERR_CUDA: return "CUDA runtime error";
    case ASI_ERR_RANK_DEFICIENT: return "rank-deficient subspace iterate";
    case ASI_ERR_TIMEOUT: return "bounded device wait expired";
  }
  return "unknown status";
}

const char* asi_last_cuda_error(void) { return g_cuda_err; }

asi_status_t asi_plan_create(const asi_layer_desc_t* desc, asi_plan_t** out) {
  if (!desc || !out) return ASI_ERR_INVALID_ARG;
  const asi_layer_desc_t& d = *desc;
  if (d.kind != ASI_CONV2D && d.kind != ASI_LINEAR) return ASI_ERR_INVALID_ARG;
  if (d.in_dtype != ASI_F32 && d.in_dtype != ASI_BF16) return ASI_ERR_INVALID_ARG;
  if (d.kind == ASI_CONV2D && d.ndim != 4) return ASI_ERR_UNSUPPORTED;
  if (d.kind == ASI_LINEAR && d.ndim != 2 && d.ndim != 3) return ASI_ERR_UNSUPPORTED;
  if (d.cout < 1) return ASI_ERR_INVALID_ARG;
  int64_t N = 1;
  for (int m = 0; m < d.ndim; ++m) {
    if (d.dims[m] < 1 || d.dims[m] > (int64_t)1 << 31) return ASI_ERR_INVALID_ARG;
    N *= d.dims[m];
    if (N > (int64_t)1 << 40) return ASI_ERR_UNSUPPORTED;
  }
  for (int m = 0; m < d.ndim; ++m) {
    const int64_t a = d.dims[m], b = N / a;
    if (d.ranks[m] < 1 || d.ranks[m] > std::min(a, b)) return ASI_ERR_RANK_RANGE;
    if (d.ranks[m] > ASI_MAX_RANK) return ASI_ERR_UNSUPPORTED;
  }
  int64_t Ho = 0, Wo = 0;
  if (d.kind == ASI_CONV2D) {
    if (d.kh < 1 || d.kw < 1 || d.stride_h < 1 || d.stride_w < 1 || d.pad_h < 0 || d.pad_w < 0 ||
        d.groups < 1)
      return ASI_ERR_INVALID_ARG;
    if (d.dil_h != 1 || d.dil_w != 1) return ASI_ERR_UNSUPPORTED;
    if (d.dims[1] % d.groups || d.cout % d.groups) return ASI_ERR_INVALID_ARG;
    if (d.kh > 16 || d.kw > 16) return ASI_ERR_UNSUPPORTED;
    const int64_t hn = d.dims[2] + 2 * d.pad_h - d.kh, wn = d.dims[3] + 2 * d.pad_w - d.kw;
    if (hn < 0 || wn < 0) return ASI_ERR_INVALID_ARG;
    Ho = hn / d.stride_h + 1;
    Wo = wn / d.stride_w + 1;
  }
  asi_plan* pl = new (std::nothrow) asi_plan;
  if (!pl) return ASI_ERR_INVALID_ARG;
  std::memset(pl, 0, sizeof(*pl));
  pl->d = d;
  pl->nd = d.ndim;
  pl->N = N;
  pl->bf16 = d.in_dtype == ASI_BF16;
  pl->Ho = Ho;
  pl->Wo = Wo;
  int64_t uo = 0, ce = 1;
  for (int m = 0; m < d.ndim; ++m) {
    pl->dims[m] = d.dims[m];
    pl->r[m] = d.ranks[m];
    pl->u_off[m] = uo;
    uo += d.dims[m] * d.ranks[m];
    ce *= d.ranks[m];
  }
  pl->u_elems = uo;
  pl->core_elems = ce;
  if (d.kind == ASI_CONV2D) {
    pl->dy_elems = d.dims[0] * d.cout * Ho * Wo;
    pl->dw_elems = (int64_t)d.cout * (d.dims[1] / d.groups) * d.kh * d.kw;
  } else {
    pl->dy_elems = N / d.dims[d.ndim - 1] * d.cout;
    pl->dw_elems = (int64_t)d.cout * d.dims[d.ndim - 1];
  }
  set_mode_views(pl);
  choose_kernels(pl);
  fit_compress(pl);
  layout_wgrad(pl);
  {
    std::lock_guard<std::mutex> lock(g_lane_mu);
    ++g_plans;
  }
  *out = pl;
  return ASI_OK;
}

asi_status_t asi_plan_destroy(asi_plan_t* plan) {
  if (!plan) return ASI_ERR_INVALID_ARG;
  delete plan;
  std::lock_guard<std::mutex> lock(g_lane_mu);
  if (--g_plans == 0) {                              // the last plan takes the side streams with it
    for (LaneSet* l : g_lane_idle) destroy_lanes(l);
    g_lane_sets -= (int)g_lane_idle.size();
    g_lane_idle.clear();
  }
  return ASI_OK;
}

asi_status_t asi_plan_query(const asi_plan_t* pl, asi_plan_info_t* info) {
  if (!pl || !info) return ASI_ERR_INVALID_ARG;
  std::memset(info, 0, sizeof(*info));
  info->compress_ws_bytes = pl->compress_ws;
  info->wgrad_ws_bytes = pl->wgrad_ws;
  double sum_r = 0, sum_r3 = 0;
  for (int m = 0; m < pl->nd; ++m) {
    info->u_offset[m] = pl->u_off[m];
    sum_r += pl->r[m];
    sum_r3 += (double)pl->r[m] * pl->r[m] * pl->r[m];
  }
  info->u_elems = pl->u_elems;
  info->core_elems = pl->core_elems;
  info->act_elems = pl->N;
  info->dy_elems = pl->dy_elems;
  info->dw_elems = pl->dw_elems;
  info->out_h = pl->Ho;
  info->out_w = pl->Wo;
  info->compressed_elems = pl->core_elems + pl->u_elems;
  info->ratio_RC = (double)pl->N / (double)info->compressed_elems;
  info->macs_O_ASI = 2.0 * (double)pl->N * sum_r + sum_r3;
  if (pl->d.kind == ASI_CONV2D) {
    const double B = pl->dims[0], C = pl->dims[1], H = pl->dims[2], W = pl->dims[3];
    const double r1 = pl->r[0], r2 = pl->r[1], r3 = pl->r[2], r4 = pl->r[3];
    const double Co = pl->d.cout, HoWo = (double)pl->Ho * pl->Wo, D2 = (double)pl->d.kh * pl->d.kw;
    info->macs_C_ASI = r1 * B * Co * HoWo + r1 * r2 * r3 * r4 * H + r1 * r2 * r4 * H * W +
                       r1 * r2 * Co * HoWo * D2 + r2 * Co * C * D2;
    info->macs_C_vanilla = D2 * C * Co * B * HoWo;
  } else {
    // linear layers (Sec. 3.1 footnote): Z = dY x_1 U_1^T (x_2 U_2^T), Z4 = Z . core over the leading ranks,
    // dW = Z4 U_last^T -- one term per contraction, like the five terms of the conv cost
    const int nd = pl->nd;
    const double Do = pl->d.cout, Din = pl->dims[nd - 1], rl = pl->r[nd - 1];
    double macs = 0.0, lead = 1.0, rest = Do;
    for (int m = 1; m < nd - 1; ++m) rest *= (double)pl->dims[m];
    for (int m = 0; m < nd - 1; ++m) {
      macs += lead * pl->r[m] * (double)pl->dims[m] * rest;      // contract mode m of the running tensor
      lead *= pl->r[m];
      if (m + 1 < nd - 1) rest /= (double)pl->dims[m + 1];
    }
    macs += lead * rl * Do + rl * Do * Din;
    info->macs_C_ASI = macs;
    info->macs_C_vanilla = (double)pl->N * pl->d.cout;
  }
  return ASI_OK;
}

int32_t asi_launch_count(const asi_plan_t* pl, int32_t which) {
  if (!pl) return -1;
  return which == 0 ? pl->launches_compress : pl->launches_wgrad;
}

// beside: CTAs of the fused layers that a batched call runs next to this one (a choice of kernels, not of results)
static asi_status_t compress_one(const asi_plan* pl, const void* act, const float* U_prev, float* U_new, float* core, void* ws,
                                 size_t ws_bytes, int beside, void* stream) {
  if (!pl || !valid_ptr(act) || !valid_ptr(U_prev) || !valid_ptr(U_new) || !valid_ptr(core))
    return ASI_ERR_INVALID_ARG;
  if (U_prev == U_new) return ASI_ERR_INVALID_ARG;
  asi_status_t s = check_ws(ws, ws_bytes, pl->compress_ws);
  if (s != ASI_OK) return s;
  if (!compress_takes(pl, act)) return ASI_ERR_INVALID_ARG;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  char* w = static_cast<char*>(ws);
  if (pl->fast_compress) {
    if (pl->tile_S) {
      SmTile1Args a;
      build_tile1(pl, act, U_prev, w, &a);
      ASI_CUDA(launch_sm_tile1(a, pl->tile_S, pl->fast_R, pl->bf16, st));
    } else {
      SmPass1Args a;
      build_fused_pass1(pl, act, U_prev, w, &a);
      ASI_CUDA(launch_sm_pass1(a, pl->fast_kind, pl->fast_R, pl->bf16, st));
    }
    return finish_compress(pl, act, U_new, core, w, U_prev, false, beside, st);
  }
  // The first kernel waits for the stream's earlier work and clears the status block; the mode passes behind it do not depend
  // on one another (each waits for its predecessor before it ends, so that what follows the last one sees all of them).
  int* const status = reinterpret_cast<int*>(w);
  bool first = true;
  auto take_clear = [&]() {
    int* c = first ? status : nullptr;
    first = false;
    return c;
  };
  GemmGroup gp, ge;
  gp.np = ge.np = 0;
  gp.clear = ge.clear = nullptr;
  bool tc[ASI_MAX_MODES] = {false, false, false, false};
  for (int m = 0; m < pl->nd; ++m) {
    const ModeView& v = pl->mv[m];
    if (pl->fiber[m] || (pl->plane && m >= 2)) continue;
    float* V = reinterpret_cast<float*>(w + pl->v_off[m]);
    tc[m] = pl->tc_mode[m] != 0 && (reinterpret_cast<uintptr_t>(act) & 15u) == 0;
    if (tc[m]) continue;
    gemm_add(&gp, gemm_project(act, U_prev + pl->u_off[m], V, v.O, v.a, v.I, v.r, v.I * v.r, 1, v.r, pl->bf16));
    gemm_add(&ge, simt_expand(pl, m, act, V, w));
  }
  // tensor-core modes: split U_m^{prev}, then V_m = A_m^T U_m (left as the stacked operand), then P_m = A_m V_m
  TcSplitArgs sp;
  sp.n = 0;
  TcCall proj[3], expd[3];
  for (int m = 0; m < pl->nd; ++m) {
    if (!tc[m]) continue;
    const ModeView& v = pl->mv[m];
    char* bu = w + pl->tcu_off[m];
    char* bv = w + pl->tcv_off[m];
    proj[sp.n] = {act, bu, nullptr, bv, tc_operand_ld(v.Q), v.O, v.a, v.I, 0, v.r, 1, 0};
    expd[sp.n] = {act, bv, reinterpret_cast<float*>(w + pl->off_Pp[m]), nullptr, 0, v.O, v.a, v.I, pl->q_per_split[m],
                  v.r, pl->nsplit[m], 1};
    tc_add_split(&sp, U_prev + pl->u_off[m], v.a, v.r, bu);
  }
  if (sp.n) {
    sp.clear = take_clear();
    ASI_CUDA(launch_tc_split(sp, st));
  }
  if (pl->plane) {
    PlaneArgs g;
    g.X = act;
    g.U3 = U_prev + pl->u_off[2];
    g.U4 = U_prev + pl->u_off[3];
    g.Pp3 = reinterpret_cast<float*>(w + pl->off_Pp[2]);
    g.Pp4 = reinterpret_cast<float*>(w + pl->off_Pp[3]);
    g.n_planes = pl->dims[0] * pl->dims[1];
    g.S = (int)pl->dims[2];
    g.H = (int)pl->dims[2];
    g.W = (int)pl->dims[3];
    g.r3 = pl->r[2];
    g.r4 = pl->r[3];
    g.status = status;
    g.stall = stalls(pl);
    g.first = first;
    g.clear = take_clear();
    const bool mma = pl->mplane && (!pl->bf16 || (reinterpret_cast<uintptr_t>(act) & 15u) == 0);   // else: odd bf16 addresses
    if (mma) ASI_CUDA(launch_mplane(g, pl->plane_grid, pl->bf16, st));
    else ASI_CUDA(pl->plane2 ? launch_plane2(g, pl->plane_grid, pl->bf16, st) : launch_wplane(g, pl->plane_grid, pl->bf16, st));
  }
  for (int m = 0; m < pl->nd; ++m) {
    const ModeView& v = pl->mv[m];
    if (!pl->fiber[m] || (pl->plane && m >= 2)) continue;
    if (pl->mfiber[m] || pl->fiber2[m] || pl->wfiber[m]) {
      Fiber2Args f;
      std::memset(&f, 0, sizeof(f));
      f.X = act;
      f.U = U_prev + pl->u_off[m];
      f.ldu = v.r;
      f.Pp = reinterpret_cast<float*>(w + pl->off_Pp[m]);
      f.O = v.O; f.I = v.I; f.a = (int)v.a; f.r = v.r;
      f.n_tiles = fiber2_tiles(v.O, v.I);
      f.first = first;
      f.clear = take_clear();
      f.status = status;
      f.stall = stalls(pl);
      const bool mma = pl->mfiber[m] && (!pl->bf16 || (reinterpret_cast<uintptr_t>(act) & 15u) == 0);
      if (mma) ASI_CUDA(launch_mfiber(f, pl->fiber_grid[m], pl->bf16, st));
      else ASI_CUDA(pl->wfiber[m] ? launch_wfiber(f, pl->fiber_grid[m], pl->bf16, st)
                             : launch_fiber2(f, pl->fiber_grid[m], pl->bf16, st));
    } else {
      FiberArgs f;
      f.X = act;
      f.U = U_prev + pl->u_off[m];
      f.Pp = reinterpret_cast<float*>(w + pl->off_Pp[m]);
      f.O = v.O; f.a = v.a; f.I = v.I;
      f.n_tiles = fiber_tiles(v.O, v.a, v.I);
      f.r = v.r;
      f.vec4 = (!pl->bf16 && v.I % 4 == 0 && (reinterpret_cast<uintptr_t>(act) & 15u) == 0) ? 1 : 0;
      f.clear = take_clear();
      ASI_CUDA(launch_fiber(f, pl->fiber_grid[m], pl->bf16, st));
    }
  }
  if (gp.np) {
    gp.clear = take_clear();
    ASI_CUDA(launch_gemm_group(gp, pl->bf16, st));
    ASI_CUDA(launch_gemm_group(ge, pl->bf16, st));
  }
  if (sp.n) {
    ASI_CUDA(launch_tc_group(proj, sp.n, status, stalls(pl), st));
    ASI_CUDA(launch_tc_group(expd, sp.n, status, stalls(pl), st));
  }
  return finish_compress(pl, act, U_new, core, w, nullptr, sp.n > 0, beside, st);
}

asi_status_t asi_compress(const asi_plan_t* pl, const void* act, const float* U_prev, float* U_new,
                          float* core, void* ws, size_t ws_bytes, void* stream) {
  return compress_one(pl, act, U_prev, U_new, core, ws, ws_bytes, 0, stream);
}

// ---------------------------------------------------------------------------------------------
// Batched entry points: the layers a training step compresses together (Algorithm 1 runs once per
// fine-tuned layer and step; Sec. 4 fine-tunes the last 2..4 layers).  Layers on the fused small-map path
// that share a kernel variant go through ONE launch of each kernel stage, their argument blocks in a
// table the CTAs index; these groups and the remaining layers are chains that run side by side (run_chains).
// ---------------------------------------------------------------------------------------------
namespace {
// layers that share launches
struct Variant {
  int kind, tile, R, bf16;
  explicit Variant(const asi_plan* p) : kind(p->fast_kind), tile(p->tile_S), R(p->fast_R), bf16(p->bf16 ? 1 : 0) {}
  bool operator==(const Variant& o) const { return kind == o.kind && tile == o.tile && R == o.R && bf16 == o.bf16; }
};
}  // namespace

asi_status_t asi_compress_batched(const asi_plan_t* const* plans, const void* const* acts,
                                  const float* const* U_prev, float* const* U_new, float* const* cores,
                                  void* const* ws, const size_t* ws_bytes, int32_t n, void* stream) try {
  if (!plans || !acts || !U_prev || !U_new || !cores || !ws || !ws_bytes || n < 1 || n > 4096)
    return ASI_ERR_INVALID_ARG;
  Written out;
  for (int i = 0; i < n; ++i) {
    const asi_plan* pl = plans[i];
    if (!pl || !valid_ptr(acts[i]) || !valid_ptr(U_prev[i]) || !valid_ptr(U_new[i]) || !valid_ptr(cores[i]))
      return ASI_ERR_INVALID_ARG;
    if (U_prev[i] == U_new[i]) return ASI_ERR_INVALID_ARG;
    const asi_status_t s = check_ws(ws[i], ws_bytes[i], pl->compress_ws);
    if (s != ASI_OK) return s;
    if (!compress_takes(pl, acts[i])) return ASI_ERR_INVALID_ARG;
    for (int j = 0; j < i; ++j)
      if (ws[j] == ws[i]) return ASI_ERR_INVALID_ARG;            // every layer needs a workspace of its own
    out.add(ws[i], pl->compress_ws);
    out.add(U_new[i], (size_t)pl->u_elems * 4);
    out.add(cores[i], (size_t)pl->core_elems * 4);
  }
  const bool apart = out.apart();
  // chains: one per group of fused layers of a variant, one per other layer
  std::vector<char> done(n, 0);
  std::vector<std::vector<int>> chains;
  const int maxb = sm_max_batch();
  for (int i = 0; i < n; ++i) {
    if (done[i]) continue;
    std::vector<int> grp(1, i);
    // layers whose activations are read value by value have launches of their own
    if (plans[i]->fast_compress && apart && four_aligned(plans[i], acts[i])) {
      const Variant v(plans[i]);
      for (int j = i + 1; j < n && (int)grp.size() < maxb; ++j) {
        const asi_plan* q = plans[j];
        if (!done[j] && q->fast_compress && v == Variant(q) && four_aligned(q, acts[j])) grp.push_back(j);
      }
    }
    for (int j : grp) done[j] = 1;
    chains.push_back(std::move(grp));
  }
  auto of = [&](int c) {                             // CTAs of a chain's core kernel
    int t = 0;
    for (int j : chains[c]) t += plans[j]->fast_compress ? plans[j]->n_tiles_core : 0;
    return t;
  };
  int all = 0;
  for (int c = 0; c < (int)chains.size() && apart; ++c) all += of(c);
  return run_chains((int)chains.size(), apart, static_cast<cudaStream_t>(stream), [&](int c, cudaStream_t st) -> asi_status_t {
    const std::vector<int>& grp = chains[c];
    const int g = (int)grp.size(), i0 = grp[0];
    if (g == 1)
      return compress_one(plans[i0], acts[i0], U_prev[i0], U_new[i0], cores[i0], ws[i0], ws_bytes[i0], all - of(c), st);
    const asi_plan* p0 = plans[i0];
    std::vector<SmPass1Args> pa(p0->tile_S ? 0 : g);
    std::vector<SmTile1Args> ta(p0->tile_S ? g : 0);
    std::vector<SmReduceArgs> ra(g);
    std::vector<SmCoreArgs> ca(g);
    std::vector<int> mc(g);
    for (int k = 0; k < g; ++k) {
      const int j = grp[k];
      char* w = static_cast<char*>(ws[j]);
      if (p0->tile_S) build_tile1(plans[j], acts[j], U_prev[j], w, &ta[k]);
      else build_fused_pass1(plans[j], acts[j], U_prev[j], w, &pa[k]);
      mc[k] = build_fused_reduce(plans[j], w, U_prev[j], &ra[k]);
      build_fused_core(plans[j], acts[j], U_new[j], cores[j], w, true, &ca[k]);
    }
    if (p0->tile_S) ASI_CUDA(launch_sm_tile1_batched(ta.data(), g, p0->tile_S, p0->fast_R, p0->bf16, st));
    else ASI_CUDA(launch_sm_pass1_batched(pa.data(), g, p0->fast_kind, p0->fast_R, p0->bf16, st));
    ASI_CUDA(launch_sm_reduce_batched(ra.data(), mc.data(), g, st));
    ASI_CUDA(launch_sm_core_batched(ca.data(), g, p0->fast_R, p0->bf16, all - of(c), st));
    return ASI_OK;
  });
} catch (const std::bad_alloc&) {
  return no_host_memory();
}

static asi_status_t conv_wgrad_one(const asi_plan* pl, const float* core, const float* U, const void* dY, float* dW, void* ws,
                                   size_t ws_bytes, int beside, void* stream);

asi_status_t asi_wgrad_batched(const asi_plan_t* const* plans, const float* const* cores, const float* const* U,
                               const void* const* dY, float* const* dW, void* const* ws, const size_t* ws_bytes,
                               int32_t n, void* stream) try {
  if (!plans || !cores || !U || !dY || !dW || !ws || !ws_bytes || n < 1 || n > 4096) return ASI_ERR_INVALID_ARG;
  Written out;
  for (int i = 0; i < n; ++i) {
    const asi_plan* pl = plans[i];
    if (!pl || !valid_ptr(cores[i]) || !valid_ptr(U[i]) || !valid_ptr(dY[i]) || !valid_ptr(dW[i]))
      return ASI_ERR_INVALID_ARG;
    const asi_status_t s = check_ws(ws[i], ws_bytes[i], pl->wgrad_ws);
    if (s != ASI_OK) return s;
    if (!element_aligned(pl, dY[i])) return ASI_ERR_INVALID_ARG;
    out.add(ws[i], pl->wgrad_ws);
    out.add(dW[i], (size_t)pl->dw_elems * 4);
  }
  const bool apart = out.apart();
  std::vector<char> done(n, 0);
  std::vector<std::vector<int>> chains;
  const int maxb = sm_max_batch();
  for (int i = 0; i < n; ++i) {
    if (done[i]) continue;
    std::vector<int> grp(1, i);
    if (plans[i]->fast_wgrad && apart)
      for (int j = i + 1; j < n && (int)grp.size() < maxb; ++j)
        if (!done[j] && plans[j]->fast_wgrad && plans[j]->fast_R == plans[i]->fast_R && plans[j]->bf16 == plans[i]->bf16 &&
            plans[j]->wgrad_nt == plans[i]->wgrad_nt)
          grp.push_back(j);
    for (int j : grp) done[j] = 1;
    chains.push_back(std::move(grp));
  }
  auto of = [&](int c) {                             // CTAs of a chain's fused kernel
    int t = 0;
    for (int j : chains[c]) t += plans[j]->fast_wgrad ? plans[j]->d.cout / plans[j]->cpb : 0;
    return t;
  };
  int all = 0;
  for (int c = 0; c < (int)chains.size() && apart; ++c) all += of(c);
  return run_chains((int)chains.size(), apart, static_cast<cudaStream_t>(stream), [&](int c, cudaStream_t st) -> asi_status_t {
    const std::vector<int>& grp = chains[c];
    const int g = (int)grp.size(), i0 = grp[0];
    const asi_plan* p0 = plans[i0];
    if (g == 1)
      return p0->d.kind == ASI_CONV2D ? conv_wgrad_one(p0, cores[i0], U[i0], dY[i0], dW[i0], ws[i0], ws_bytes[i0], all - of(c), st)
                                      : asi_linear_wgrad(p0, cores[i0], U[i0], dY[i0], dW[i0], ws[i0], ws_bytes[i0], st);
    std::vector<SmWgradArgs> wa(g);
    for (int k = 0; k < g; ++k) {
      const int j = grp[k];
      build_fused_wgrad(plans[j], cores[j], U[j], dY[j], dW[j], static_cast<char*>(ws[j]), &wa[k]);
    }
    ASI_CUDA(launch_sm_wgrad_batched(wa.data(), g, p0->fast_R, p0->bf16, all - of(c), st));
    return ASI_OK;
  });
} catch (const std::bad_alloc&) {
  return no_host_memory();
}

// ---------------------------------------------------------------------------------------------
// asi_compress with the workspace in the library image, for callers that may not allocate.
// g_static_ws names the array only in device code; host code must ask the runtime for its device
// address (once per device, with that device current) and hand that address to the kernels.
// ---------------------------------------------------------------------------------------------
static __device__ __align__(256) unsigned char g_static_ws[ASI_STATIC_WS_MAX_BYTES];

asi_status_t asi_compress_static_ws(const asi_plan_t* pl, const void* act, const float* U_prev,
                                    float* U_new, float* core, void* stream) {
  constexpr int kMaxDevices = 64;
  static void* addr_of_device[kMaxDevices] = {};
  static std::mutex setup_lock;
  if (!pl) return ASI_ERR_INVALID_ARG;
  if (pl->compress_ws > (size_t)ASI_STATIC_WS_MAX_BYTES) {
    snprintf(g_cuda_err, sizeof(g_cuda_err),
             "asi_compress_static_ws: the plan needs %zu bytes of scratch, the built-in array holds %u",
             pl->compress_ws, (unsigned)ASI_STATIC_WS_MAX_BYTES);
    return ASI_ERR_WORKSPACE;
  }
  int dev = -1;
  ASI_CUDA(cudaGetDevice(&dev));
  if (dev < 0 || dev >= kMaxDevices) return ASI_ERR_UNSUPPORTED;
  void* ws = nullptr;
  {
    std::lock_guard<std::mutex> guard(setup_lock);
    if (!addr_of_device[dev]) {
      void* p = nullptr;
      ASI_CUDA(cudaGetSymbolAddress(&p, g_static_ws));
      addr_of_device[dev] = p;
    }
    ws = addr_of_device[dev];
  }
  // asi_compress clears the status word and the completion counters itself; everything else in the
  // array is written before it is read.
  return asi_compress(pl, act, U_prev, U_new, core, ws, (size_t)ASI_STATIC_WS_MAX_BYTES, stream);
}

asi_status_t asi_init_factors(const asi_plan_t* pl, const void* act, const float* omega, float* U_new,
                              float* core, void* ws, size_t ws_bytes, void* stream) {
  if (!pl || !valid_ptr(act) || !valid_ptr(omega) || !valid_ptr(U_new) || !valid_ptr(core))
    return ASI_ERR_INVALID_ARG;
  asi_status_t s = check_ws(ws, ws_bytes, pl->compress_ws);
  if (s != ASI_OK) return s;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  char* w = static_cast<char*>(ws);
  if (!element_aligned(pl, act)) return ASI_ERR_INVALID_ARG;
  const float* om[ASI_MAX_MODES];
  for (int m = 0; m < pl->nd; ++m) {
    om[m] = omega;
    omega += pl->mv[m].Q * pl->r[m];
  }
  const asi_plan cold = cold_plan(pl, act);
  s = expand_modes(&cold, act, om, w, true, st);
  if (s != ASI_OK) return s;
  return finish_compress(&cold, act, U_new, core, w, nullptr, false, 0, st);
}

static size_t omega_scratch_bytes(const asi_plan* pl) {
  size_t all = 0;
  for (int m = 0; m < pl->nd; ++m) all += align_up((size_t)pl->mv[m].Q * pl->r[m] * 4, 256);
  return all;
}

size_t asi_init_seeded_ws_bytes(const asi_plan_t* pl) {
  return pl ? align_up(pl->compress_ws, 256) + omega_scratch_bytes(pl) : 0;
}

asi_status_t asi_init_factors_seeded(const asi_plan_t* pl, const void* act, uint64_t seed, float* U_new,
                                     float* core, void* ws, size_t ws_bytes, void* stream) {
  if (!pl || !valid_ptr(act) || !valid_ptr(U_new) || !valid_ptr(core)) return ASI_ERR_INVALID_ARG;
  asi_status_t s = check_ws(ws, ws_bytes, asi_init_seeded_ws_bytes(pl));
  if (s != ASI_OK) return s;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  char* w = static_cast<char*>(ws);
  float* omega = reinterpret_cast<float*>(w + align_up(pl->compress_ws, 256));
  if (!element_aligned(pl, act)) return ASI_ERR_INVALID_ARG;
  FillArgs f;
  size_t at = 0;
  for (int m = 0; m < pl->nd; ++m) {
    f.out[m] = reinterpret_cast<float*>(reinterpret_cast<char*>(omega) + at);
    f.n[m] = pl->mv[m].Q * pl->r[m];
    f.stream[m] = (uint32_t)m;
    at += align_up((size_t)f.n[m] * 4, 256);
  }
  f.clear = reinterpret_cast<int*>(w);
  ASI_CUDA(launch_fill_gaussian(seed, f, pl->nd, st));
  const asi_plan cold = cold_plan(pl, act);
  s = expand_modes(&cold, act, f.out, w, false, st);
  if (s != ASI_OK) return s;
  return finish_compress(&cold, act, U_new, core, w, nullptr, false, 0, st);
}

asi_status_t asi_gaussian_stream(uint64_t seed, uint32_t stream_id, int64_t n, float* out, void* stream) {
  if (n < 0 || (n > 0 && !valid_ptr(out))) return ASI_ERR_INVALID_ARG;
  FillArgs f;
  f.out[0] = out;
  f.n[0] = n;
  f.stream[0] = stream_id;
  f.clear = nullptr;
  ASI_CUDA(launch_fill_gaussian(seed, f, 1, static_cast<cudaStream_t>(stream)));
  return ASI_OK;
}

asi_status_t asi_philox_words(uint64_t seed, uint32_t stream_id, int64_t n_groups, uint32_t* out, void* stream) {
  if (n_groups < 0 || (n_groups > 0 && (!valid_ptr(out) || (reinterpret_cast<uintptr_t>(out) & 15u))))
    return ASI_ERR_INVALID_ARG;
  ASI_CUDA(launch_philox_words(seed, stream_id, n_groups, out, static_cast<cudaStream_t>(stream)));
  return ASI_OK;
}

static asi_status_t conv_wgrad_one(const asi_plan* pl, const float* core, const float* U, const void* dY, float* dW, void* ws,
                                   size_t ws_bytes, int beside, void* stream) {
  if (!pl || !valid_ptr(core) || !valid_ptr(U) || !valid_ptr(dY) || !valid_ptr(dW))
    return ASI_ERR_INVALID_ARG;
  if (pl->d.kind != ASI_CONV2D || !element_aligned(pl, dY)) return ASI_ERR_INVALID_ARG;
  asi_status_t s = check_ws(ws, ws_bytes, pl->wgrad_ws);
  if (s != ASI_OK) return s;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  char* w = static_cast<char*>(ws);
  if (pl->fast_wgrad) {
    SmWgradArgs g;
    build_fused_wgrad(pl, core, U, dY, dW, w, &g);
    ASI_CUDA(launch_sm_wgrad(g, pl->fast_R, pl->bf16, beside, st));
    return ASI_OK;
  }
  float* Z1 = reinterpret_cast<float*>(w + pl->off_Z[0]);
  float* Z3 = reinterpret_cast<float*>(w + pl->off_Z[1]);
  const int64_t B = pl->dims[0], H = pl->dims[2], W = pl->dims[3];
  const int r1 = pl->r[0], r2 = pl->r[1], r3 = pl->r[2], r4 = pl->r[3];
  const int64_t per_sample = (int64_t)pl->d.cout * pl->Ho * pl->Wo;

  ModeProdArgs a;
  // term 1: Z1 = dY x_1 U_1^T
  a.X = dY; a.B = U + pl->u_off[0]; a.Y = Z1;
  a.O = 1; a.a = B; a.I = per_sample; a.Q = per_sample;
  a.n_out = r1;
  a.so = (int64_t)r1 * per_sample; a.sj = per_sample; a.si = 1;
  ASI_CUDA(stream_modeprod(pl, a, pl->bf16, true, st));
  // terms 2-3 in one launch
  ASI_CUDA(launch_z3(core, U + pl->u_off[2], U + pl->u_off[3], Z3, r1 * r2, r3, r4, (int)H, (int)W, st));
  // terms 4 and 5
  ConvTailArgs t;
  t.Z1 = Z1; t.Z3 = Z3; t.U2 = U + pl->u_off[1]; t.dW = dW;
  t.r1 = r1; t.r2 = r2; t.C = (int)pl->dims[1]; t.Cout = pl->d.cout;
  t.H = (int)H; t.W = (int)W; t.Ho = (int)pl->Ho; t.Wo = (int)pl->Wo;
  t.kh = pl->d.kh; t.kw = pl->d.kw; t.sh = pl->d.stride_h; t.sw = pl->d.stride_w;
  t.ph = pl->d.pad_h; t.pw = pl->d.pad_w; t.groups = pl->d.groups;
  if (pl->conv_nsp > 1)
    ASI_CUDA(launch_conv_tail_split(t, reinterpret_cast<float*>(w + pl->off_Z4p), pl->conv_nsp, st));
  else
    ASI_CUDA(launch_conv_tail(t, st));
  return ASI_OK;
}

asi_status_t asi_conv_wgrad(const asi_plan_t* pl, const float* core, const float* U, const void* dY,
                            float* dW, void* ws, size_t ws_bytes, void* stream) {
  return conv_wgrad_one(pl, core, U, dY, dW, ws, ws_bytes, 0, stream);
}

asi_status_t asi_linear_wgrad(const asi_plan_t* pl, const float* core, const float* U, const void* dY,
                              float* dW, void* ws, size_t ws_bytes, void* stream) {
  if (!pl || !valid_ptr(core) || !valid_ptr(U) || !valid_ptr(dY) || !valid_ptr(dW))
    return ASI_ERR_INVALID_ARG;
  if (pl->d.kind != ASI_LINEAR || !element_aligned(pl, dY)) return ASI_ERR_INVALID_ARG;
  asi_status_t s = check_ws(ws, ws_bytes, pl->wgrad_ws);
  if (s != ASI_OK) return s;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  char* w = static_cast<char*>(ws);
  const int64_t B = pl->nd == 3 ? pl->dims[0] : 1, N = pl->nd == 3 ? pl->dims[1] : pl->dims[0], Dout = pl->d.cout;
  const int m2 = pl->nd - 2;                         // the mode contracted first: tokens (two modes: the rows)
  float* Y1 = reinterpret_cast<float*>(w + pl->off_Z[0]);
  float* Z4 = reinterpret_cast<float*>(w + pl->off_Z[1]);
  // Y1[b][o][j] = sum_n dY[b][n][o] U_2[n][j]
  ModeProdArgs a;
  a.X = dY; a.B = U + pl->u_off[m2]; a.Y = Y1;
  a.O = B; a.a = N; a.I = Dout; a.Q = B * Dout;
  a.n_out = pl->r[m2];
  a.so = Dout * a.n_out; a.sj = 1; a.si = a.n_out;
  if (pl->lin_tc && (reinterpret_cast<uintptr_t>(dY) & 15u) == 0) {
    TcSplitArgs sp;
    sp.n = 0;
    sp.clear = reinterpret_cast<int*>(w);
    tc_add_split(&sp, a.B, N, a.n_out, w + pl->off_wtc);
    ASI_CUDA(launch_tc_split(sp, st));
    const TcCall t = {dY, w + pl->off_wtc, Y1, nullptr, 0, B, N, Dout, 0, a.n_out, 1, 0};
    ASI_CUDA(launch_tc_group(&t, 1, reinterpret_cast<int*>(w), stalls(pl), st));
  } else {
    GemmGroup g;
    g.np = 0;
    g.clear = nullptr;
    gemm_add(&g, gemm_project(a.X, a.B, a.Y, a.O, a.a, a.I, a.n_out, a.so, a.sj, a.si, pl->bf16));
    ASI_CUDA(launch_gemm_group(g, pl->bf16, st));
  }
  LinMidArgs mid;
  mid.Y1 = Y1; mid.core = core; mid.Z4 = Z4;
  mid.U1 = pl->nd == 3 ? U + pl->u_off[0] : nullptr;
  mid.B = (int)B; mid.Dout = (int)Dout;
  mid.r1 = pl->nd == 3 ? pl->r[0] : 1;
  mid.r2 = pl->r[m2]; mid.r3 = pl->r[pl->nd - 1];
  ASI_CUDA(launch_lin_mid(mid, st));
  LinTailArgs t;
  t.Z4 = Z4; t.U = U + pl->u_off[pl->nd - 1]; t.dW = dW;
  t.Dout = (int)Dout; t.Din = (int)pl->dims[pl->nd - 1]; t.r = pl->r[pl->nd - 1];
  ASI_CUDA(launch_lin_tail(t, st));
  return ASI_OK;
}

size_t asi_spectrum_ws_bytes(const asi_plan_t* pl) { return pl ? spectrum_ws_bytes(pl) : 0; }

asi_status_t asi_mode_spectrum(const asi_plan_t* pl, const void* act, double* eig, double* energy, void* ws,
                               size_t ws_bytes, void* stream) {
  if (!pl || !valid_ptr(act) || !eig || !energy) return ASI_ERR_INVALID_ARG;
  const asi_status_t s = check_ws(ws, ws_bytes, spectrum_ws_bytes(pl));
  if (s != ASI_OK) return s;
  ASI_CUDA(launch_mode_spectrum(pl, act, eig, energy, static_cast<char*>(ws), static_cast<cudaStream_t>(stream)));
  return ASI_OK;
}

asi_status_t asi_pick_ranks(const asi_plan_t* pl, const double* eig, const double* energy, double eps,
                            int32_t r_max, int32_t* ranks, void* stream) {
  if (!pl || !eig || !energy || !ranks || !(eps > 0.0) || !(eps <= 1.0) || r_max < 1) return ASI_ERR_INVALID_ARG;
  ASI_CUDA(launch_pick_ranks(pl, eig, energy, eps, r_max, ranks, static_cast<cudaStream_t>(stream)));
  return ASI_OK;
}

size_t asi_perplexity_ws_bytes(void) { return perplexity_ws_bytes(); }

asi_status_t asi_perplexity(const float* dW, const float* dW_approx, int64_t n, double* out, void* ws,
                            size_t ws_bytes, void* stream) {
  if (!dW || !dW_approx || !out || n < 1) return ASI_ERR_INVALID_ARG;
  const asi_status_t s = check_ws(ws, ws_bytes, perplexity_ws_bytes());
  if (s != ASI_OK) return s;
  ASI_CUDA(launch_perplexity(dW, dW_approx, n, out, static_cast<double*>(ws), static_cast<cudaStream_t>(stream)));
  return ASI_OK;
}

size_t asi_step_host_arena_bytes(const asi_plan_t* pl) {
  if (!pl) return 0;
  const size_t eb = elem_bytes(pl);
  size_t off = 0;
  off = align_up(off + (size_t)pl->N * eb, 256);
  off = align_up(off + (size_t)pl->dy_elems * eb, 256);
  off = align_up(off + (size_t)pl->u_elems * 4, 256) * 1;
  off = align_up(off + (size_t)pl->u_elems * 4, 256);
  off = align_up(off + (size_t)pl->core_elems * 4, 256);
  off = align_up(off + (size_t)pl->dw_elems * 4, 256);
  off += align_up(std::max(pl->compress_ws, pl->wgrad_ws), 256);
  return off;
}

asi_status_t asi_step_host(const asi_plan_t* pl, const void* act_host, const void* dY_host,
                           const float* U_prev_host, float* U_new_host, float* core_host,
                           float* dW_host, void* arena, size_t arena_bytes, void* stream) {
  if (!pl || !act_host || !dY_host || !U_prev_host || !U_new_host || !core_host || !dW_host)
    return ASI_ERR_INVALID_ARG;
  asi_status_t s = check_ws(arena, arena_bytes, asi_step_host_arena_bytes(pl));
  if (s != ASI_OK) return s;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const size_t eb = elem_bytes(pl);
  char* base = static_cast<char*>(arena);
  size_t off = 0;
  char* d_act = base + off; off = align_up(off + (size_t)pl->N * eb, 256);
  char* d_dy = base + off; off = align_up(off + (size_t)pl->dy_elems * eb, 256);
  float* d_up = reinterpret_cast<float*>(base + off); off = align_up(off + (size_t)pl->u_elems * 4, 256);
  float* d_un = reinterpret_cast<float*>(base + off); off = align_up(off + (size_t)pl->u_elems * 4, 256);
  float* d_core = reinterpret_cast<float*>(base + off); off = align_up(off + (size_t)pl->core_elems * 4, 256);
  float* d_dw = reinterpret_cast<float*>(base + off); off = align_up(off + (size_t)pl->dw_elems * 4, 256);
  void* d_ws = base + off;
  const size_t ws_bytes = align_up(std::max(pl->compress_ws, pl->wgrad_ws), 256);
  ASI_CUDA(cudaMemcpyAsync(d_act, act_host, (size_t)pl->N * eb, cudaMemcpyHostToDevice, st));
  ASI_CUDA(cudaMemcpyAsync(d_up, U_prev_host, (size_t)pl->u_elems * 4, cudaMemcpyHostToDevice, st));
  // The gradient follows the activation over the bus while compress runs (64 x 128 x 28 x 28 fp32: 1053 -> 996 us), on a side stream that
  // forks behind the activation's copy -- two copies at once would share the bus and hold up compress -- and joins before
  // the weight gradient.  Without one (a capture, all sets lent) the copies stay on the caller's stream
  LaneSet* l = borrow_lanes(st);
  cudaError_t e = cudaSuccess, e1 = cudaSuccess;
  if (l) {
    e = cudaEventRecord(l->fork, st);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(l->s[0], l->fork, 0);
    if (e == cudaSuccess) e = cudaMemcpyAsync(d_dy, dY_host, (size_t)pl->dy_elems * eb, cudaMemcpyHostToDevice, l->s[0]);
  }
  s = e == cudaSuccess ? asi_compress(pl, d_act, d_up, d_un, d_core, d_ws, ws_bytes, stream) : ASI_OK;
  if (l) {                                           // joined whatever happened: nothing of this call stays behind
    e1 = cudaEventRecord(l->join[0], l->s[0]);
    if (e1 == cudaSuccess) e1 = cudaStreamWaitEvent(st, l->join[0], 0);
    return_lanes(l);
  }
  if (s != ASI_OK) return s;
  ASI_CUDA(e);
  ASI_CUDA(e1);
  if (!l) ASI_CUDA(cudaMemcpyAsync(d_dy, dY_host, (size_t)pl->dy_elems * eb, cudaMemcpyHostToDevice, st));
  if (pl->d.kind == ASI_CONV2D)
    s = asi_conv_wgrad(pl, d_core, d_un, d_dy, d_dw, d_ws, ws_bytes, stream);
  else
    s = asi_linear_wgrad(pl, d_core, d_un, d_dy, d_dw, d_ws, ws_bytes, stream);
  if (s != ASI_OK) return s;
  ASI_CUDA(cudaMemcpyAsync(U_new_host, d_un, (size_t)pl->u_elems * 4, cudaMemcpyDeviceToHost, st));
  ASI_CUDA(cudaMemcpyAsync(core_host, d_core, (size_t)pl->core_elems * 4, cudaMemcpyDeviceToHost, st));
  ASI_CUDA(cudaMemcpyAsync(dW_host, d_dw, (size_t)pl->dw_elems * 4, cudaMemcpyDeviceToHost, st));
  return ASI_OK;
}

asi_status_t asi_step_host_status(const asi_plan_t* pl, const void* arena, void* stream,
                                  asi_status_t* device_status) {
  if (!pl || !arena || !device_status) return ASI_ERR_INVALID_ARG;
  const size_t eb = elem_bytes(pl);
  size_t off = 0;                                   // the same carve-up as asi_step_host
  off = align_up(off + (size_t)pl->N * eb, 256);
  off = align_up(off + (size_t)pl->dy_elems * eb, 256);
  off = align_up(off + (size_t)pl->u_elems * 4, 256);
  off = align_up(off + (size_t)pl->u_elems * 4, 256);
  off = align_up(off + (size_t)pl->core_elems * 4, 256);
  off = align_up(off + (size_t)pl->dw_elems * 4, 256);
  return asi_poll_status(pl, static_cast<const char*>(arena) + off, stream, device_status);
}

asi_status_t asi_profile_begin(int32_t kernel_id, void** events, int32_t n_pairs) {
  if (kernel_id < 1 || !events || n_pairs < 1) return ASI_ERR_INVALID_ARG;
  g_prof.ev = reinterpret_cast<cudaEvent_t*>(events);
  g_prof.n_pairs = n_pairs;
  g_prof.used = 0;
  g_prof.bytes = 0.0;
  g_prof.id = kernel_id;
  return ASI_OK;
}

int32_t asi_profile_end(double* alg_bytes) {
  const int used = g_prof.used;
  if (alg_bytes) *alg_bytes = g_prof.bytes;
  g_prof = ProfState{0, nullptr, 0, 0, 0.0};
  return used;
}

asi_status_t asi_poll_status(const asi_plan_t* pl, const void* ws, void* stream,
                             asi_status_t* device_status) {
  if (!pl || !ws || !device_status) return ASI_ERR_INVALID_ARG;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  int v = 0;
  ASI_CUDA(cudaMemcpyAsync(&v, ws, sizeof(int), cudaMemcpyDeviceToHost, st));
  ASI_CUDA(cudaStreamSynchronize(st));
  *device_status = static_cast<asi_status_t>(v);
  return ASI_OK;
}

}  // extern "C"
