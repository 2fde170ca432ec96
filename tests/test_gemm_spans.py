"""Host-side check of the grouped products' index arithmetic: the k that the splits of an expansion take, and where they
find them in the tensor and in the factor, for modes up to far beyond 2^31 columns.  A small program walks the
descriptors the library makes and compares with plain 64-bit arithmetic.  No GPU work."""
import os
import subprocess

import pytest

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include "asi_internal.h"
using namespace asi;
static long long checked = 0;
static const int64_t kBase = 1ll << 45;
static int fail(const char* what, int64_t a, int64_t b) {
  printf("%s: %lld, %lld\n", what, (long long)a, (long long)b);
  exit(1);
}
// k-th column of the span in the tile's first row: the address the kernel forms, from 32-bit k and kin
static void at(const GemmProb& p, const GemmArg& w, int64_t a, int64_t I, int64_t m0, int64_t q, int64_t first) {
  const int64_t k = w.k0 + (q - first);
  if (k < w.k0 || k >= w.K) fail("k outside the span", k, w.K);
  const int64_t o = p.km && w.kin < w.K ? k / w.kin : 0;
  const int64_t x = (int64_t)(uintptr_t)w.X - kBase + (p.km ? o * w.sxo + (k - o * w.kin) : k * w.ld);
  const int64_t want = q / I * a * I + m0 * I + q % I;
  if (x != want) fail("address", x, want);
  if (((int64_t)(uintptr_t)w.B - kBase) / 4 + k * w.ldb != q * p.n) fail("factor row", k, q);
  const int64_t base = (int64_t)(uintptr_t)w.X - kBase;      // lanes without work read there
  if (base < 0 || base >= p.K * a) fail("base", base, p.K * a);
  ++checked;
}
int main(int argc, char** argv) {
  const int64_t O = atoll(argv[1]), a = atoll(argv[2]), I = atoll(argv[3]), Q = O * I;
  const int n = atoi(argv[4]);
  int64_t ns = argc > 5 ? atoll(argv[5]) : gemm_expand_splits(a, Q);
  int64_t kps = ((Q + ns - 1) / ns + 127) / 128 * 128;
  if (argc <= 5) ns = (Q + kps - 1) / kps;               // with a fixed count the last splits may be empty
  const GemmProb p = gemm_expand((const void*)kBase, (const float*)kBase, (float*)kBase, O, a, I, n, (int)ns, kps, true);
  if (p.K != Q || p.M != a || kps > kGemmMaxSpan) fail("sizes", p.K, kps);
  if (gemm_narrow(p) && (Q + kps >= INT32_MAX || a >= INT32_MAX)) fail("narrow", Q, kps);
  if (!gemm_narrow(p) && Q < 1000000) fail("wide", Q, kps);
  const int64_t tiles_m = (a + 31) / 32;
  int64_t next = 0;
  for (int64_t s = 0; s < ns; ++s) {
    const int64_t len = Q - next < kps ? Q - next : kps;
    for (int64_t mt : {(int64_t)0, tiles_m - 1}) {
      const GemmArg w = gemm_tile_arg(p, s * tiles_m + mt, 1);
      if (w.K - w.k0 != len || w.k0 < 0 || w.K < 0) fail("span", w.K - w.k0, len);
      if (w.M != (a - 32 * mt < 32 ? a - 32 * mt : 32)) fail("rows", w.M, mt);
      if (((int64_t)(uintptr_t)w.Y - kBase) / 4 != (s * a + 32 * mt) * n) fail("output", s, mt);
      // ends and middle of the span, and both sides of the first and the last slab end it holds
      const int64_t e0 = (next / I + 1) * I, e1 = (next + len - 1) / I * I;
      for (int64_t q : {next, next + 1, next + len / 2, next + len - 1, e0 - 1, e0, e1 - 1, e1})
        if (q >= next && q < next + len) at(p, w, a, I, 32 * mt, q, next);
    }
    next += len;
  }
  if (next != Q) fail("columns", next, Q);
  // a projection keeps its sizes; a tile of it starts where it should
  const GemmProb v = gemm_project((const void*)kBase, (const float*)kBase, (float*)kBase, O, a, I, n, I * n, 1, n, true);
  if (v.K != a || v.M * v.O != Q) fail("projection", v.K, v.M * v.O);
  const int64_t rows = (v.M + 31) / 32, t = rows * v.O - 1;  // the last tile of the last outer index
  const GemmArg w = gemm_tile_arg(v, t, 1);
  const int64_t m0 = (rows - 1) * 32;
  const int64_t want_x = I == 1 ? m0 * a : (O - 1) * a * I + m0, want_y = (I == 1 ? m0 : (O - 1) * I + m0) * n;
  if ((int64_t)(uintptr_t)w.X - kBase != want_x || ((int64_t)(uintptr_t)w.Y - kBase) / 4 != want_y || w.K != a || w.k0 != 0)
    fail("projected tile", want_x, want_y);
  printf("ok %lld\n", checked);
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory, repo_root):
    from paper_2505_05086_b200 import build
    lib = build.build()
    d = tmp_path_factory.mktemp("spans")
    src, exe = d / "spans.cpp", d / "spans"
    src.write_text(PROGRAM)
    cuda = os.path.dirname(os.path.dirname(os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")))
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", build.CSRC, "-I", os.path.join(repo_root, "include"), "-I",
                    os.path.join(cuda, "include"), "-o", str(exe), str(src), lib, f"-Wl,-rpath,{build.PKG}"], check=True)
    return str(exe)


BIG = 1 << 29


@pytest.mark.parametrize("O,a,I,n,ns", [
    (1, 8, 192, 4, None), (8, 3, 49, 5, None), (5, 7, 1, 2, None), (1000, 40, 49, 8, 7),        # ordinary modes
    (1, 2, 1 << 31, 1, None), (1, 128, 4096 * 4096 * 4, 4, 148), (1, 1, (1 << 33) + 5, 1, None),   # one slab beyond 2^31
    (2, 2, 1 << 30, 1, None), (2, 2, 1 << 30, 1, 148), (3, 5, BIG - 4, 3, None), (3, 5, BIG, 3, None),   # slabs about as long
    (3, 5, BIG + 4, 3, None), (7, 2, (1 << 32) + 12, 2, None),                                     # as a span, and longer
    ((1 << 26) + 3, 9, 49, 9, None), ((1 << 32) + 1, 4, 1, 3, None), ((1 << 31) - 1, 8, 3, 8, 296),    # many short slabs
])
def test_the_splits_cover_every_column_once(program, O, a, I, n, ns):
    args = [str(v) for v in (O, a, I, n)] + ([] if ns is None else [str(ns)])
    r = subprocess.run([program] + args, capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout.startswith("ok"), r.stdout
