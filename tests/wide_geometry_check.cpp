// Host-side check of the wide bases' launch geometries on tensor cores and bulk
// copies (launch_geometry.h).  Built and run by tests/test_multi_geometry.py; prints
// "ok" or the first violation and exits non-zero.
#include <cstdio>
#include <initializer_list>

#include "launch_geometry.h"

using namespace dfm::geom;

static int fail(const char* what, int a, int b, long long c) {
  std::printf("violation: %s (%d, %d, %lld)\n", what, a, b, c);
  return 1;
}

int main() {
  for (int np = kWideMmaMinNp; np <= kWideMaxNp; ++np) {
    const WideMma g = wide_mma_geometry(np);
    const int nb = (np + 1) * (np + 2) / 2;
    // every order m >= 1 starts at an even position, so pairs share a 4-byte word
    int pos = np / 2 + 1;
    pos += pos & 1;
    for (int m = 1; m <= np; ++m) pos += 2 * ((np - m) / 2 + 1);
    if (g.nb != nb || g.total != pos || g.total > 256) return fail("positions", np, g.total, pos);
    const int NT = (g.total + 7) / 8;
    if (g.TN < 2 || g.TN > kWideMmaMaxTn || g.WM * g.WN > kWideMmaWarps || g.WM < 1) return fail("warps", np, g.TN, g.WM);
    if (g.rows * g.ntile < g.total || g.rows * (g.ntile - 1) >= g.total || g.rows % 32) return fail("row tiles", np, g.rows, g.ntile);
    if (g.WN * g.TN < NT) return fail("column tiles", np, g.WN, g.TN);
    // staged nodes: room for every position read, 16-byte rows of an odd number of units
    if (g.ldq < g.rows || g.ldp < 8 * NT || g.ldq % 8 || g.ldp % 8 || g.ldq / 8 % 2 == 0 || g.ldp / 8 % 2 == 0)
      return fail("strides", np, g.ldq, g.ldp);
    if (g.smem != 2ll * kWideMmaNodes * (g.ldq + g.ldp) * 4 || g.smem > 220 * 1024) return fail("assembly shared memory", np, 0, g.smem);
  }
  // the orders the FMA kernel assembles faster (measured)
  for (int np = 9; np <= kWideMaxNp; ++np)
    for (long long tets : {6, 162, 750, 48000}) {
      const bool fma = np == 9 || (np <= 11 && tets >= 750);
      if (wide_mma_faster(np, 12 * tets) == fma) return fail("assembly rule", np, (int)tets, 0);
    }
  for (int nb = 55; nb <= 256; ++nb)
    for (int R = 1; R <= kWideApplyMaxRhs; ++R) {
      const WideApply g = wide_apply_geometry(nb, R);
      if (g.stages < kWideApplyGroups || g.stages > kWideApplyMaxStages || g.stages % kWideApplyGroups)
        return fail("stages", nb, R, g.stages);
      // a piece: rounded down by up to 3 floats, its end rounded up to a multiple of 4
      if (g.piece % 4 || g.piece < (3 + kWideApplyChunk * nb + 3) / 4 * 4) return fail("piece", nb, R, g.piece);
      const long long smem = kWideApplyHead + 12ll * g.stages * g.piece + 32ll * R * nb;
      if (g.smem != smem || smem > 227 * 1024 || kWideApplyHead % 16) return fail("application shared memory", nb, R, g.smem);
    }
  // row blocks where they are faster (measured): one right-hand side of the smaller
  // bases, and never a basis the ring does not hold
  for (int nb : {55, 66, 78})
    for (long long tets : {162, 768, 3072})
      if (wide_apply_faster(nb, 1, tets)) return fail("application rule, one", nb, (int)tets, 0);
  for (int nb : {105, 153, 231})
    for (long long tets : {6, 162, 768, 3072})
      for (int R : {1, 2, 3, 8, 19})
        if (!wide_apply_faster(nb, R, tets)) return fail("application rule", nb, (int)tets, R);
  if (wide_apply_faster(55, 2, 768) || !wide_apply_faster(55, 3, 768) || !wide_apply_faster(55, 1, 48) ||
      wide_apply_faster(45, 8, 768) || wide_apply_faster(257, 8, 768))
    return fail("application rule, edges", 55, 2, 0);
  if (wide_apply_geometry(257, 1).stages || wide_apply_geometry(1 << 14, 1).stages) return fail("too large a basis", 257, 1, 0);
  std::printf("ok\n");
  return 0;
}
