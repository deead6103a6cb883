// Host-side check of spmv_multi_kernel's launch geometry and of the rule that
// chooses it (launch_geometry.h).  Built and run by tests/test_multi_geometry.py;
// prints "ok" or the first violation and exits non-zero.
#include <cstdio>

#include "launch_geometry.h"

using namespace dfm::geom;

static int fail(const char* what, int nb, int K, int R) {
  std::printf("violation: %s (nb=%d, K=%d, R=%d)\n", what, nb, K, R);
  return 1;
}

int main() {
  const int nbs[] = {1, 3, 6, 10, 15, 21, 28, 36, 45, 55};
  for (int nb : nbs)
    for (int K = 1; K <= kMultiMaxOps; ++K)
      for (int R = 1; R <= kMultiMaxRhs; ++R) {
        const Multi g = multi_geometry(nb, K, R);
        const bool taken = multi_faster(nb, K, R);
        if (taken && (nb == 1 || nb == 55)) return fail("a basis without a kernel", nb, K, R);
        if (taken && g.producers < 1) return fail("taken where it does not fit", nb, K, R);
        // one right-hand side of several operators, two of the small bases: the
        // streamed tiles are faster (measured)
        if (taken && R == 1 && (K > 1 || nb <= 21)) return fail("one right-hand side", nb, K, R);
        if (taken && R == 2 && nb <= 6) return fail("two right-hand sides", nb, K, R);
        // once it is the faster one it stays so
        if (!taken && R > 1 && multi_faster(nb, K, R - 1) && g.producers > 0) return fail("order", nb, K, R);
        if (g.producers < 1) continue;
        const int depth = 1 << g.log_depth, slots = 1 << g.log_slots;
        if (depth > kMultiMaxDepth || slots > kMultiMaxDepth || slots < 2 || slots < depth) return fail("ring", nb, K, R);
        // a barrier's previous phase is consumed by the warps that wait for it
        if (depth % g.producers || depth % g.groups || slots % g.producers || slots % g.groups)
          return fail("depth a multiple of producers and groups", nb, K, R);
        const int threads = 32 * (g.producers + 4 * multi_m_tiles(nb) * g.groups);
        if (threads > 32 * (kMultiMaxProducers + 4 * multi_m_tiles(nb) * multi_max_groups(nb)) || threads > 1024)
          return fail("threads", nb, K, R);
        // bulk copies: 16-byte aligned rows, slots and sizes
        const long long stage = K * op_row_stride(nb) * 4, slot = (long long)R * multi_slot_stride(nb) * 4;
        if (kMultiHead % 128 || stage % 16 || slot % 16 || (multi_slot_stride(nb) * 4) % 16 || (4 * nb * 4) % 16)
          return fail("alignment", nb, K, R);
        // eight right-hand sides in distinct bank groups
        if (multi_slot_stride(nb) / 4 % 2 == 0 || multi_slot_stride(nb) < 4 * nb) return fail("slot stride", nb, K, R);
        // what the last m-tile's unused rows and the padded contraction read past the
        // last stage lies within the slots or the reserve behind them
        const long long rows_end = kMultiHead + 4ll * depth * stage;
        const long long last_read = rows_end - (op_row_stride(nb) - 3ll * nb * nb) * 4 + 16ll * nb * 4;
        if (last_read > g.smem || g.smem > 227 * 1024) return fail("shared memory", nb, K, R);
      }
  std::printf("ok\n");
  return 0;
}
