// Host-side check of the launch configurations that the autotuner may pick against
// the table in lgt.h (compiled and run by test_launch_table_host.py): every pair of
// sweep format and gauge has kernels in just the configurations documented for it.
#include <cstdio>
#include <initializer_list>

#include "lgt_internal.h"

using namespace lgt;

static int check(const char *what, int fmt, int gauge, std::initializer_list<int> want) {
  for (int c = -1; c <= LGT_NCFG_TUNED; c++) {
    bool in = false;
    for (int w : want) in = in || w == c;
    if (lgt_cfg_supported_gauge(fmt, gauge, c) != in)
      return printf("%s, gauge %d, configuration %d: %s\n", what, gauge, c, in ? "missing" : "not documented");
  }
  return 0;
}

int main() {
  for (int gauge : {(int)GAUGE_LANDAU, (int)GAUGE_COULOMB}) {
    if (check("FP64", FMT_F64, gauge, {0, 1, 2, 3, 16})) return 1;
    if (check("FP32 pairs", FMT_PAIR, gauge, {0, 1, 2, 3})) return 1;
    if (check("FP32-18", FMT_F32_18, gauge, {0, 1, 2, 3, 4, 5, 6, 8, 9, 11})) return 1;
    if (check("FP32-12", FMT_F32_12, gauge, {0, 1, 2, 3, 4, 5, 6, 7, 8, 9, 10, 11, 12, 13, 14, 15})) return 1;
    if (check("anchored polish", FMT_ANCHOR, gauge, {0, 1, 2, 3, 4, 11, 16})) return 1;
    if (check("anchored polish by SR", FMT_ANCHOR_SR, gauge, {0, 1, 2, 3, 11})) return 1;
    if (check("fixed links, 18 reals", FMT_FIX_18, gauge, {3, 4, 8, 9, 16})) return 1;
    if (check("fixed links, 12 reals", FMT_FIX_12, gauge, {3, 4, 8, 9, 16})) return 1;
  }
  if (check("FP64", FMT_F64, GAUGE_MAG, {0, 1, 2, 3})) return 1;
  if (check("FP32-18", FMT_F32_18, GAUGE_MAG, {0, 1, 2, 3})) return 1;
  if (check("FP32-12", FMT_F32_12, GAUGE_MAG, {0, 1, 2, 3, 13, 14})) return 1;
  for (int fmt : {(int)FMT_PAIR, (int)FMT_ANCHOR, (int)FMT_ANCHOR_SR, (int)FMT_FIX_18, (int)FMT_FIX_12})
    if (check("a format without this gauge", fmt, GAUGE_MAG, {})) return 1;
  printf("ok\n");
  return 0;
}
