// C entry to the layout of a plan's tables, compiled by the host compiler for tests/test_plan_tables.py.
#include "../paper_2411_17686_b200/csrc/plan_tables.h"

extern "C" void plan_layout(const size_t* n, size_t* at) {
  const ficoco::PlanTables t = ficoco::plan_tables(n[0], n[1], n[2], n[3], n[4], n[5], n[6]);
  const size_t out[6] = {t.rows, t.corr, t.out, t.cta_first, t.out_cu, t.bytes};
  for (int i = 0; i < 6; ++i) at[i] = out[i];
}
