// C entry to the deal of the fused filter's pieces, compiled by the host compiler for tests/test_filter_plan.py.
#include "../paper_2411_17686_b200/csrc/filter_plan.h"

extern "C" int plan_deal(const int* np, int batch, int n_ctas, long long max_pieces, int max_items, int* rc, int* cap,
                         int* max_piece) {
  const ficoco::PieceDeal d = ficoco::best_deal(np, batch, n_ctas, max_pieces, max_items);
  *rc = d.rc;
  *cap = d.cap;
  *max_piece = d.max_piece;
  return d.cost >= 0;
}
extern "C" int plan_piece_rows(int np, int rc) { return ficoco::piece_rows(np, rc); }
extern "C" int plan_ctas(const int* np, int batch, int rc, int cap, int max_items) {
  int most = 0;
  return ficoco::deal_pieces(np, batch, rc, cap, max_items, &most);
}
