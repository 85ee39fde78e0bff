// Where a plan's tables lie in its slot on the device and in the staging buffer (host only, no CUDA).
//
// The tables lie one behind the other, each as long as the plan needs it: what is uploaded when a shape is planned are
// the tables, not the slot, which is sized for the largest plan that the context can meet (a context for 256 images of
// 577 tokens: slots of 1.1 MB, of which a plan of these images takes a tenth).
#pragma once
#include <stddef.h>

namespace ficoco {

struct PlanTables {
  size_t rows, corr, out;        // work items (the image descriptors come first)
  size_t cta_first, out_cu;      // ints
  size_t bytes;                  // of all of them
};

inline PlanTables plan_tables(size_t desc_bytes, size_t item_bytes, size_t n_rows, size_t n_corr, size_t n_out,
                              size_t n_cta_first, size_t n_out_cu) {
  auto up = [](size_t x) { return (x + 255) / 256 * 256; };
  PlanTables t;
  t.rows = up(desc_bytes);
  t.corr = t.rows + up(n_rows * item_bytes);
  t.out = t.corr + up(n_corr * item_bytes);
  t.cta_first = t.out + up(n_out * item_bytes);
  t.out_cu = t.cta_first + up(n_cta_first * sizeof(int));
  t.bytes = t.out_cu + n_out_cu * sizeof(int);
  return t;
}

}  // namespace ficoco
