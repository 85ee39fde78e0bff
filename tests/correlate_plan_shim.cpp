// C entries to the tiling of the bf16 correlate, compiled by the host compiler for tests/test_correlate_plan.py.
#include "../paper_2411_17686_b200/csrc/correlate_plan.h"

extern "C" int plan_tiling(const int* n_src, const int* n_tgt, const int* list_len, int batch, int dim, int n_text, int num_sms,
                           long long max_tiles, long long max_entries, int* rows, int* splits) {
  const auto shapes = ficoco::distinct_shapes(n_src, n_tgt, list_len, batch);
  const ficoco::Tiling t = ficoco::best_tiling(shapes, dim, n_text, num_sms, max_tiles, max_entries);
  *rows = t.rows;
  *splits = t.splits;
  return (int)shapes.size();
}
// Stages of the operand ring; out: its bytes, where the text weights lie, whether they take its place, shared memory of a CTA.
extern "C" int plan_ring(int a_rows, int cols, long long n_ctas, int dim, int n_text, int list_cap, int num_sms, long long* out) {
  const ficoco::UmRing r = ficoco::um_ring(a_rows, cols, n_ctas, dim, n_text, list_cap, num_sms);
  out[0] = (long long)r.nstage * r.stage_bytes;
  out[1] = r.text_off;
  out[2] = r.text_late;
  out[3] = (long long)r.smem;
  return r.nstage;
}
