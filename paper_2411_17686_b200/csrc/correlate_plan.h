// How the bf16 tensor-core correlate is cut into tiles (host only, no CUDA).
//
// A CTA takes a tile of discarded tokens and one split of the preserved ones.  Tile height and number of splits are the
// pair with the least estimated time over the whole batch.  What the estimate needs of an image follows its counts
// alone, and of the two choices one decides the rows and the other the columns: images alike are looked at once, an
// image once per tile height and once per number of splits, and a pair costs it three products (search alone: 256 and
// 1000 images alike 1.5 and 3 us, all different 47 and 183; pair by pair and image by image 142 and 552).
#pragma once
#include <stddef.h>
#include <stdint.h>

#include <algorithm>
#include <vector>

namespace ficoco {

constexpr int KCAP = 16;         // longest per-token top list (targets + 1 order statistic)
constexpr int UM = 128;          // accumulator rows per MMA (one TMEM lane each)
constexpr int UN_MAX = 256;      // accumulator columns per CTA
constexpr int UKB = 64;          // bf16 elements per k-block (one 128-byte swizzle row)
constexpr int UM_STAGES = 8;     // most stages of the operand ring
constexpr int NSPLIT_MAX = 16;
constexpr int UM_TEXT_MAX = 101; // text tokens of a FiCoCo-L sequence

struct TileShape {
  int n_src, n_tgt, list_len;    // discarded tokens, preserved tokens, entries of a top list
  int count;                     // images of the batch that are like this
};

// a / b rounded up, for counts below 2^31 (the quotient's rounding error is far below 1 / b; several times as fast as an
// integer division, and a search makes up to 36 of them per image).
inline int ceil_div(int a, int b) { return (int)((double)(a + (long long)b - 1) / (double)b); }

// Columns per split: ns splits, or more if they got too wide.
inline int split_columns(int n_tgt, int ns, int cols_max, int granule) {
  ns = std::max(ns, (n_tgt - 1) / cols_max + 1);
  return (ceil_div(n_tgt, ns) + granule - 1) / granule * granule;
}
// Rows per tile: tiles of equal size, a multiple of 8.
inline int tile_height(int n_src, int rows_max) {
  return (ceil_div(n_src, ceil_div(n_src, rows_max)) + 7) / 8 * 8;
}

// Images with lists, those that are alike counted together.
inline std::vector<TileShape> distinct_shapes(const int* n_src, const int* n_tgt, const int* list_len, int batch) {
  std::vector<uint64_t> keys;
  std::vector<TileShape> out;
  keys.reserve(batch);
  for (int b = 0; b < batch; ++b)
    if (list_len[b] > 0) keys.push_back((uint64_t)n_src[b] << 40 | (uint64_t)n_tgt[b] << 8 | (uint64_t)list_len[b]);
  if (!std::is_sorted(keys.begin(), keys.end())) std::sort(keys.begin(), keys.end());
  for (size_t i = 0; i < keys.size(); ++i) {
    if (i > 0 && keys[i] == keys[i - 1]) ++out.back().count;
    else out.push_back({(int)(keys[i] >> 40), (int)(keys[i] >> 8 & 0xFFFFFFFFu), (int)(keys[i] & 255u), 1});
  }
  return out;
}

// Shared memory of a CTA.
struct UmRing {
  int nstage = 0, ksub = 1, stage_bytes = 0;
  int text_off = 0;              // where FiCoCo-L's text weights lie, behind the ring's start
  bool text_late = false;        // gathered into the ring behind the k-loop instead of beside it, ahead of the operands
  size_t smem = 0;
};

constexpr size_t UM_SMEM_ONE = 220 * 1024, UM_SMEM_TWO = 106 * 1024;    // most for a CTA alone on its SM, for two
// Entries that a thread's list of the kernel holds, for lists of at most `longest`.
inline int list_capacity(int longest) { return longest <= 2 ? 2 : longest <= 4 ? 4 : KCAP; }

// As many stages as fit, with four k-blocks per stage where that leaves four stages, else two (a stage costs about 400
// cycles besides its copies and MMAs: one FiCoCo-L sequence, 80 rows per CTA: k-loop 15 us with one, 11 with two, 9
// with four).  A grid of more CTAs than SMs keeps to what lets two share an SM, if need be by having the text weights
// take the ring's place when it is idle, behind the top lists that pass through it (whole step with one CTA per SM and with
// two: 8 sequences of 4096 + 64 tokens of 4096, a ninth kept, 483 and 396 us; 8 x 2880 + 64 307 and 262; 30 x 864 + 46,
// 523 kept, 300 and 277; 32 x 1024 + 100 320 and 297); a smaller grid has them beside the ring, ahead of the operands.
// No stages: it does not fit.
inline UmRing um_ring(int a_rows, int cols, long long n_ctas, int dim, int n_text, int list_cap, int num_sms) {
  UmRing r;
  cols = (cols + 15) / 16 * 16;
  const size_t kblock = (size_t)(a_rows + cols) * 128;
  const size_t text = (size_t)n_text * (a_rows + cols) * 4, lists = (size_t)UM * list_cap * 8;
  // every MMA reads 128 A rows: behind the last k-block there must be room for the rows past the tile
  const size_t slack = 1024 + (kblock < (size_t)UM * 128 ? (size_t)UM * 128 - kblock : 0);
  bool late = false;
  size_t limit = 0;
  auto fit = [&](int ksub, int ns) {
    const size_t ring = (size_t)ns * ksub * kblock + slack;
    const size_t smem = late ? std::max(ring, 1024 + lists + text) : std::max(ring + text, 1024 + lists);
    if (smem > limit) return;
    r.nstage = ns;
    r.ksub = ksub;
    r.stage_bytes = (int)(ksub * kblock);
    r.text_off = (int)(late ? lists : ring - 1024);
    r.text_late = late;
    r.smem = smem;
  };
  const int nk = dim / UKB;
  auto stages = [&]() {
    for (int ns = std::min(UM_STAGES, (nk + 3) / 4); ns >= 4 && !r.nstage; --ns) fit(4, ns);
    for (int ksub = 2; ksub >= 1; --ksub)
      for (int ns = std::max(2, std::min(UM_STAGES, (nk + ksub - 1) / ksub)); ns >= 2 && !r.nstage; --ns) fit(ksub, ns);
  };
  if (n_ctas > num_sms) {
    limit = UM_SMEM_TWO;
    stages();
    late = n_text > 0;
    if (late) stages();
    late = false;
  }
  limit = UM_SMEM_ONE;
  stages();
  return r;
}

struct Tiling {
  int rows = UM, splits = 1;
};

// Tile of the bf16 tensor-core correlate: rows, and column splits, by the least estimated time (ns), fitted to the
// kernel's time on eleven batches (one to 32 images of 144 to 2880 tokens of 1024, one to 16 FiCoCo-L sequences of 4096)
// under twenty tilings each: a chain of phases and k-blocks that no tiling shortens, the rows that a CTA gathers, the
// columns that its epilogue reads (with a text term per text token), a trip through L2 where a tile is split and one for
// every four entries per lane when its lists are merged.  A second CTA on the SM costs its rows again, and a grid that
// needs more than one round of two is on average half empty in the last.  Tiles below 128 rows serve small grids:
// one sequence of 576 + 64 tokens of 4096, 512 x 64 entries: 22.5 us in 16 CTAs of 128 x 16, 15 in 128 of 16 x 16;
// 32 x 288 tokens, 144 x 144 entries: 9.25 us in tiles of 72 x 80, 8.75 in 48 x 144 (no split, no counters); 32 x 576
// tokens take 13.5 us in tiles of 96 x 96 and 22 to 82 in any that make a second round.  At other widths (768, 1280, 1664;
// FiCoCo-L 2048, 3072, 5120), 42 batches of one to 64 images, whole step under up to 40 tilings each: the choice is the best
// within 0.5 % in 31 of them, within 1.6 % in all.  A grid whose CTAs have an SM each to themselves goes in rounds of one per
// SM; with 8 to 101 text tokens, 15 batches of 4 to 32 sequences under ten tilings: the best in 14, 1.5 % off in one.
inline Tiling best_tiling(const std::vector<TileShape>& shapes, int dim, int n_text, int num_sms, long long max_tiles,
                          long long max_entries) {
  constexpr int HEIGHTS[4] = {128, 64, 32, 16};
  Tiling best;
  if (shapes.empty()) return best;
  // sums over the batch, in whole numbers: CTAs, the rows and the columns that they gather, entries of the partial lists
  double ctas[4][NSPLIT_MAX] = {}, rows_all[4][NSPLIT_MAX] = {}, cols_all[4][NSPLIT_MAX] = {}, entries[NSPLIT_MAX] = {};
  int cols_most[NSPLIT_MAX], list_most[NSPLIT_MAX], rows_most[4] = {8, 8, 8, 8}, list_longest = 0;
  for (int w = 0; w < NSPLIT_MAX; ++w) { cols_most[w] = 16; list_most[w] = 0; }
  for (const TileShape& s : shapes) {
    double ns[NSPLIT_MAX], wide[NSPLIT_MAX];           // splits, and their columns together
    for (int w = 0; w < NSPLIT_MAX; ++w) {
      const int cols = split_columns(s.n_tgt, w + 1, UN_MAX, 16), k = ceil_div(s.n_tgt, cols);
      ns[w] = k;
      wide[w] = (double)k * cols;
      entries[w] += (double)s.n_src * k * s.list_len * s.count;
      cols_most[w] = std::max(cols_most[w], cols);
      list_most[w] = std::max(list_most[w], k * s.list_len);
    }
    for (int t = 0; t < 4; ++t) {
      const int height = tile_height(s.n_src, HEIGHTS[t]);
      const double tiles = (double)ceil_div(s.n_src, HEIGHTS[t]) * s.count, tall = tiles * height;
      rows_most[t] = std::max(rows_most[t], height);
      for (int w = 0; w < NSPLIT_MAX; ++w) {
        ctas[t][w] += tiles * ns[w];
        rows_all[t][w] += tall * ns[w];
        cols_all[t][w] += tiles * wide[w];
      }
    }
    list_longest = std::max(list_longest, s.list_len);
  }

  const double k_scale = dim / 1024.0, text_scale = n_text > 0 ? 1.0 + n_text / 9.5 : 1.0;
  double least = 0;
  for (int t = 0; t < 4; ++t)
    for (int w = 0; w < NSPLIT_MAX; ++w) {
      const long long n_ctas = (long long)ctas[t][w];
      const double cols = cols_all[t][w];
      if ((w > 0 || t > 0) && (n_ctas > max_tiles || entries[w] > (double)max_entries)) break;
      const UmRing ring = um_ring(rows_most[t], cols_most[w], n_ctas, dim, n_text, list_capacity(list_longest), num_sms);
      if (ring.nstage == 0) continue;
      int lanes = 1;                                   // lanes that share a token when the lists are merged
      while (lanes < 8 && rows_most[t] * 2 * lanes <= 256) lanes *= 2;
      const double rows = k_scale * (rows_all[t][w] + cols) / n_ctas;
      double cost = 2900.0 + 2270.0 * k_scale + 9.0 * rows + 10.0 * cols / n_ctas * text_scale +
                    600.0 * ((list_most[w] + 4 * lanes - 1) / (4 * lanes)) + (list_most[w] > list_longest ? 700.0 : 0.0);
      const long long wave = ring.smem > UM_SMEM_TWO ? num_sms : 2LL * num_sms;
      if (n_ctas > num_sms && wave > num_sms) cost += 26.0 * rows;
      if (n_ctas > wave) cost *= 0.5 * ((double)n_ctas / wave + (double)((n_ctas + wave - 1) / wave));
      if (least == 0 || cost < least) { least = cost; best.rows = HEIGHTS[t]; best.splits = w + 1; }
    }
  return best;
}

}  // namespace ficoco
