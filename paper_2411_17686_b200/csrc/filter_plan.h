// How the fused filter kernel's work is dealt out (host only, no CUDA).
//
// The patch rows of every image are cut into pieces of equal size, at most `rc` rows each, and the pieces are dealt
// to the CTAs in order, so that no CTA gets more than `cap` rows or `max_items` pieces.  The kernel's time follows
// the fullest CTA, and every piece adds a fold, a hand-over and, with an image of its own, a selection
// (F_PIECE_ROWS rows' worth): of the sizes tried the one with the least of both is taken.
#pragma once
#include <algorithm>

namespace ficoco {

constexpr int F_PIECE_ROWS = 128;    // rows that a piece costs besides its own

// Rows per piece of an image of np rows, in pieces of about equal size: a multiple of 8, so up to 7 more than rc.  (The
// last piece of the image may be smaller.)
inline int piece_rows(int np, int rc) {
  const int n = (np + rc - 1) / rc;
  return ((np + n - 1) / n + 7) / 8 * 8;
}

// CTAs that a deal with at most `cap` rows and `max_items` pieces per CTA takes; *most: pieces of the fullest CTA.
inline int deal_pieces(const int* np, int batch, int rc, int cap, int max_items, int* most) {
  int n_cta = 1, acc = 0, items = 0;
  *most = 0;
  for (int b = 0; b < batch; ++b) {
    const int step = np[b] > 0 ? piece_rows(np[b], rc) : 1;
    for (int r = 0; r < np[b]; r += step) {
      const int n = std::min(step, np[b] - r);
      if (items > 0 && (acc + n > cap || items >= max_items)) { ++n_cta; acc = items = 0; }
      acc += n;
      ++items;
      if (items > *most) *most = items;
    }
  }
  return n_cta;
}

struct PieceDeal {
  int rc = 0;            // piece_rows(np, rc) rows per piece
  int max_piece = 0;     // rows of the largest piece: the kernel's shared memory is sized by it
  int cap = 0;           // most rows of a CTA
  int even = 0;          // rows per CTA of a perfectly even deal
  long long cost = -1;   // rows of the fullest CTA + F_PIECE_ROWS per piece of the CTA with the most pieces; -1: no deal
};

// Best deal of `batch` images to at most `n_ctas` CTAs with at most max_pieces pieces in all.
inline PieceDeal best_deal(const int* np, int batch, int n_ctas, long long max_pieces, int max_items) {
  PieceDeal best;
  long long total = 0;
  int np_max = 0;
  for (int b = 0; b < batch; ++b) { total += np[b]; np_max = std::max(np_max, np[b]); }
  best.even = (int)((total + n_ctas - 1) / n_ctas);
  const int rc_lo = std::max(32, best.even / 4 / 8 * 8);
  const int rc_hi = std::max(rc_lo, std::min(2 * best.even + 8, (np_max + 7) / 8 * 8));
  const int rc_step = std::max(8, (rc_hi - rc_lo) / 24 / 8 * 8);
  for (int rc = rc_hi; rc >= rc_lo; rc -= rc_step) {
    long long n_pieces = 0;
    int biggest = 0, np_last = 0, step = 1, n = 0;
    for (int b = 0; b < batch; ++b) {
      if (np[b] <= 0) continue;
      if (np[b] != np_last) { np_last = np[b]; step = piece_rows(np[b], rc); n = (np[b] + step - 1) / step; }
      n_pieces += n;
      biggest = std::max(biggest, std::min(step, np[b]));
    }
    int lo = std::max(best.even, biggest), hi = 2 * lo, most = 0;
    if (n_pieces > max_pieces) break;
    if (n_pieces <= n_ctas) { hi = lo = biggest; }              // one piece each
    else {
      // (no deal can do better than this: most sizes are ruled out without one)
      if (best.cost >= 0 && lo + (n_pieces + n_ctas - 1) / n_ctas * F_PIECE_ROWS >= best.cost) continue;
      if (deal_pieces(np, batch, rc, hi, max_items, &most) > n_ctas) continue;
      while (lo < hi) {
        const int mid = (lo + hi) / 2;
        if (deal_pieces(np, batch, rc, mid, max_items, &most) <= n_ctas) hi = mid; else lo = mid + 1;
      }
    }
    deal_pieces(np, batch, rc, hi, max_items, &most);
    const long long cost = hi + (long long)most * F_PIECE_ROWS;
    if (best.cost < 0 || cost < best.cost) { best.cost = cost; best.rc = rc; best.cap = hi; best.max_piece = biggest; }
  }
  return best;
}

}  // namespace ficoco
