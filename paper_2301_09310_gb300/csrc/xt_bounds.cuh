// xt_bounds.cuh -- the bounds under which a pair is extended without its whole
// band (a query that nearly matches its target) or without its last rows.
//
// Notation: a = match, o = gap_open, e = gap_extend, P_k = h0 + a (k + 1).
// No cell (i, j) exceeds P_min(i,j) (every base a match, no gap), and a path
// that opens a gap and moves d diagonals away from the seed's has paid at
// least o + e d of that.  Cells on the diagonals |i - j| <= c are extended
// exactly (c = 0: base by base; c > 0: a band of 2c + 1 diagonals), giving
// lower bounds H' <= H; every path that leaves those diagonals is worth at
// most P - Q, Q = o + e (c + 1).  So, with best_i the running best of the
// near rows:
//   (1) P_min(i, qlen-1) - best_i < Q on every row i: no cell outside raises
//       the best or ties the row maximum of a row that does, so score, qle,
//       tle and max_off are the near ones;
//   (2) the near end-to-end score g > 0 and P_(qlen-1) - g < Q: gscore and
//       gtle are the near ones.  Rows from qlen on hold at most
//       P_(qlen-1) - o - e (i - qlen + 1), so once that is <= g no later row
//       changes anything;
//   (3) z-drop: a row's true maximum is at least the near one, so best_i -
//       m'_i <= zdrop excludes a stop on the rows extended.  Later rows hold
//       the deletion run from the end cell (row r, column qlen-1), and their
//       drop is at most best - g + o + e (d_best - d_end), d the diagonal
//       i - j of the best and of the end cell;
//   (4) the last live row (the cells output counts rows up to it): the
//       deletion run from the end cell reaches the last row of the band or of
//       the target; or no path can live longer: a path's last row is at most
//       qlen-1 + (Y - o - 1) / e with Y the largest H(i,j) + e (i - j), and Y
//       is at most max(best, P_(qlen-1) - o, g + e d_end) -- when the last
//       is the largest, the run itself attains the bound.
// A pair that fails any of these is extended over its whole band as before.
//
// For a band of half width c that is a good part of the query (xt_band.cu) (1)
// and (2) count what an excursion to diagonal +-(c + 1) costs in matches too.
// A path to (i, j) with I query and D target bases in gaps makes j + 1 - I =
// i + 1 - D matches at most.
//   (1') A cell of row i that an excursion reaches, outside the band or back
//        inside, is worth at most h0 + a f(i) - Q, f(i) = min(i + 1, max(qlen -
//        c - 1, min(i - c, qlen))): an insertion excursion has I > c and at
//        most min(i + 1, qlen - c - 1) matches (outside the band j > i + c; back
//        inside it pays a deletion too), a deletion excursion has D > c and at
//        most min(i - c, qlen).
//   (2') The last column: an insertion excursion loses c + 1 matches besides Q.
//        A deletion excursion that ends in row qlen - 1 + d, d <= c, inserts
//        c + 1 - d bases at least, which cost o + (a + e)(c + 1 - d); if the
//        target has rows beyond qlen - 1 + c, one that ends there costs Q alone.
#pragma once
#include <cstdint>

#include "xt_common.cuh"

namespace xt {

// What the near part of a pair found; diagonals are i - j.
struct NearEnd {
  int32_t best, d_best;  // local best and its diagonal
  int32_t g, row;        // end-to-end score and its row
};

// Conditions (3), after the rows extended, and (4): the last live row, or -1
// when it is not known.
__device__ __forceinline__ int32_t near_last_row(const NearEnd& n, int32_t qlen, int32_t tlen,
                                                 int32_t h0, int32_t match, const Score& sc) {
  const int32_t e = sc.beta, o = sc.alpha - sc.beta;
  const int32_t d_end = n.row - (qlen - 1);
  if (sc.zdrop > 0 && n.best - n.g + o + e * (n.d_best - d_end) > sc.zdrop) return -1;
  const int32_t cap = (int32_t)min((int64_t)tlen - 1, (int64_t)qlen - 1 + sc.w);
  if (cap <= n.row || e * (cap - n.row) <= n.g - o - 1) return cap;
  const int32_t y = n.g + e * d_end;
  const int32_t p = h0 + match * qlen;
  if (e == 0 || d_end < 0 || y < n.best || p - y > o) return -1;
  const int32_t k = y - o - 1 >= 0 ? (y - o - 1) / e : 0;
  return min(cap, max(n.row, qlen - 1 + k));
}

// (1') on row i with best the running best of the row or a lower one.
__device__ __forceinline__ bool near_row_ok(int32_t i, int32_t qlen, int32_t h0, int32_t match,
                                            int32_t c, int32_t best, const Score& sc) {
  const int64_t q = sc.alpha - sc.beta + (int64_t)sc.beta * (c + 1);
  const int32_t f = min(i + 1, max(qlen - c - 1, min(i - c, qlen)));
  return h0 + (int64_t)match * f - best < q;
}

// (2') for the end-to-end score g.
__device__ __forceinline__ bool near_end_ok(int32_t g, int32_t qlen, int32_t tlen, int32_t h0,
                                            int32_t match, int32_t c, const Score& sc) {
  const int64_t a = match, e = sc.beta, o = sc.alpha - e;
  const int64_t d = max(tlen - qlen, 0);
  const int64_t more = d > c ? 0 : min(a * (c + 1), o + (a + e) * (c + 1 - d));
  return h0 + a * qlen - g < o + e * (c + 1) + more;
}

}  // namespace xt
