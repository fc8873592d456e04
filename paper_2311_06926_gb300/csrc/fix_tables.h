// Tables of the fixed-point FP64 passes, formed on the host at set-up (layouts: fix_band.h).
#pragma once
#include <algorithm>
#include <cmath>
#include <vector>

#include "fix_band.h"
#include "host_setup.h"

namespace shp {

// Limbs of a band: per row one scale 2^ex, at which the entries are integers of magnitude at most
// 2^58, and 2 H + 2 entries (8 if rectangular) as {hi, lo} with v = hi 2^29 + lo, |lo| <= 2^28.
// (One scale for the 8 rows of a segment is not enough: the rows beside the penalty row of T-check
// are 2^4 to 2^10 smaller, and held only that many bits fewer.) rows: {w, w, ex, 0} of row r of
// segment seg at 4 (r segs + seg); the bytes of the words w are the magnitudes, in 256ths of the
// scale (rounded down), of the entries that band_weak weighs, at their places in the window.
// Empty: the band has no such table.
struct BandLimbs {
  std::vector<int> tab, rows, w0;
};

// row i of a table of `segs` segments
inline int* band_row_of(BandLimbs& t, int segs, int i) {
  return &t.rows[((size_t)(i % kR) * segs + i / kR) * 4];
}
// the entry x of row i of scale 2^ex, entry `win` of the window, into slot `at` of the limbs and, if
// it is weighed, into the row's weights
inline void band_limb_entry(BandLimbs& t, size_t at, int* row, int H, int i, int win, double x,
                            int ex) {
  const long long v = std::llrint(std::ldexp(x, -ex));
  const int h = (int)((v + (1ll << 28)) >> 29);
  t.tab[2 * at] = h;
  t.tab[2 * at + 1] = (int)(v - ((long long)h << 29));
  const int first = band_first(H, i % kR), n = H == 0 ? 8 : (H == 1 ? 3 : 5);
  if (win < first || win >= first + n) return;
  const unsigned w = (unsigned)std::min(255.0, std::ldexp(std::fabs(x), 8 - 58 - ex));
  const int k = win - first / 4 * 4;   // byte of the row's two words
  row[k / 4] = (int)((unsigned)row[k / 4] | w << (8 * (k % 4)));
}

// the scale of row i (0: a row of zeros)
inline int band_row_scale(const Band& b, int i) {
  double mx = 0;
  for (int w = 0; w < b.width; ++w) mx = std::max(mx, std::fabs(b.val[(size_t)i * b.width + w]));
  return mx > 0 ? std::ilogb(mx) + 1 - 58 : 0;
}

// A square band, centred with half width H >= its own.
inline BandLimbs band_limbs_square(const Band& b, int H) {
  const int segs = band_segs(b.rows), per = 2 * band_row(H);
  BandLimbs t;
  t.tab.assign((size_t)segs * kR * per * 2, 0);
  t.rows.assign((size_t)segs * kR * 4, 0);
  for (int i = 0; i < b.rows; ++i) {
    const int ex = band_row_scale(b, i);
    int* row = band_row_of(t, segs, i);
    row[2] = ex;
    for (int w = 0; w < b.width; ++w) {
      const int k = b.start[i] + w - i + H;
      if (k < 0 || k > 2 * H) continue;   // (zero entries only: |k - H| > the half width)
      band_limb_entry(t, (size_t)i * per + k, row, H, i, i % kR + k,
                      b.val[(size_t)i * b.width + w], ex);
    }
  }
  return t;
}

// A pair of rectangular bands over the same inputs (a table's values and derivatives), which a pass
// with two results applies to one window: every segment's window (first input w0) holds the inputs
// of both, although exact zeros may make the bands start at different inputs. Returns false, with
// empty tables, if a segment of the pair reads more than 8 inputs.
inline bool band_limbs_rect(const Band& b0, const Band& b1, BandLimbs& t0, BandLimbs& t1) {
  const Band* b[2] = {&b0, &b1};
  BandLimbs* t[2] = {&t0, &t1};
  const int rows = b0.rows, segs = band_segs(rows), per = 2 * band_row(0);
  bool ok = b1.rows == rows && b1.cols == b0.cols;
  for (int o = 0; o < 2; ++o) {
    t[o]->tab.assign((size_t)segs * kR * per * 2, 0);
    t[o]->rows.assign((size_t)segs * kR * 4, 0);
    t[o]->w0.assign(segs, 0);
  }
  for (int sg = 0; ok && sg < segs; ++sg) {
    const int i1 = std::min(rows, kR * sg + kR);
    int lo = b0.cols, hi = 0;
    for (int i = kR * sg; i < i1; ++i)
      for (int o = 0; o < 2; ++o) {
        lo = std::min(lo, b[o]->start[i]);
        hi = std::max(hi, std::min(b[o]->start[i] + b[o]->width, b[o]->cols));
      }
    ok = hi - lo <= per;
    for (int o = 0; ok && o < 2; ++o) {
      t[o]->w0[sg] = lo;
      for (int i = kR * sg; i < i1; ++i) {
        const int ex = band_row_scale(*b[o], i);
        int* row = band_row_of(*t[o], segs, i);
        row[2] = ex;
        for (int w = 0; w < b[o]->width && b[o]->start[i] + w < b[o]->cols; ++w) {
          const int k = b[o]->start[i] + w - lo;
          band_limb_entry(*t[o], (size_t)i * per + k, row, 0, i, k,
                          b[o]->val[(size_t)i * b[o]->width + w], ex);
        }
      }
    }
  }
  if (!ok) t0 = t1 = BandLimbs{};
  return ok;
}

}  // namespace shp
