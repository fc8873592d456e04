// Host entry points to the rules, tables and arithmetic of the fixed-point FP64 passes, for
// test_fix_host.py (compiled with the host compiler).
#include <cmath>

#include "fix_tables.h"

using namespace shp;

namespace {
// One line of m entries through the passes of the library's 1D matrices: y = D0 x0 (+ D1 x1), and
// with a third matrix y2 = D2 x(last).
template <int H, int NT, bool DUAL>
void line(const BandLimbs* t, int m, const double* const* x, double* y, double* y2) {
  const int segs = band_segs(m);
  constexpr int per = kR * band_row(H);
  for (int seg = 0; seg < segs; ++seg) {
    int4 c[3 * per];
    for (int o = 0; o < NT + (DUAL ? 1 : 0); ++o)
      for (int w = 0; w < per; ++w) {
        const int* v = &t[o].tab[((size_t)seg * per + w) * 4];
        c[o * per + w] = int4{v[0], v[1], v[2], v[3]};
      }
    const unsigned redo = band_outputs<H, NT, DUAL, false>(
        c, per,
        [&](int o, int r) {
          const int* v = &t[o].rows[((size_t)r * segs + seg) * 4];
          return int4{v[0], v[1], v[2], v[3]};
        },
        [&](int k, double (&w)[kR + 2 * H]) {
          for (int j = 0; j < kR + 2 * H; ++j) {
            const int i = kR * seg + j - H;
            w[j] = i >= 0 && i < m ? x[k][i] : 0.0;
          }
        },
        [] {},
        [&](int q, int r, double v) {
          if (kR * seg + r < m) (q ? y2 : y)[kR * seg + r] = v;
        });
    for (int r = 0; r < kR && kR * seg + r < m; ++r) {   // outputs left to FMA chains
      if (redo >> (kR - 1 - r) & 1) y[kR * seg + r] = NAN;
      if (redo >> (2 * kR - 1 - r) & 1) y2[kR * seg + r] = NAN;
    }
  }
}

Dense matrix(const Univariate& u, int which) {
  return which == 0 ? u.M : (which == 1 ? u.K : (which == 2 ? u.Mc : u.Tc));
}
}  // namespace

extern "C" {
// Dense row-major copies of the bands (M, K: a x a; M-check, T-check: b x b) that the passes of n
// elements of degree p take, into val (one after the other), and the passes' results for `lines`
// lines of x0 (and x1), NaN where an output is left to an FMA chain; nterms and results as in
// line(). Returns the half width.
int band_lines(int n, int p, int nterms, int results, const int* which, double* val, int lines,
               const double* x0, const double* x1, double* y, double* y2) {
  const Univariate u = build_univariate(n, p, 14.0);
  const int nops = nterms + results - 1, H = p + 1;
  BandLimbs t[3];
  int m = 0;
  for (int o = 0; o < nops; ++o) {
    const Band b = to_band(matrix(u, which[o]), 1e-15);
    m = b.rows;
    t[o] = band_limbs_square(b, H);
    for (int i = 0; i < m; ++i)
      for (int w = 0; w < b.width; ++w)
        val[((size_t)o * m + i) * m + b.start[i] + w] = b.val[(size_t)i * b.width + w];
  }
  for (int l = 0; l < lines; ++l) {
    const double* x[2] = {x0 + (size_t)l * m, x1 ? x1 + (size_t)l * m : nullptr};
    double *r = y + (size_t)l * m, *r2 = y2 ? y2 + (size_t)l * m : nullptr;
#define LINE(h)                                                                      \
  case h:                                                                            \
    if (nterms == 1 && results == 1) line<h, 1, false>(t, m, x, r, r2);              \
    if (nterms == 1 && results == 2) line<h, 1, true>(t, m, x, r, r2);               \
    if (nterms == 2 && results == 1) line<h, 2, false>(t, m, x, r, r2);              \
    if (nterms == 2 && results == 2) line<h, 2, true>(t, m, x, r, r2);               \
    break;
    switch (H) {
      LINE(2) LINE(3) LINE(4) LINE(5) LINE(6)
      default: return -1;
    }
  }
  return H;
}

// steps between the moves of a level's sums
int level_every(int level, int xbits) { return fix_every(level, xbits); }

int fits(int b, int H) { return fix_band_fits(b, H); }
long long along_smem(int nops, int nline, int segs, int H) {
  return band_along_smem(nops, nline, segs, H);
}

// The pair of rectangular tables of bands with `width` entries a row, from inputs start[0] and
// start[1]: the segments' first inputs and entry i, j of each band as the table holds it. Returns
// whether there are tables.
int rect_pair(int rows, int cols, int width, const int* start0, const double* val0,
              const int* start1, const double* val1, int* w0, double* dense) {
  Band b[2];
  const int* start[2] = {start0, start1};
  const double* val[2] = {val0, val1};
  for (int o = 0; o < 2; ++o) {
    b[o].rows = rows;
    b[o].cols = cols;
    b[o].width = width;
    b[o].start.assign(start[o], start[o] + rows);
    b[o].val.assign(val[o], val[o] + (size_t)rows * width);
  }
  BandLimbs t[2];
  if (!band_limbs_rect(b[0], b[1], t[0], t[1])) return 0;
  for (int o = 0; o < 2; ++o)
    for (int sg = 0; sg < band_segs(rows); ++sg) {
      w0[o * band_segs(rows) + sg] = t[o].w0[sg];
      for (int i = kR * sg; i < rows && i < kR * sg + kR; ++i)
        for (int k = 0; k < 8; ++k) {
          const int* v = &t[o].tab[((size_t)i * 8 + k) * 2];
          const int ex = t[o].rows[((size_t)(i % kR) * band_segs(rows) + sg) * 4 + 2];
          const double x = std::ldexp((double)v[0] * 0x1p29 + v[1], ex);
          if (t[o].w0[sg] + k < cols) dense[((size_t)o * rows + i) * cols + t[o].w0[sg] + k] = x;
          else if (x != 0) return -1;
        }
    }
  return 1;
}
}
