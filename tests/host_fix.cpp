// Host entry points to the rules, tables and arithmetic of the fixed-point FP64 passes, for
// test_fix_host.py (compiled with the host compiler).
#include "fix_tables.h"

using namespace shp;

extern "C" {
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
          const double x = std::ldexp((double)v[0] * 0x1p29 + v[1], t[o].ex[sg]);
          if (t[o].w0[sg] + k < cols) dense[((size_t)o * rows + i) * cols + t[o].w0[sg] + k] = x;
          else if (x != 0) return -1;
        }
    }
  return 1;
}
}
