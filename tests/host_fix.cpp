// Host entry points to the rules, tables and arithmetic of the fixed-point FP64 passes, for
// test_fix_host.py (compiled with the host compiler).
#include "fix_band.h"

using namespace shp;

extern "C" {
int fits(int b, int H) { return fix_band_fits(b, H); }
long long along_smem(int nops, int nline, int segs, int H) {
  return band_along_smem(nops, nline, segs, H);
}
}
