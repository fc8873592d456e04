// The fixed-point banded passes (k_fix_band.cu): sizes that the kernels, the set-up and the rules of
// the dispatch share, and the arithmetic of a thread, which the host compiles too (for its tests).
#pragma once
#include "fix.h"

namespace shp {

constexpr int kR = 8;              // outputs per thread along the band (rows of a segment)
constexpr int kFixBandHalf = 6;    // largest half width of the limb tables
constexpr int kFixBandLimit = 227 * 1024;   // shared memory a block can have
constexpr int kFixBandThreads = 256;        // most threads of a block

// Half width H >= 1: centred square bands, row r of a segment reads entries r .. r + 2 H of the
// window (2 H + 2 stored, the last one zero). H = 0: rectangular bands (the quadrature tables: several
// points per element), whose segments read at most 8 inputs; every row has all 8.
SHP_HD constexpr int band_row(int H) { return H ? H + 1 : 4; }   // int4 per row
// int4 per segment in shared memory: one more than the rows take, so that lanes on neighbouring
// segments read different banks
SHP_HD constexpr int band_seg(int H) { return kR * band_row(H) + 1; }
SHP_HD constexpr int band_segs(int rows) { return (rows + kR - 1) / kR; }

// Staged x1 lines (shared memory): entry j, -H <= j < 8 segs + H, of a line at
// ((j + H) % 8) S + (j + H) / 8 with S odd, zero outside the line; neighbouring threads (segments)
// then read and write neighbouring words, and no window needs a bound.
SHP_HD constexpr int band_stage_s(int segs, int H) { return (segs + (2 * H + 7) / 8) | 1; }

// shared memory of a block of x1 lines: the operators' limbs, and nline staged lines
constexpr int64_t band_along_smem(int nops, int nline, int segs, int H) {
  return (int64_t)nops * segs * band_seg(H) * 16 + (int64_t)nline * kR * band_stage_s(segs, H) * 8;
}

// Whether the passes of operators of b rows fit a block. The limb tables of a whole operator are
// staged for a pass along x1, so a launch grows with the mesh; the largest has two terms and two
// results (three operators, four lines per group of segments). Longer operators keep the FMA
// passes, which stage nothing.
constexpr bool fix_band_fits(int b, int H) {
  const int segs = band_segs(b);
  return H >= 1 && H <= kFixBandHalf && segs <= kFixBandThreads &&
         band_along_smem(3, 4 * (kFixBandThreads / segs), segs, H) <= kFixBandLimit;
}

// ---- arithmetic -------------------------------------------------------------------------------
// bits of a limb and of a scaled window entry: two terms of 13 products of hi limbs, 2^29 by 2^29,
// stay below 2^63
constexpr int kBandLimb = 29, kBandXBits = 58;

SHP_HD void band_mad(long long& c, int a, int b) {
  c += (long long)a * b;
}

// Row r of a segment weighs the 5 entries around its centre (H = 1: 3; rectangular: the whole
// window). first: the first of them in the window; words of four entries, two per row, from
// first / 4 on.
SHP_HD constexpr int band_first(int H, int r) { return H ? r + (H > 2 ? H - 2 : 0) : 0; }
SHP_HD constexpr int band_words(int H) { return band_first(H, H ? kR - 1 : 0) / 4 + 2; }

// The window's exponent (the biased one of its largest entry; -1 if all are zero; slow set when it
// cannot be scaled), its entries as limbs: x / 2^(exponent - 1022) 2^58 rounded to
// hi 2^29 + lo, |lo| <= 2^28, and their magnitudes in 128ths of the scale, four to a word.
template <int N, int NW>
SHP_HD int band_limbs(const double (&x)[N], int2 (&v)[N], unsigned (&mag)[NW], bool& slow) {
  unsigned key = 0, low = 0;   // key: the largest exponent and leading bits, one place to the left
#pragma unroll
  for (int k = 0; k < N; ++k) {
    const unsigned m = hi_word(x[k]) << 1;
    key = m > key ? m : key;
    low |= lo_word(x[k]);
  }
#pragma unroll
  for (int w = 0; w < NW; ++w) mag[w] = 0;
  const int e = (int)(key >> 21);
  const bool zero = (key | low) == 0;
  slow = slow || (!zero && (e < (int)kFixMinExp || e > (int)kFixMaxExp));
  const int top = zero ? 4000 : 62 - kBandXBits + e;   // (4000: everything shifts out)
#pragma unroll
  for (int k = 0; k < N; ++k) {
    const unsigned hi = hi_word(x[k]), lo = lo_word(x[k]);
    // the significand with its leading one at bit 62 (an entry without one shifts out)
    const unsigned long long n =
        ((unsigned long long)funnel_left(lo, (hi & 0xfffffu) | 0x100000u, 10) << 32) |
        (lo << 10);
    // one bit more than kept, then rounded (truncated entries would all err towards zero, and that
    // smooth error is what the preconditioner amplifies), the low limb of either sign
    const int sh0 = top - (int)((hi >> 20) & 0x7ffu), sh = sh0 < 63 ? sh0 : 63;
    const unsigned long long t = (n >> sh) + (1ull << kBandLimb) + 1;
    const int h = (int)(t >> (kBandLimb + 1));
    const int l = (int)((unsigned)(t >> 1) - (1u << (kBandLimb - 1)) - ((unsigned)h << kBandLimb));
    if (k < 4 * NW) mag[k / 4] |= (unsigned)(h >> (kBandXBits - kBandLimb - 7)) << (8 * (k % 4));
    const int sg = (int)hi >> 31;
    v[k].x = (h ^ sg) - sg;
    v[k].y = (l ^ sg) - sg;
  }
  return zero ? -1 : e;
}

// sum of the products of the bytes of a and b, plus c
SHP_HD unsigned dot_bytes(unsigned a, unsigned b, unsigned c) {
#ifdef __CUDA_ARCH__
  return __dp4a(a, b, c);
#else
  for (int k = 0; k < 32; k += 8) c += (a >> k & 255u) * (b >> k & 255u);
  return c;
#endif
}

// Rows whose own entries are too small for the scales of the window and the row (weak rows), bit
// 7 - r: the sum of the products of the weighed magnitudes (rounded down: a lower bound of
// sum |D| |x|) is below 2^-6 of the product of the scales. Above that line the roundings at the
// common scale, about 2^-59 of it, stay below those of an FMA chain over the row: host emulation,
// p = 1 .. 4, lines that are normal, spiked or geometric (factors 4 and 10): rms 0.26 to 0.46 units of
// 2^-53 sum |D| |x|, at most 2.2, against 0.42 to 0.85 and 5.6. (At 2^-7 0.58 and 4.1.) Weighing all
// rows before the products costs about 10% of a launch; within their loop its registers spilled.
constexpr unsigned kBandWeak = 1u << (7 + 8 - 6);
template <int H, int NW, typename Row>
SHP_HD unsigned band_weak(const unsigned (&mag)[NW], Row&& row, int o) {
  unsigned weak = 0;
#pragma unroll
  for (int r = 0; r < kR; ++r) {
    const int4 w = row(o, r);
    const int m = band_first(H, r) / 4;
    const unsigned s = dot_bytes(mag[m], (unsigned)w.x, 0u - kBandWeak);
    weak = funnel_left(dot_bytes(mag[m + 1], (unsigned)w.y, s), weak, 1);   // (its sign bit)
  }
  return weak;
}

// Row r of the segment times the window, in units of 2^58 of the product of the two scales, plus hh.
template <int H, int N>
SHP_HD long long band_row_dot(const int4* c, const int2 (&v)[N], int r, long long hh = 0) {
  long long md = 1ll << (kBandLimb - 1);
  const int k0 = H ? r : 0;
#pragma unroll
  for (int q = 0; q < band_row(H); ++q) {
    const int4 w = c[r * band_row(H) + q];
    const int2 a = v[k0 + 2 * q];
    band_mad(hh, a.x, w.x);
    band_mad(md, a.x, w.y);
    band_mad(md, a.y, w.x);
    if (H == 0 || q < H) {   // (entry 2 H + 1 is padding)
      const int2 b = v[k0 + 2 * q + 1];
      band_mad(hh, b.x, w.z);
      band_mad(md, b.x, w.w);
      band_mad(md, b.y, w.z);
    }
  }
  return hh + (md >> kBandLimb);
}

// Scale of a window of zeros (below every other) and from scales to the exponent of a result.
constexpr int kNoScale = -(1 << 20);
constexpr int kBandShift = 2 * kBandLimb - 1022 - kBandXBits;

// The outputs 8 seg .. 8 seg + 7 of one line. load(t, x): the window of term t; c: the operators'
// limbs of the segment, cstep int4 apart; row(o, r): weights and scale of row r of operator o
// (BandLimbs); put(y, r, value): output r of Y (y = 0) or Y2 (1). Returns the outputs that are left
// to FMA chains, bit 7 - r (Y) and 15 - r (Y2): all if a window cannot be scaled, else those of weak
// rows (of either term). ONCE: these are not put before; else they may be, and are put again.
// ready(): called once the first window is scaled, before the limbs and scales are read.
template <int H, int NT, bool DUAL, bool ONCE, typename Row, typename Load, typename Ready,
          typename Put>
SHP_HD unsigned band_outputs(const int4* c, int cstep, Row&& row, Load&& load, Ready&& ready,
                             Put&& put) {
  constexpr int N = kR + 2 * H, NW = band_words(H);
  bool slow = false;
  int2 v[N];
  long long s[kR];   // NT = 2: the first term's sums
  int e0 = 0, e = 0;
  unsigned weak = 0, weak2 = 0;
#pragma unroll
  for (int t = 0; t < NT; ++t) {
    double x[N];
    unsigned mag[NW];
    load(t, x);
    e = band_limbs<N, NW>(x, v, mag, slow);
    if (t == 0) ready();
    if (e >= 0) {   // (a window of zeros is exact at any scale)
      weak |= band_weak<H, NW>(mag, row, t);
      if (DUAL && t + 1 == NT) weak2 = band_weak<H, NW>(mag, row, NT);
    }
    if (t + 1 < NT) {
      e0 = e;
#pragma unroll
      for (int r = 0; r < kR; ++r) s[r] = band_row_dot<H, N>(c, v, r);
      c += cstep;
      continue;
    }
    if (slow) return DUAL ? 0xffffu : 0xffu;
#pragma unroll
    for (int r = 0; r < kR; ++r) {
      int top = e < 0 ? kNoScale : e + row(t, r).z;
      long long y;
      if (NT > 1) {
        // both sums at the larger of the two scales, half a unit added to one that is shifted
        const int en = top, es = e0 < 0 ? kNoScale : e0 + row(0, r).z;
        top = es > en ? es : en;
        const int da = top - es < 62 ? top - es : 62, db = top - en < 62 ? top - en : 62;
        y = band_row_dot<H, N>(c, v, r, (1ll << db) >> 1);
        y = ((s[r] + ((1ll << da) >> 1)) >> da) + (y >> db);
      } else {
        y = band_row_dot<H, N>(c, v, r);
      }
      if (!ONCE || !(weak >> (kR - 1 - r) & 1u)) put(0, r, fix_to_double(y, top + kBandShift));
      if (DUAL)
        put(1, r, fix_to_double(band_row_dot<H, N>(c + cstep, v, r),
                                (e < 0 ? kNoScale : e + row(NT, r).z) + kBandShift));
    }
  }
  return weak | weak2 << kR;
}

}  // namespace shp
