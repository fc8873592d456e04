// Fixed-point evaluation of FP64 dot products on the FP16 tensor cores.
//
// GB300 runs 2 FP64 FMAs per clock and SM, but 1024 FP16 multiply-adds with FP32 sums (mma.sync;
// measured: 0.62 against 300 T per second). A dot product of doubles is therefore cheaper in
// slices: the entries of one input line are scaled by one power of two (that of the line's largest
// entry) to integers, those of an operator column to integers below 2^58, and each integer is
// written in six balanced digits of ten bits, sum_i d_i 2^(50 - 10 i), |d_i| <= 512, which FP16
// holds exactly. Products of digits are exact in the tensor cores, and the 21 digit pairs with
// i + j <= 5 are summed by level l = i + j in FP32, which holds integers up to 2^24. The levels are
// moved to integers before they can pass that, whatever the digits (fix_every, fix_peak): 3 after
// every step of 16 terms, 2 after two, 0 and 1 after five (input integers below 2^57: folded entries
// and modes) or four (below 2^58: plain matrices). Lines and columns of equal entries do reach the
// bounds: level 3 over 66 equal terms passed 2^24 for one pair of values in twenty when it was moved
// every five steps, and truncated sums cost 2^-48 of the result. Level 4, in units of the result,
// may reach 2^25 over its two steps and lose its last bit; level 5 stays until the end and loses
// less than 2^-4 of a unit. (The moves cost 1% of P_0^-1 at 128^3: 906 -> 915 us; with 64-bit sums
// in place of the moved integers 974 to 994.) The integer result is rounded to a double once, where
// an FMA chain rounds at every term. The dropped pairs (i + j >= 6) and the scaling leave an error
// below that of the FMA chain (host emulation, 9 to 66 terms, rms over random, decaying and smooth
// lines: 0.2 to 0.56 of the chain's). Splitting products into slices that the matrix unit sums
// exactly follows Ozaki, Ogita, Oishi and Rump, "Error-free transformations of matrix
// multiplication by using fast routines of matrix multiplication", 2012.
//
// The integer sums do not depend on the tile or the kernel that forms them, so every launch form
// gives the same bits.
//
// A line with an infinity or a NaN, or whose largest entry is outside [2^-823, 2^777] (its scaled
// result could leave the normal range), takes the FMA chain instead.
#pragma once
#include <cuda_runtime.h>

#include <cstdint>
#include <cstring>

#ifdef __CUDACC__
#define SHP_HD __host__ __device__ __forceinline__
#else
#define SHP_HD inline
#endif

namespace shp {

constexpr int kFixSlices = 6, kFixDigit = 10;
// bits of a scaled operator entry, and of the sum of an output's operator magnitudes: the 64-bit
// sums, in units of 2^60, stay below 2^62
constexpr int kFixUBits = 58, kFixSumBits = 63, kFixUnit = 60;

// Steps of 16 terms after which level l's sums are moved, for input integers below 2^xbits, and the
// largest sum they can reach by then (leading digits are smaller than the others).
SHP_HD constexpr int fix_drain(int xbits) { return xbits == 58 ? 4 : 5; }
SHP_HD constexpr int fix_every(int l, int xbits) {
  return l == 2 || l == 4 ? 2 : (l == 3 ? 1 : fix_drain(xbits));
}
constexpr int64_t fix_digit_max(int i, int bits) {
  return 1ll << (i ? kFixDigit - 1 : bits - kFixDigit * (kFixSlices - 1));
}
constexpr int64_t fix_peak(int l, int xbits) {
  int64_t sum = 0;
  for (int i = 0; i <= l; ++i) sum += fix_digit_max(i, xbits) * fix_digit_max(l - i, kFixUBits);
  return 16 * fix_every(l, xbits) * sum;
}
constexpr bool fix_exact(int xbits) {
  for (int l = 0; l < 4; ++l)
    if (fix_peak(l, xbits) > 1 << 24) return false;
  return fix_peak(4, xbits) <= 1 << 25;
}
static_assert(fix_exact(56) && fix_exact(57) && fix_exact(58), "level sums must stay exact");

// One direction of a parity-split operator (host_setup.h, generalized_eigh_parity) as digit slices
// in the operand order of mma.sync m16n8k16: half `par` (0: even terms, 1: odd terms), 8 outputs
// per column tile t < nt, 16 terms per step s < ks, the half zero-padded (a plain matrix has half 0
// only):
//   frag[(((par nt + t) ks + s) 3 + c) 32 + lane] = the lane's two registers of slice 2 c, then
//   those of slice 2 c + 1.
// Output i of half par is the integer sum times 2^ex[par 8 nt + i].
struct FixTab {
  const uint4* frag = nullptr;
  const int* ex = nullptr;
  int nt = 0, ks = 0;
};

// The uses of an operator U (columns [even modes; odd modes]): fw contracts the folded entries of a
// line with the columns (outputs: modes), bw the modes with the rows (outputs: the even and the
// odd part of the mirrored entries k and n - 1 - k). A plain matrix has one table, fw, of one half
// with every entry as a term.
enum { kFixForward = 0, kFixBackward = 1, kFixPlain = 2 };
struct FixTabs {
  FixTab fw, bw;
};

// biased exponents of the largest entry of a line that the fixed-point form takes
constexpr unsigned kFixMinExp = 200, kFixMaxExp = 1800;

// The words of a double, and a funnel shift (the arithmetic below also compiles for the host, where
// its tests run it).
SHP_HD unsigned hi_word(double x) {
#ifdef __CUDA_ARCH__
  return (unsigned)__double2hiint(x);
#else
  uint64_t u;
  std::memcpy(&u, &x, sizeof u);
  return (unsigned)(u >> 32);
#endif
}
SHP_HD unsigned lo_word(double x) {
#ifdef __CUDA_ARCH__
  return (unsigned)__double2loint(x);
#else
  uint64_t u;
  std::memcpy(&u, &x, sizeof u);
  return (unsigned)u;
#endif
}
SHP_HD double from_words(unsigned hi, unsigned lo) {
#ifdef __CUDA_ARCH__
  return __hiloint2double((int)hi, (int)lo);
#else
  const uint64_t u = (uint64_t)hi << 32 | lo;
  double x;
  std::memcpy(&x, &u, sizeof x);
  return x;
#endif
}
SHP_HD unsigned funnel_left(unsigned lo, unsigned hi, int n) {   // 0 < n < 32
#ifdef __CUDA_ARCH__
  return __funnelshift_l(lo, hi, n);
#else
  return hi << n | lo >> (32 - n);
#endif
}

// Magnitude key of an entry: its exponent field and leading bits (the low word only marks a
// nonzero). The largest key of a line gives its scale; 0 only for a line of zeros.
SHP_HD unsigned fix_key(double x) {
  return (hi_word(x) & 0x7fffffffu) | (lo_word(x) != 0 ? 1u : 0u);
}
SHP_HD bool fix_slow(unsigned key) {
  const unsigned e = key >> 20;
  return key != 0u && (e < kFixMinExp || e > kFixMaxExp);
}
// x / 2^(emax - 1022) * 2^xbits, rounded (emax: exponent field of the largest entry)
SHP_HD long long fix_of(double x, int emax, int xbits) {
  const unsigned hi = hi_word(x), lo = lo_word(x);
  const int e = (int)((hi >> 20) & 0x7ffu);
  const unsigned m = (hi & 0xfffffu) | (e ? 0x100000u : 0u);
  // the 53-bit significand with its leading bit at bit 62
  const unsigned long long n = ((unsigned long long)funnel_left(lo, m, 10) << 32) | (lo << 10);
  const int t = 62 - xbits + emax - e, sh = t < 63 ? t : 63;
  const long long v = (long long)(((n >> sh) + 1) >> 1);
  return (int)hi < 0 ? -v : v;
}
// s * 2^ex as a double (ex keeps it in the normal range). By the conversion instruction, on the FP64
// pipe that these kernels leave idle (in about 20 integer instructions instead: 128^3 K apply 526
// against 501 us, P_0^-1 914 against 901).
SHP_HD double fix_to_double(long long s, int ex) {
  const double d = (double)s;
  return s == 0 ? 0.0 : from_words(hi_word(d) + (unsigned)ex * (1u << 20), lo_word(d));
}

}  // namespace shp
