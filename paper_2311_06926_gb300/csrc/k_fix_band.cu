// FP64 banded Kronecker passes in fixed point on the integer multipliers.
//
// GB300 runs 64 32 x 32 + 64-bit integer multiply-adds per clock and SM against 2 FP64 FMAs
// (measured: 18.4 against 0.62 T per second). A thread forms 8 consecutive outputs of one line from
// the window of 8 + 2 H inputs they read. It scales the window by one power of two (that of its
// largest entry) to integers below 2^58 and splits each into two limbs of 29 bits; the operator's
// entries are kept as two limbs of integers below 2^58, one scale per row. A product of two
// such pairs takes three multiply-adds, xh ch and xh cl + xl ch, into two 64-bit sums that cannot
// overflow (13 terms); xl cl, below 2^-58 of the largest product, is dropped. The sum is rounded
// to a double once, where an FMA chain rounds at every term.
//
// The scale is that of a window's largest entry, which not every row of the segment reads, and the
// row's scale that of its largest coefficient, which may meet a small entry. So every output is
// weighed: where its own sum |D| |x| is too far below the product of the scales (band_weak), its
// thread forms it by an FMA chain as well and stores that. Every output is as close as a chain
// then: its error is relative to its own terms, not to the window (1e-4 to 1.6e-3 of the outputs are
// left to chains for lines of normal entries).
//
// Bound by instruction issue: about 140 instructions per result, of which the 27 multiply-adds of a
// row of 9 take twice their slots. Measured against the FMA passes: K apply 1052 -> 613 us at 128^3
// p = 3 (533 without weighing and chains), 61^3 p = 2 81, 48^3 p = 3 65 (66 and 50 without).
//
// A window with an infinity or a NaN, or outside [2^-823, 2^777], takes FMA chains instead.
#include <algorithm>
#include <atomic>

#include "fix_band.h"
#include "internal.h"
#include "profile.h"

namespace shp {
namespace {

struct FixBandOp {
  const int4* tab;   // [segment][8 rows][band_row]: {hi, lo, hi, lo} of entries 2 q, 2 q + 1
  const int4* rows;  // weights and scale of row r of segment seg at r segs + seg
  const int* w0;     // rectangular bands (H = 0): first input of each segment's window
  // the band in doubles (outputs left to FMA chains): row i's `width` entries at val + i pitch, from
  // input start[i] or, start null, i - half
  const double* val;
  const int* start;
  int width, pitch, half;
};

struct FixBandJob {
  const double* X[2];
  FixBandOp D[3];    // terms 0 .. nterms - 1 of Y, then the operator of Y2
  double* Y;
  double* Y2;        // = D[nterms] X[nterms - 1], or null
  const double* g;
  int gaxis;
  int gd1, gd12;     // strides of g along x2 and x3
  int hmode;
  double *hr, *hacc;
  const double* hx;
  Dims in;
  int rows;          // outputs of a line (the extent of Y along the axis)
  unsigned n1_mul;   // line / n1 = umulhi(line, n1_mul) >> n1_sh for line < 2^31
  int n1_sh;
  int axis, nterms, nops, nb, segs;
  int64_t bs;
};
struct FixBandBatch {
  FixBandJob job[kMaxPassJobs];
  int first[kMaxPassJobs + 1];
  int njobs;
};

// position of entry j - H of a staged line (fix_band.h)
__device__ __forceinline__ int band_stage(int j, int S) { return (j & 7) * S + (j >> 3); }

// Outputs left to FMA chains (band_outputs): at(t, j): entry j of term t's line of nin entries. Few
// threads come here; what they cost is latency, so nothing is looked up before the operands.
template <typename At, typename Put>
__device__ __forceinline__ void band_chains(const FixBandJob& J, int seg, int m, int nin,
                                            unsigned redo, At&& at, Put&& put) {
  const int rows = min(m - kR * seg, kR);
  redo &= (0xff00u >> rows & 0xffu) * 0x101u;
  while (redo) {
    const int bit = __ffs(redo) - 1, r = kR - 1 - bit % kR, i = kR * seg + r;
    redo &= redo - 1;
    const int o0 = bit < kR ? 0 : J.nterms, o1 = bit < kR ? J.nterms : J.nops;
    double y = 0.0;
#pragma unroll 1
    for (int o = o0; o < o1; ++o) {
      const FixBandOp& D = J.D[o];
      const int t = min(o, J.nterms - 1);
      const int j0 = D.start ? D.start[i] : i - D.half;   // input of the row's first entry
      const int k0 = max(0, -j0), k1 = min(D.width, nin - j0);
      const double* d = D.val + (int64_t)i * D.pitch;
#pragma unroll 4
      for (int k = k0; k < k1; ++k) y = fma(d[k], at(t, j0 + k), y);
    }
    put(bit / kR, r, y);
  }
}

// The segment of a thread of a pass along x2 or x3 (block `local` of the job).
struct BandPlace {
  int64_t first, at0;   // entry 0 of the line and output 0 of the segment
  int64_t kb;           // offset of the line's item
  int i1, q;            // x1 index, and x3 (axis 2) or x2 index
  int stride, i0, m, rows;   // rows: of the segment to write
};
__device__ __forceinline__ BandPlace band_place(const FixBandJob& J, int local) {
  BandPlace p;
  const int lb = local / J.segs, seg = local - lb * J.segs;
  const int n1 = J.in.n1, n12 = n1 * J.in.n2;
  const bool ax2 = J.axis == 2;
  const int lines1 = ax2 ? n1 * J.in.n3 : n12;
  int line = lb * (int)blockDim.x + (int)threadIdx.x;
  const bool on = line < lines1 * J.nb;
  if (!on) line = 0;
  p.kb = 0;
  if (J.nb > 1) {
    const int k = line / lines1;
    p.kb = (int64_t)k * J.bs;
    line -= k * lines1;
  }
  p.q = n1 == 1 ? line : (int)(__umulhi((unsigned)line, J.n1_mul) >> J.n1_sh);
  p.i1 = line - p.q * n1;
  p.first = p.kb + (ax2 ? p.i1 + (int64_t)n12 * p.q : (int64_t)line);
  p.stride = ax2 ? n1 : n12;
  p.i0 = kR * seg;
  p.m = J.rows;
  p.rows = on ? p.m - p.i0 : 0;
  // (a rectangular pass along x2 has result planes of another size)
  p.at0 = (ax2 ? p.kb + p.i1 + (int64_t)n1 * p.m * p.q : p.first) + (int64_t)p.stride * p.i0;
  return p;
}

// Stores output r of the segment: a result, or with EPI what the job makes of it.
template <bool EPI>
__device__ __forceinline__ void band_put(const FixBandJob& J, const BandPlace& p, int y, int r,
                                         double v) {
  if (r >= p.rows) return;
  const int64_t o = p.at0 + (int64_t)p.stride * r;
  if (EPI) {
    if (J.g) {
      const bool ax2 = J.axis == 2;
      const int gstride = ax2 ? J.gd1 : J.gd12;
      const int gstep = J.gaxis == 1 ? 1 : (J.gaxis == 2 ? J.gd1 : J.gd12);
      const double* g = J.g + p.kb + p.i1 + (int64_t)(ax2 ? J.gd12 : J.gd1) * p.q +
                        (int64_t)gstride * (p.i0 + r);
      v += g[0] - g[gstep];
    }
    if (J.hmode == 1) {
      const double xi = J.hx[o], ri = xi - v;
      J.hr[o] = ri;
      J.hacc[o] = xi + ri;
      return;
    }
    if (J.hmode == 2) {
      const double ri = J.hr[o] - v;
      J.hr[o] = ri;
      J.hacc[o] += ri;
      return;
    }
  }
  (y ? J.Y2 : J.Y)[o] = v;
}

// A pass along x2 or x3: the block takes one segment of blockDim neighbouring lines, so every load
// and store is coalesced and the operators' limbs are read as broadcasts.
template <int H, int NT, bool DUAL, bool EPI>
__device__ __forceinline__ void band_across(const FixBandJob& J, int local, int4* sh) {
  constexpr int N = kR + 2 * H, kSegIn = kR * band_row(H), kOps = NT + (DUAL ? 1 : 0);
  const int tid = threadIdx.x, nth = blockDim.x;
  const int lb = local / J.segs, seg = local - lb * J.segs;
  int4* rw = sh + kOps * kSegIn;   // [kOps][8]
  // (the operators are written once at setup: their copy does not wait for the preceding kernel)
#pragma unroll
  for (int o = 0; o < kOps; ++o) {
    for (int w = tid; w < kSegIn; w += nth)
      sh[o * kSegIn + w] = __ldg(J.D[o].tab + (int64_t)seg * kSegIn + w);
    if (tid < kR) rw[kR * o + tid] = __ldg(J.D[o].rows + tid * J.segs + seg);
  }
  pdl_begin();
  const BandPlace p = band_place(J, local);
  const int64_t stride = p.stride;
  auto put = [&](int y, int r, double v) { band_put<EPI>(J, p, y, r, v); };
  const unsigned redo = band_outputs<H, NT, DUAL, EPI>(
      sh, kSegIn, [&](int o, int r) { return rw[kR * o + r]; },
      [&](int t, double (&x)[N]) {
        if constexpr (H == 0) {
          const int w0 = __ldg(J.D[t].w0 + seg), nin = J.axis == 2 ? J.in.n2 : J.in.n3;
          const double* x0 = J.X[t] + p.first + stride * w0;
#pragma unroll
          for (int k = 0; k < N; ++k) x[k] = w0 + k < nin ? x0[stride * k] : 0.0;
          return;
        }
        const double* x0 = J.X[t] + p.at0;
        if (p.i0 >= H && p.i0 + kR + H <= p.m) {
#pragma unroll
          for (int k = 0; k < N; ++k) x[k] = x0[stride * (k - H)];
        } else {
#pragma unroll
          for (int k = 0; k < N; ++k)
            x[k] = p.i0 + k >= H && p.i0 + k < p.m + H ? x0[stride * (k - H)] : 0.0;
        }
      },
      [] { __syncthreads(); }, put);
  if (redo && p.rows > 0)
    band_chains(J, seg, p.m, J.axis == 2 ? J.in.n2 : J.in.n3, redo,
                [&](int t, int j) { return J.X[t][p.first + stride * j]; }, put);
}

// zeros around the m entries of nl staged lines
template <int H>
__device__ __forceinline__ void band_stage_zero(double* raw, int nl, int m, int segs, int S) {
  const int per = kR * segs - m + 2 * H;
  for (int idx = threadIdx.x; idx < nl * per; idx += blockDim.x) {
    const int l = idx / per, k = idx - l * per;
    raw[l * kR * S + band_stage(k < H ? k : m + k, S)] = 0.0;
  }
}

// the limbs of all segments of one operator (pitch band_seg)
template <int H>
__device__ __forceinline__ void band_stage_op(const FixBandOp& D, int segs, int4* sh) {
  constexpr int kSegIn = kR * band_row(H);
  for (int idx = threadIdx.x; idx < segs * kSegIn; idx += blockDim.x) {
    const int sg = idx / kSegIn;
    sh[sg * band_seg(H) + idx - sg * kSegIn] = __ldg(D.tab + idx);
  }
}

// A pass along x1: the block takes whole lines, staged in shared memory with their results, one
// thread per segment.
template <int H, int NT, bool DUAL>
__device__ __forceinline__ void band_along(const FixBandJob& J, int local, int4* sh) {
  constexpr int N = kR + 2 * H, kOps = NT + (DUAL ? 1 : 0);
  const int tid = threadIdx.x, nth = blockDim.x;
  const int segs = J.segs, m = J.in.n1, lines1 = J.in.n2 * J.in.n3;
  const int lpb = nth / segs, line0 = local * lpb, nl = min(lpb, lines1 * J.nb - line0);
  const int S = band_stage_s(segs, H);
  double* raw = reinterpret_cast<double*>(sh + kOps * segs * band_seg(H));   // [NT][lpb][8 S]
  double* out = raw + NT * lpb * kR * S;                                    // [1 or 2][lpb][8 S]
#pragma unroll
  for (int o = 0; o < kOps; ++o)
    band_stage_op<H>(J.D[o], segs, sh + o * segs * band_seg(H));
#pragma unroll
  for (int t = 0; t < NT; ++t) band_stage_zero<H>(raw + t * lpb * kR * S, nl, m, segs, S);
  auto line_of = [&](int idx) -> int {   // idx / m
    return m == 1 ? idx : (int)(__umulhi((unsigned)idx, J.n1_mul) >> J.n1_sh);
  };
  auto first_of = [&](int line) -> int64_t {
    int64_t kb = 0;
    if (J.nb > 1) {
      const int k = line / lines1;
      kb = (int64_t)k * J.bs;
      line -= k * lines1;
    }
    return kb + (int64_t)m * line;
  };
  pdl_begin();
#pragma unroll 2
  for (int idx = tid; idx < nl * m; idx += nth) {
    const int l = line_of(idx), j = idx - l * m;
    const int64_t o = first_of(line0 + l) + j;
#pragma unroll
    for (int t = 0; t < NT; ++t)
      raw[(t * lpb + l) * kR * S + band_stage(j + H, S)] = J.X[t][o];
  }
  __syncthreads();
  const int l = tid / segs, seg = tid - l * segs;
  if (l < nl) {
    const double* p = raw + l * kR * S + seg;
    double* q = out + l * kR * S + seg;
    auto put = [&](int y, int r, double v) { q[(y ? lpb * kR * S : 0) + r * S] = v; };
    const unsigned redo = band_outputs<H, NT, DUAL, false>(
        sh + seg * band_seg(H), segs * band_seg(H),
        [&](int o, int r) { return __ldg(J.D[o].rows + r * segs + seg); },
        [&](int t, double (&x)[N]) {
#pragma unroll
          for (int k = 0; k < N; ++k) x[k] = p[t * lpb * kR * S + (k & 7) * S + (k >> 3)];
        },
        [] {}, put);
    if (redo)
      band_chains(J, seg, m, m, redo,
                  [&](int t, int j) { return raw[(t * lpb + l) * kR * S + band_stage(j + H, S)]; },
                  put);
  }
  __syncthreads();
  for (int idx = tid; idx < nl * m; idx += nth) {
    const int w = line_of(idx), j = idx - w * m;
    const int64_t o = first_of(line0 + w) + j;
    const int at = w * kR * S + band_stage(j, S);
    J.Y[o] = out[at];
    if (DUAL) J.Y2[o] = out[lpb * kR * S + at];
  }
}

// NT: the most terms of a job (fewer registers where every job has one). EPI: jobs may have a g
// term or a Horner step (passes along x2 and x3 with one result; a kernel of their own because the
// compiler executes their FP64 additions whether taken or not).
template <int H, int NT, bool EPI>
__global__ void __launch_bounds__(256, 3)
    k_fix_band(const __grid_constant__ FixBandBatch fb) {
  extern __shared__ __align__(16) int4 shb[];
  int jb = 0;
  while (jb + 1 < fb.njobs && (int)blockIdx.x >= fb.first[jb + 1]) ++jb;
  const FixBandJob& J = fb.job[jb];
  const int local = (int)blockIdx.x - fb.first[jb];
  if constexpr (H == 0) {
    if (J.Y2) band_across<H, 1, true, false>(J, local, shb);
    else band_across<H, 1, false, false>(J, local, shb);
    return;
  } else if constexpr (NT == 2) {
    if (J.nterms == 2) {
      if constexpr (EPI) {
        band_across<H, 2, false, true>(J, local, shb);
      } else {
        if (!J.Y2) band_across<H, 2, false, false>(J, local, shb);
        else if (J.axis == 1) band_along<H, 2, true>(J, local, shb);
        else band_across<H, 2, true, false>(J, local, shb);
      }
      return;
    }
  }
  if constexpr (H == 0) {
  } else if constexpr (EPI) {
    band_across<H, 1, false, true>(J, local, shb);
  } else if (J.axis == 1) {
    if (J.Y2) band_along<H, 1, true>(J, local, shb);
    else band_along<H, 1, false>(J, local, shb);
  } else {
    if (J.Y2) band_across<H, 1, true, false>(J, local, shb);
    else band_across<H, 1, false, false>(J, local, shb);
  }
}

// The divergence and the first pressure-mass pass (see k_div_band_x1), the band in fixed point:
// y0 = D .x1 delta and, with q, y1 = D .x1 (nu delta + q).
template <int H>
__global__ void __launch_bounds__(256, 2) k_fix_div_x1(const double* __restrict__ u1,
                                                       const double* __restrict__ u2,
                                                       const double* __restrict__ u3, int a, int b,
                                                       const double* __restrict__ q, double nu,
                                                       const __grid_constant__ FixBandJob J,
                                                       double* __restrict__ y1) {
  extern __shared__ __align__(16) int4 shb[];
  constexpr int N = kR + 2 * H;
  const int tid = threadIdx.x, nth = blockDim.x;
  const int nv = q ? 2 : 1;
  const int segs = J.segs, lpb = nth / (segs * nv), m = b, S = band_stage_s(segs, H);
  const int lines = b * b, line0 = (int)blockIdx.x * lpb, nl = min(lpb, lines - line0);
  double* raw = reinterpret_cast<double*>(shb + segs * band_seg(H));   // delta, then e
  double* out = raw + nv * lpb * kR * S;
  band_stage_op<H>(J.D[0], segs, shb);
  band_stage_zero<H>(raw, nv * lpb, m, segs, S);
  pdl_begin();
  const int64_t b2 = (int64_t)b * b;
  auto div_b = [&](int idx) -> int {   // idx / b
    return b == 1 ? idx : (int)(__umulhi((unsigned)idx, J.n1_mul) >> J.n1_sh);
  };
#pragma unroll 2
  for (int idx = tid; idx < nl * b; idx += nth) {
    const int l = div_b(idx), i1 = idx - l * b;
    const int line = line0 + l, i3 = div_b(line), i2 = line - i3 * b;
    const double* p1 = u1 + (int64_t)a * line + i1;
    const double* p2 = u2 + (int64_t)b * ((int64_t)a * i3 + i2) + i1;
    const double* p3 = u3 + b2 * i3 + (int64_t)b * i2 + i1;
    // the six neighbours are loaded before the first addition
    const double t[6] = {i1 < a ? p1[0] : 0.0,  i1 >= 1 ? p1[-1] : 0.0, i2 < a ? p2[0] : 0.0,
                         i2 >= 1 ? p2[-b] : 0.0, i3 < a ? p3[0] : 0.0,   i3 >= 1 ? p3[-b2] : 0.0};
    const double d = ((((t[0] - t[1]) + t[2]) - t[3]) + t[4]) - t[5];
    const int at = l * kR * S + band_stage(i1 + H, S);
    raw[at] = d;
    if (q) raw[lpb * kR * S + at] = fma(nu, d, q[(int64_t)line * b + i1]);
  }
  __syncthreads();
  // threads: segments of the lines of delta, then of e
  const int row = tid / segs, seg = tid - row * segs;
  const int o = row / lpb, l = row - o * lpb;
  if (l < nl && o < nv) {
    const double* p = raw + row * kR * S + seg;
    double* y = out + row * kR * S + seg;
    auto put = [&](int, int r, double v) { y[r * S] = v; };
    const unsigned redo = band_outputs<H, 1, false, false>(
        shb + seg * band_seg(H), 0, [&](int, int r) { return __ldg(J.D[0].rows + r * segs + seg); },
        [&](int, double (&x)[N]) {
#pragma unroll
          for (int k = 0; k < N; ++k) x[k] = p[(k & 7) * S + (k >> 3)];
        },
        [] {}, put);
    if (redo)
      band_chains(J, seg, m, m, redo,
                  [&](int, int j) { return raw[row * kR * S + band_stage(j + H, S)]; }, put);
  }
  __syncthreads();
  const int64_t o0 = (int64_t)b * line0;
  for (int idx = tid; idx < nl * b; idx += nth) {
    const int w = div_b(idx), at = w * kR * S + band_stage(idx - w * b, S);
    J.Y[o0 + idx] = out[at];
    if (q) y1[o0 + idx] = out[lpb * kR * S + at];
  }
}

FixBandOp band_op(const BandCore<double>& D, const BandFix& f) {
  if (f.half == 0) return FixBandOp{f.tab, f.rows, f.w0, D.val, D.start, D.width, D.width, 0};
  return FixBandOp{f.tab, f.rows, nullptr, D.cval, nullptr, 2 * D.half + 1, D.cpitch, D.half};
}

void band_divisor(int n1, FixBandJob& J) {
  int sh = 31 - __builtin_clz((unsigned)n1);
  if ((n1 & (n1 - 1)) == 0) --sh;   // (a power of two: one bit less, the multiplier fits)
  J.n1_sh = std::max(sh, 0);
  J.n1_mul = n1 == 1 ? 0 : (unsigned)(((uint64_t)1 << (32 + J.n1_sh)) / (unsigned)n1 + 1);
}

// threads of a block whose x1 lines need `segs` threads each
int band_threads(int block, int segs) {
  const int t = block > 0 ? std::min(block, kFixBandThreads) : kFixBandThreads;
  return std::max(t, (segs + 31) / 32 * 32);
}
template <int H, int NT, bool EPI>
void launch_fix_band(const FixBandBatch& fb, int blocks, int threads, int smem, cudaStream_t s) {
  static std::atomic<int> attr{0};
  // (a refused size is left as the thread's last error, which every caller of the passes checks)
  if (raise_smem_limit(k_fix_band<H, NT, EPI>, attr, smem) != cudaSuccess) return;
  launch_k(k_fix_band<H, NT, EPI>, blocks, threads, smem, s, fb);
}
template <int H>
void launch_fix_band(const FixBandBatch& fb, int nt, bool epi, int blocks, int threads, int smem,
                     cudaStream_t s) {
  if (nt > 1)
    epi ? launch_fix_band<H, 2, true>(fb, blocks, threads, smem, s)
        : launch_fix_band<H, 2, false>(fb, blocks, threads, smem, s);
  else
    epi ? launch_fix_band<H, 1, true>(fb, blocks, threads, smem, s)
        : launch_fix_band<H, 1, false>(fb, blocks, threads, smem, s);
}
template <int H>
void launch_fix_div(const double* u1, const double* u2, const double* u3, int a, int b,
                    const double* q, double nu, const FixBandJob& J, double* y1, int blocks,
                    int threads, int smem, cudaStream_t s) {
  static std::atomic<int> attr{0};
  if (raise_smem_limit(k_fix_div_x1<H>, attr, smem) != cudaSuccess) return;
  launch_k(k_fix_div_x1<H>, blocks, threads, smem, s, u1, u2, u3, a, b, q, nu, J, y1);
}

}  // namespace

bool fix_band_ok(const PassArgs<double>* jobs, int njobs) {
  const int H = jobs[0].f0.half;
  // (a launch with a g term or a Horner step has passes along x2 and x3 with one result only)
  bool epi = false;
  for (int j = 0; j < njobs; ++j) epi = epi || jobs[j].g || jobs[j].hmode;
  for (int j = 0; j < njobs; ++j) {
    const PassArgs<double>& a = jobs[j];
    if (epi && (a.axis == 1 || a.Y2)) return false;
    // rectangular bands: single-term passes along x2 and x3 of one item
    if (H == 0 && (epi || a.axis == 1 || a.nterms > 1 || a.nb > 1)) return false;
    const int m = H ? a.in.get(a.axis) : a.D0.rows, nb = a.nb > 1 ? a.nb : 1;
    if (!a.f0.tab || a.f0.half != H || a.D0.rows != m || a.Z ||
        (a.nterms > 1 && (!a.f1.tab || a.f1.half != H || a.D1.rows != m || a.c1 != 1.0)) ||
        (a.Y2 && (!a.D2.fix.tab || a.D2.fix.half != H || a.D2.rows != m)) ||
        a.c0 != 1.0 ||
        (a.axis == 1 && (a.g || a.hmode || (a.nterms > 1 && !a.Y2) || !fix_band_fits(m, H))) ||
        (a.Y2 && (a.g || a.hmode)) ||
        (H == 0 && a.D0.cols != a.in.get(a.axis)) ||
        a.in.size() / a.in.get(a.axis) * nb >= ((int64_t)1 << 30))
      return false;
  }
  return true;
}

void fix_band_multi(const PassArgs<double>* jobs, int njobs, cudaStream_t s) {
  FixBandBatch fb{};
  fb.njobs = njobs;
  const int H = jobs[0].f0.half;
  int threads = 32;
  for (int j = 0; j < njobs; ++j)
    threads = std::max(threads, band_threads(jobs[j].block, jobs[j].axis == 1
                                                               ? band_segs(jobs[j].D0.rows)
                                                               : 1));
  int blocks = 0, smem = 3 * kR * (band_row(H) + 1) * 16;   // (passes along x2 and x3)
  bool epi = false;
  int nt = 1;
  double flops = 0, bytes = 0;
  for (int j = 0; j < njobs; ++j) {
    const PassArgs<double>& a = jobs[j];
    FixBandJob& J = fb.job[j];
    J.X[0] = a.X0;
    J.X[1] = a.X1;
    J.D[0] = band_op(a.D0, a.f0);
    if (a.nterms > 1) J.D[1] = band_op(a.D1, a.f1);
    if (a.Y2) J.D[a.nterms] = band_op(a.D2, a.D2.fix);
    epi = epi || a.g || a.hmode;
    nt = std::max(nt, a.nterms);
    J.Y = a.Y;
    J.Y2 = a.Y2;
    J.g = a.g;
    J.gaxis = a.gaxis;
    J.gd1 = a.gdims.n1;
    J.gd12 = a.gdims.n1 * a.gdims.n2;
    J.hmode = a.hmode;
    J.hr = a.hr;
    J.hacc = a.hacc;
    J.hx = a.hx;
    J.in = a.in;
    band_divisor(a.in.n1, J);
    J.axis = a.axis;
    J.nterms = a.nterms;
    J.nops = a.nterms + (a.Y2 ? 1 : 0);
    J.nb = a.nb > 1 ? a.nb : 1;
    J.bs = a.bs;
    const int m = a.D0.rows;
    J.rows = m;
    J.segs = band_segs(m);
    const int lines = (int)(a.in.size() / a.in.get(a.axis)) * J.nb;
    fb.first[j] = blocks;
    if (a.axis == 1) {
      const int lpb = threads / J.segs;
      blocks += (lines + lpb - 1) / lpb;
      smem = std::max(smem, (int)band_along_smem(J.nops, lpb * (a.nterms + (a.Y2 ? 2 : 1)), J.segs, H));
    } else {
      blocks += (lines + threads - 1) / threads * J.segs;
    }
    const double outs = (double)lines * m;
    double fl = 2.0 * a.D0.width * outs, by = (double)a.in.size() * J.nb + outs;
    if (a.nterms > 1) { fl += 2.0 * a.D1.width * outs; by += outs; }
    if (a.Y2) { fl += 2.0 * a.D2.width * outs; by += outs; }
    if (a.g) { fl += 2.0 * outs; by += (double)a.gdims.size() * J.nb; }
    flops += fl;
    bytes += by * sizeof(double);
  }
  fb.first[njobs] = blocks;
  launch_begin(kClassBand64, s);
  switch (H) {
#define SHP_FIX_H(h) case h: launch_fix_band<h>(fb, nt, epi, blocks, threads, smem, s); break;
    case 0: launch_fix_band<0, 1, false>(fb, blocks, threads, smem, s); break;
    SHP_FIX_H(1) SHP_FIX_H(2) SHP_FIX_H(3) SHP_FIX_H(4) SHP_FIX_H(5) SHP_FIX_H(6)
#undef SHP_FIX_H
    default: break;
  }
  launch_end(kClassBand64, s, flops, bytes);
}

void fix_div_band_x1(const double* u1, const double* u2, const double* u3, int a, int b,
                     const double* q, double nu, const BandD<double>& D, double* y0, double* y1,
                     int block, cudaStream_t s) {
  FixBandJob J{};
  J.D[0] = band_op(D, D.fix);
  J.Y = y0;
  J.nterms = J.nops = 1;
  J.nb = 1;
  band_divisor(b, J);
  J.segs = band_segs(b);
  const int nv = q ? 2 : 1;
  const int H = D.fix.half, threads = band_threads(block, J.segs * nv);
  const int lpb = threads / (J.segs * nv), blocks = (b * b + lpb - 1) / lpb;
  const int smem = (int)band_along_smem(1, 2 * nv * lpb, J.segs, H);
  const double np = (double)b * b * b;
  launch_begin(kClassDiv, s);
  switch (H) {
#define SHP_FIX_H(h)                                                                  \
  case h: launch_fix_div<h>(u1, u2, u3, a, b, q, nu, J, y1, blocks, threads, smem, s); break;
    SHP_FIX_H(1) SHP_FIX_H(2) SHP_FIX_H(3) SHP_FIX_H(4) SHP_FIX_H(5) SHP_FIX_H(6)
#undef SHP_FIX_H
    default: break;
  }
  launch_end(kClassDiv, s, (q ? 8.0 : 6.0) * np + (q ? 4.0 : 2.0) * D.width * np,
             (3.0 * a * b * b + (q ? 3.0 : 1.0) * np) * sizeof(double));
}

}  // namespace shp
