// FP64 mode products of the fast diagonalisation (App. A.4) in fixed point on the FP16 tensor cores
// (fix.h). A block owns a group of lines: it finds the scale of each, writes its folded entries
// (or modes) as digit slices into shared memory in the operand order of mma.sync, and its warps
// form tiles of 16 lines by 8 outputs of both halves, the operator slices read from the
// cache in operand order. Bound by instruction issue (scaling and slicing the lines, adding the
// levels up and converting the sums take more slots than the multiplications). Measured against the
// FMA-chain kernels they replace on lines of 25 entries or more: P_0^-1 4947 -> 860 us at 128^3
// p = 3, 406 -> 200 at 64^3 (the pressure block of both by line solves), 60 -> 47 at 32^3.
#include <algorithm>
#include <atomic>

#include <cooperative_groups.h>

#include "fix.h"
#include "internal.h"
#include "profile.h"

namespace shp {
namespace {

// What a block needs of one operator: the slice table, and for lines that cannot be scaled the
// operator in doubles (K x K, row-major). Forward and backward: columns [even modes; odd modes],
// two halves of terms, he even ones; fold: the terms are x_k + x_{K-1-k} and x_k - x_{K-1-k} and
// the outputs the modes i and he + i, else the terms are the modes and the outputs the mirrored
// pair (i, K - 1 - i), the sum and the difference of the two halves. Plain: one half, he = K.
struct FixOp {
  FixTab t;
  const double* U;
  int K, he, fold, halves;
  int xbits, drain;   // bits of the scaled entries; steps between additions of the levels (fix.h)
};
FixOp fix_op(const FixTabs& f, const double* U, int K, int he, int use) {
  return FixOp{use == kFixBackward ? f.bw : f.fw, U, K, use == kFixPlain ? K : he,
               use == kFixForward, use == kFixPlain ? 1 : 2,
               use == kFixPlain ? 58 : (use == kFixBackward ? 57 : 56),
               fix_drain(use == kFixPlain ? 58 : 57)};
}

// uint4 entries of the line operand: the halves of mt tiles of 16 lines
__host__ __device__ constexpr int fix_frag_size(int mt, int ks, int halves = 2) {
  return halves * mt * ks * kFixSlices * 32;
}
// position of a lane's 16 bytes within the 512 of one (tile, step, slice): swizzled so that the
// word stores of neighbouring lines fall on different banks
__device__ __forceinline__ int fix_swz(int lane) { return lane ^ ((lane >> 3) & 3); }

__device__ __forceinline__ void fix_mma(float (&c)[4], const uint4& a, unsigned b0, unsigned b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a.x), "r"(a.y), "r"(a.z), "r"(a.w), "r"(b0), "r"(b1));
}

// the product alone
__device__ __forceinline__ void fix_mma0(float (&c)[4], const uint4& a, unsigned b0, unsigned b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%10,%10,%10,%10};"
      : "=f"(c[0]), "=f"(c[1]), "=f"(c[2]), "=f"(c[3])
      : "r"(a.x), "r"(a.y), "r"(a.z), "r"(a.w), "r"(b0), "r"(b1), "f"(0.f));
}

// a b + c
__device__ __forceinline__ long long mad_wide(int a, int b, long long c) {
  return c + (long long)a * b;
}

// s0, s1: the integer sums of the even and the odd half (units of 2^kFixUnit): line 16 mt + lane / 4
// + 8 (r / 2), output 8 t + 2 (lane % 4) + r % 2. mts: line tiles of the block. One rolled loop
// over both halves keeps the code in the instruction cache; the operator slices of a step are
// loaded while the step before is multiplied.
__device__ __forceinline__ void fix_gemm(const FixOp& op, const uint4* xf, int mts, int mt, int t,
                                         long long (&s0)[4], long long (&s1)[4]) {
  const int lane = threadIdx.x & 31, ks = op.t.ks;
  const uint4* bp = op.t.frag + (int64_t)t * ks * 96 + lane;
  const uint4* ap = xf + mt * ks * (kFixSlices * 32) + fix_swz(lane);
  const int bjump = (op.t.nt - 1) * ks * 96;                    // to the odd half
  const int ajump = (mts - 1) * ks * (kFixSlices * 32);
  uint4 b[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) b[c] = __ldg(bp + 32 * c);
  float acc[kFixSlices][4];
  int i2[4], i3[4], i4[4];   // moved sums of levels 2, 3, 4
#pragma unroll
  for (int r = 0; r < 4; ++r) {
#pragma unroll
    for (int l = 0; l < kFixSlices; ++l) acc[l][r] = 0.f;
    s1[r] = 0;
    i2[r] = i3[r] = i4[r] = 0;
  }
  const int total = op.halves * ks;
  int left = min(ks, op.drain);   // steps until the levels are added up
#pragma unroll 1
  for (int it = 0; it < total; ++it) {
    const unsigned bw[kFixSlices][2] = {{b[0].x, b[0].y}, {b[0].z, b[0].w}, {b[1].x, b[1].y},
                                        {b[1].z, b[1].w}, {b[2].x, b[2].y}, {b[2].z, b[2].w}};
    bp += 96;
    if (it + 1 == ks) bp += bjump;
    if (it + 1 < total) {
#pragma unroll
      for (int c = 0; c < 3; ++c) b[c] = __ldg(bp + 32 * c);
    }
#pragma unroll
    for (int i = 0; i < kFixSlices; ++i) {
      const uint4 a = ap[i * 32];
#pragma unroll
      for (int j = 0; i + j < kFixSlices; ++j) {
        // (level 3 is moved after every step)
        if (i == 0 && j == 3) fix_mma0(acc[j], a, bw[j][0], bw[j][1]);
        else fix_mma(acc[i + j], a, bw[j][0], bw[j][1]);
      }
    }
    ap += kFixSlices * 32;
    --left;
#pragma unroll
    for (int r = 0; r < 4; ++r) i3[r] += __float2int_rn(acc[3][r]);
    if (left == 0) {
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const int a5 = __float2int_rn(acc[5][r]), a4 = i4[r] + __float2int_rn(acc[4][r]);
        long long v = s1[r] + (a4 + ((a5 + (1 << (kFixDigit - 1))) >> kFixDigit));
        v = mad_wide(i3[r], 1 << kFixDigit, v);
        v = mad_wide(i2[r] + __float2int_rn(acc[2][r]), 1 << (2 * kFixDigit), v);
        v = mad_wide(__float2int_rn(acc[1][r]), 1 << (3 * kFixDigit), v);
        s1[r] = v + ((long long)__float2int_rn(acc[0][r]) << (4 * kFixDigit));
#pragma unroll
        for (int l = 0; l < kFixSlices; ++l) acc[l][r] = 0.f;
        i2[r] = i3[r] = i4[r] = 0;
      }
      left = min(it + 1 < ks ? ks - it - 1 : (it + 1 == ks ? ks : 2 * ks - it - 1), op.drain);
    } else if (((op.drain - left) & 1) == 0) {   // 32 terms
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        i2[r] += __float2int_rn(acc[2][r]);
        i4[r] += __float2int_rn(acc[4][r]);
        acc[2][r] = acc[4][r] = 0.f;
      }
    }
    if (it + 1 == ks) {   // the even half is complete
      ap += ajump;
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        s0[r] = s1[r];
        s1[r] = 0;
      }
    }
  }
}

// index of output i of half par along the line, -1 if it does not exist
__device__ __forceinline__ int fix_index(const FixOp& op, int par, int i) {
  const int he = op.he, h = op.K - he;
  if (i >= (par ? h : he)) return -1;
  return par == 0 ? i : (op.fold ? he + i : op.K - 1 - i);
}

// The outputs of a tile of 16 lines by 8 outputs of both halves, except those of lines that cannot
// be scaled: emit(row(line), index, value).
template <typename Row, typename Emit>
__device__ __forceinline__ void fix_tile(const FixOp& op, const uint4* xf, int mts, int mt, int t,
                                         const unsigned* key, int nl, Row&& row, Emit&& emit) {
  long long s0[4], s1[4];
  fix_gemm(op, xf, mts, mt, t, s0, s1);
  const int lane = threadIdx.x & 31;
  const int i0 = 8 * t + 2 * (lane & 3);
  const int* ex = op.t.ex + i0;
  const int2 e0 = __ldg(reinterpret_cast<const int2*>(ex));
  const int2 e1 = __ldg(reinterpret_cast<const int2*>(ex + 8 * op.t.nt));
  const int ja[2] = {fix_index(op, 0, i0), fix_index(op, 0, i0 + 1)};
  const int jb[2] = {fix_index(op, 1, i0), fix_index(op, 1, i0 + 1)};
#pragma unroll
  for (int hf = 0; hf < 2; ++hf) {
    const int line = 16 * mt + (lane >> 2) + 8 * hf;
    if (line >= nl) continue;
    const unsigned ky = key[line];
    if (fix_slow(ky)) continue;
    const int sh = (int)(ky >> 20) - 1022 - op.xbits + kFixUnit;
    const auto rw = row(line);
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      const long long a = s0[2 * hf + c], b = s1[2 * hf + c];
      if (ja[c] >= 0) emit(rw, ja[c], fix_to_double(op.fold ? a : a + b, sh + (c ? e0.y : e0.x)));
      if (jb[c] >= 0) emit(rw, jb[c], fix_to_double(op.fold ? b : a - b, sh + (c ? e1.y : e1.x)));
    }
  }
}

// The outputs of the lines that cannot be scaled, by FMA chains; ptr(line)[j stride]: entry j of a
// line.
template <typename ST, typename Ptr, typename Row, typename Emit>
__device__ __forceinline__ void fix_chains(const FixOp& op, const unsigned* key, int nl, ST stride,
                                           Ptr&& ptr, Row&& row, Emit&& emit) {
  const int he = op.he, K = op.K, h = K - he;
#pragma unroll 1
  for (int idx = threadIdx.x; idx < nl * he; idx += blockDim.x) {
    const int l = idx / he, i = idx - l * he;
    if (!fix_slow(key[l])) continue;
    const double* x = ptr(l);
    double ae = 0.0, ao = 0.0;
#pragma unroll 1
    for (int k = 0; k < he; ++k) {
      const double a = x[k * stride];
      const double b = k < h ? x[(op.fold ? K - 1 - k : he + k) * stride] : 0.0;
      ae = fma(op.fold ? op.U[(int64_t)k * K + i] : op.U[(int64_t)i * K + k],
               op.fold && k < h ? a + b : a, ae);
      if (k < h && i < h)
        ao = fma(op.fold ? op.U[(int64_t)k * K + he + i] : op.U[(int64_t)i * K + he + k],
                 op.fold ? a - b : b, ao);
    }
    const bool pair = !op.fold && i < h;
    emit(row(l), i, pair ? ae + ao : ae);
    if (i < h) emit(row(l), fix_index(op, 1, i), pair ? ae - ao : ao);
  }
}

// Digit slices of terms 2 kp and 2 kp + 1 of one line into both halves of the operand. v: the entries
// of the two terms, then their partners (zero where there is none). A line that cannot be scaled
// leaves zeros.
__device__ __forceinline__ void fix_slices(const FixOp& op, uint4* xf, int mts, int line, int kp,
                                           unsigned key, const double (&v)[4]) {
  const int h = op.K - op.he, ks = op.t.ks;
  const int emax = fix_slow(key) ? 4000 : (int)(key >> 20);   // (4000: everything shifts out)
  unsigned lo[2][2], hi[2][2];   // [half][term]
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const long long a = fix_of(v[q], emax, op.xbits), b = fix_of(v[2 + q], emax, op.xbits);
    const long long ve = op.fold ? a + b : a;
    const long long vo = op.fold ? (2 * kp + q < h ? a - b : 0) : b;
    // the bias makes every ten-bit field of the sum a digit plus 512
    constexpr unsigned long long kBias = 0x802008020080200ull;
    const unsigned long long we = (unsigned long long)ve + kBias;
    const unsigned long long wo = (unsigned long long)vo + kBias;
    lo[0][q] = (unsigned)we;
    hi[0][q] = (unsigned)(we >> 32);
    lo[1][q] = (unsigned)wo;
    hi[1][q] = (unsigned)(wo >> 32);
  }
  // operand position: row line % 16, terms 2 kp, 2 kp + 1 of step kp / 8
  const int row = line & 15, kk = kp & 7;
  const int lane = (row & 7) * 4 + (kk & 3), reg = (row >> 3) + 2 * (kk >> 2);
  unsigned* dst = reinterpret_cast<unsigned*>(
                      xf + (((line >> 4) * ks + (kp >> 3)) * kFixSlices) * 32 + fix_swz(lane)) + reg;
  const int half = mts * ks * kFixSlices * 128;   // words
#pragma unroll
  for (int par = 0; par < 2; ++par) {
    if (par == op.halves) break;
#pragma unroll
    for (int i = 0; i < kFixSlices; ++i) {
      const int bit = kFixDigit * (kFixSlices - 1 - i);
      unsigned d[2];
#pragma unroll
      for (int q = 0; q < 2; ++q)
        d[q] = bit >= 32 ? hi[par][q] >> (bit - 32)
                         : (bit > 22 ? __funnelshift_r(lo[par][q], hi[par][q], bit)
                                     : lo[par][q] >> bit);
      // 1024 + field as FP16, then minus 1536: the digit
      const unsigned w = (d[0] & 0x3ffu) | ((d[1] & 0x3ffu) << 16) | 0x64006400u;
      unsigned out;
      asm("sub.f16x2 %0, %1, %2;" : "=r"(out) : "r"(w), "r"(0x66006600u));
      dst[par * half + i * 128] = out;
    }
  }
}

// The line operand of a block: nl lines (16 mts rows, the rest zero), ptr(line)[j stride] entry j of
// a line. Each thread takes pairs of terms of single lines; it loads the entries of kFixHold of
// them before anything waits for one, finds the lines' scales (key, zeroed before by the block;
// any: set when a line cannot be scaled), and slices them from registers. along: neighbouring
// threads take neighbouring terms (contiguous lines), else neighbouring lines. Ends without a
// barrier. MTS: line tiles if fixed at compile time, else 0.
constexpr int kFixHold = 4;
template <int MTS = 0, typename ST, typename Ptr>
__device__ __forceinline__ void fix_load(const FixOp& op, uint4* xf, int mts_, int nl, bool along,
                                         unsigned* key, int* any, ST stride, Ptr&& ptr) {
  const int mts = MTS ? MTS : mts_;
  const int rows = 16 * mts, kps = 8 * op.t.ks, total = rows * kps;
  const int tid = threadIdx.x, nth = blockDim.x;
  const int he = op.he, h = op.K - he;
  // line and pair of task idx, packed (both below 2^16)
  auto place = [&](int idx) -> unsigned {
    const int w = along ? kps : rows;
    const int q = idx / w, r = idx - q * w;
    return along ? ((unsigned)q << 16 | (unsigned)r) : ((unsigned)r << 16 | (unsigned)q);
  };
  auto fetch = [&](unsigned at, double (&v)[4]) {
    const int l = (int)(at >> 16), k = 2 * (int)(at & 0xffffu);
#pragma unroll
    for (int c = 0; c < 4; ++c) v[c] = 0.0;
    if (l < nl && k < he) {
      const double* x = ptr(l);
      const double* p = x + (ST)k * stride;
      const ST back = op.fold ? -stride : stride;
      const double* pp = x + (ST)(op.fold ? op.K - 1 - k : he + k) * stride;
      v[0] = *p;
      if (k + 1 < he) v[1] = p[stride];
      if (k < h) v[2] = *pp;
      if (k + 1 < h) v[3] = pp[back];
    }
  };
  auto raise = [&](unsigned at, const double (&v)[4]) {
    unsigned m = max(max(fix_key(v[0]), fix_key(v[1])), max(fix_key(v[2]), fix_key(v[3])));
    unsigned* k = key + (at >> 16);
    if (along) {   // the eight threads of a step's pairs share a line (kps and nth: multiples of 8)
      const unsigned mask = 0xffu << (tid & 24);
#pragma unroll
      for (int o = 4; o; o >>= 1) m = max(m, __shfl_xor_sync(mask, m, o));
      if ((tid & 7) == 0) atomicMax(k, m);
    } else {
      atomicMax(k, m);
    }
  };
  double v[kFixHold][4];
  unsigned at[kFixHold];
#pragma unroll
  for (int n = 0; n < kFixHold; ++n) {
    const int idx = tid + n * nth;
    if (idx < total) {
      at[n] = place(idx);
      fetch(at[n], v[n]);
    }
  }
#pragma unroll
  for (int n = 0; n < kFixHold; ++n)
    if (tid + n * nth < total) raise(at[n], v[n]);
#pragma unroll 1
  for (int idx = tid + kFixHold * nth; idx < total; idx += nth) {
    const unsigned w = place(idx);
    double x[4];
    fetch(w, x);
    raise(w, x);
  }
  __syncthreads();
#pragma unroll 1
  for (int idx = tid, n = 0; idx < total; idx += nth, ++n) {
    if (n >= kFixHold) {
      at[0] = place(idx);
      fetch(at[0], v[0]);
    }
    const int l = (int)(at[0] >> 16);
    const unsigned m = key[l];
    if (fix_slow(m)) *any = 1;
    fix_slices(op, xf, mts, l, (int)(at[0] & 0xffffu), m, v[0]);
#pragma unroll
    for (int q = 0; q + 1 < kFixHold; ++q) {   // (a rolled loop: the registers move up)
      at[q] = at[q + 1];
#pragma unroll
      for (int c = 0; c < 4; ++c) v[q][c] = v[q + 1][c];
    }
  }
}

// ---- one direction ---------------------------------------------------------------------------
struct FixJob {
  const double* X;
  double* Y;
  FixOp op;
  int64_t L, R;            // extents before and after the contracted direction
  const double* invd;      // optional multiplier per output entry
  double post;
  int has_post;            // post != 1 (an integer: an FP64 compare costs as much as an FMA)
};
struct FixBatch {
  FixJob job[kMaxModeJobs];
  int first[kMaxModeJobs + 1];
  int njobs;
};

// A block owns 16 neighbouring lines and all their outputs (blocks of 32 lines read the operator
// half as often, but leave fewer warps per SM and a longer last wave: 128^3 P_0^-1 867 against
// 1002 us, 96^3 350 against 431). IT: index type of the line and
// entry arithmetic (int below 2^31 entries: 64-bit division issues FP64-pipe instructions).
template <typename IT>
__global__ void __launch_bounds__(320, 2) k_fix_mode(const __grid_constant__ FixBatch fb) {
  extern __shared__ __align__(16) uint4 xf[];
  constexpr int lb = 16;
  __shared__ unsigned key[lb];
  __shared__ IT base[lb];   // first entry of each line
  __shared__ int any;
  int jb = 0;
  while (jb + 1 < fb.njobs && (int)blockIdx.x >= fb.first[jb + 1]) ++jb;
  const FixJob& J = fb.job[jb];
  const FixOp& op = J.op;
  const int K = op.K;
  const int tid = threadIdx.x, nth = blockDim.x, warp = tid >> 5, nw = nth >> 5;
  const IT JL = (IT)J.L;
  const IT lines = JL * (IT)J.R;
  const IT line0 = (IT)((int)blockIdx.x - fb.first[jb]) * lb;
  const int nl = (int)(lines - line0 < lb ? lines - line0 : lb);
  for (int l = tid; l < lb; l += nth) {
    key[l] = 0;
    const IT line = line0 + l, r = line / JL;
    base[l] = (line - r * JL) + JL * ((IT)K * r);
  }
  if (tid == 0) any = 0;
  pdl_begin();
  __syncthreads();
  const auto ptr = [&](int l) { return J.X + base[l]; };
  const auto row = [&](int l) { return base[l]; };
  fix_load<1>(op, xf, 1, nl, JL == 1, key, &any, JL, ptr);
  __syncthreads();
  const auto emit = [&](IT first, int i, double v) {
    const IT o = first + JL * i;
    if (J.invd) v *= J.invd[o];
    else if (J.has_post) v *= J.post;
    J.Y[o] = v;
  };
  for (int t = warp; t < op.t.nt; t += nw) fix_tile(op, xf, 1, 0, t, key, nl, row, emit);
  if (any) fix_chains(op, key, nl, JL, ptr, row, emit);
}

// ---- fused passes ------------------------------------------------------------------------------
struct FixPlaneJob {
  const double* X;
  double* Y;
  FixOp first, second;   // the two products in their order: x1, x2 forward; x2, x1 backward
  int n1, n2;
  double post;
  int has_post;
};
struct FixPlaneBatch {
  FixPlaneJob job[kMaxModeJobs];
  int first[kMaxModeJobs + 1];   // first plane of each job
  int njobs;
  int fwd;
  int raw_off;                   // offset of the intermediate (uint4)
};

__device__ __forceinline__ void st_cluster(double* p, int rank, double v) {
  const uint32_t local = (uint32_t)__cvta_generic_to_shared(p);
  uint32_t remote;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(local), "r"(rank));
  asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(remote), "d"(v) : "memory");
}

__host__ __device__ constexpr int fix_slice(int n, int cs) { return (n + cs - 1) / cs; }
__host__ __device__ constexpr int fix_mts(int lines) { return (lines + 15) / 16; }

// The x1 and x2 products of every x1-x2 plane, one cluster of cs blocks per plane. Each block
// takes a slice of the lines of the first product and stores every result into the block that owns
// its line of the second product; after the cluster barrier each block forms the second product
// of its own slice of lines. Between the products the values are doubles, as if stored, so the
// results have the bits of two k_fix_mode launches.
__global__ void __launch_bounds__(512) k_fix_plane(const __grid_constant__ FixPlaneBatch pb) {
  namespace cg = cooperative_groups;
  cg::cluster_group cl = cg::this_cluster();
  const int cs = (int)cl.num_blocks(), rank = (int)cl.block_rank();
  extern __shared__ __align__(16) uint4 xf[];
  __shared__ unsigned key[2][256];
  __shared__ int any[2];
  const int pidx = (int)blockIdx.x / cs;
  int jb = 0;
  while (jb + 1 < pb.njobs && pidx >= pb.first[jb + 1]) ++jb;
  const FixPlaneJob& J = pb.job[jb];
  const int plane = pidx - pb.first[jb];
  const int n1 = J.n1, n2 = J.n2;
  const bool fwd = pb.fwd != 0;
  // lines of the two products: forward rows (x2 index) then columns (x1 index), backward the
  // other way round; slices of fix_slice lines per block
  const int la_n = fwd ? n2 : n1, lb_n = fwd ? n1 : n2;
  const int sa = fix_slice(la_n, cs), sb = fix_slice(lb_n, cs);
  const int a0 = min(sa * rank, la_n), na = min(sa, la_n - a0);
  const int b0 = min(sb * rank, lb_n), nbl = min(sb, lb_n - b0);
  const int ma = fix_mts(na), mb = fix_mts(nbl);
  const int Pb = sb | 1;   // pitch of the intermediate [entry][line]
  double* raw = reinterpret_cast<double*>(xf + pb.raw_off);
  const int tid = threadIdx.x, nth = blockDim.x, warp = tid >> 5, nw = nth >> 5;
  const int64_t np = (int64_t)n1 * n2;
  const double* X = J.X + plane * np;
  double* Y = J.Y + plane * np;
  const FixOp& A = J.first;
  const FixOp& B = J.second;
  for (int l = tid; l < 512; l += nth) (&key[0][0])[l] = 0;
  if (tid < 2) any[tid] = 0;
  pdl_begin();
  __syncthreads();
  const auto ptr_a = [&](int l) { return X + (fwd ? (a0 + l) * n1 : a0 + l); };
  const auto ptr_b = [&](int l) { return (const double*)raw + l; };
  const int stride_a = fwd ? 1 : n1;
  const auto row = [](int l) { return l; };
  fix_load(A, xf, ma, na, fwd, key[0], &any[0], stride_a, ptr_a);
  if (cs > 1) cl.sync(); else __syncthreads();   // (every block runs before any store into it)
  const auto emit_a = [&](int l, int i, double v) {
    const int owner = i / sb;
    double* dst = raw + (a0 + l) * Pb + (i - owner * sb);
    if (owner == rank) *dst = v;
    else st_cluster(dst, owner, v);
  };
  for (int u = warp; u < ma * A.t.nt; u += nw)
    fix_tile(A, xf, ma, u % ma, u / ma, key[0], na, row, emit_a);
  if (any[0]) fix_chains(A, key[0], na, stride_a, ptr_a, row, emit_a);
  if (cs > 1) cl.sync(); else __syncthreads();
  if (nbl <= 0) return;
  fix_load(B, xf, mb, nbl, false, key[1], &any[1], Pb, ptr_b);
  __syncthreads();
  const auto emit_b = [&](int l, int i, double v) {
    if (J.has_post) v *= J.post;
    Y[fwd ? i * n1 + b0 + l : (b0 + l) * n1 + i] = v;
  };
  for (int u = warp; u < mb * B.t.nt; u += nw)
    fix_tile(B, xf, mb, u % mb, u / mb, key[1], nbl, row, emit_b);
  if (any[1]) fix_chains(B, key[1], nbl, Pb, ptr_b, row, emit_b);
}

struct FixLineJob {
  const double* X;
  double* Y;
  FixOp fwd, bwd;
  int64_t L;
  int n1;
  const double* invd;   // multiplier per entry between the products
  double post;
  int has_post;
};
struct FixLineBatch {
  FixLineJob job[kMaxModeJobs];
  int first[kMaxModeJobs + 1];
  int njobs;
  int raw_off;
};

// The forward x3 product, the eigenvalue scaling and the backward x3 product of 16 neighbouring x3
// lines.
__global__ void __launch_bounds__(512) k_fix_line3(const __grid_constant__ FixLineBatch fb) {
  extern __shared__ __align__(16) uint4 xf[];
  constexpr int lb = 16, P = lb + 1;
  __shared__ unsigned key[2][lb];
  __shared__ int any[2];
  int jb = 0;
  while (jb + 1 < fb.njobs && (int)blockIdx.x >= fb.first[jb + 1]) ++jb;
  const FixLineJob& J = fb.job[jb];
  const FixOp& A = J.fwd;
  const int64_t line0 = (int64_t)((int)blockIdx.x - fb.first[jb]) * lb;
  const int nl = (int)(J.L - line0 < lb ? J.L - line0 : lb);
  double* raw = reinterpret_cast<double*>(xf + fb.raw_off);
  const int tid = threadIdx.x, nth = blockDim.x, warp = tid >> 5, nw = nth >> 5;
  for (int l = tid; l < 2 * lb; l += nth) (&key[0][0])[l] = 0;
  if (tid < 2) any[tid] = 0;
  pdl_begin();
  __syncthreads();
  const auto ptr_a = [&](int l) { return J.X + line0 + l; };
  const auto ptr_b = [&](int l) { return (const double*)raw + l; };
  const auto row = [](int l) { return l; };
  fix_load<1>(A, xf, 1, nl, false, key[0], &any[0], J.L, ptr_a);
  __syncthreads();
  const auto emit_a = [&](int l, int i, double v) {
    v *= J.invd[line0 + l + J.L * i];
    raw[i * P + l] = v;
  };
  for (int t = warp; t < A.t.nt; t += nw) fix_tile(A, xf, 1, 0, t, key[0], nl, row, emit_a);
  if (any[0]) fix_chains(A, key[0], nl, J.L, ptr_a, row, emit_a);
  __syncthreads();
  fix_load<1>(J.bwd, xf, 1, nl, false, key[1], &any[1], P, ptr_b);
  __syncthreads();
  const auto emit_b = [&](int l, int i, double v) {
    if (J.has_post) v *= J.post;
    J.Y[line0 + l + J.L * i] = v;
  };
  for (int t = warp; t < J.bwd.t.nt; t += nw)
    fix_tile(J.bwd, xf, 1, 0, t, key[1], nl, row, emit_b);
  if (any[1]) fix_chains(J.bwd, key[1], nl, P, ptr_b, row, emit_b);
}

double eo_flops(int K, int he) {
  const double e = he, o = K - he;
  return 2.0 * (e * e + o * o);
}

// warps of a block whose tiles come in `units`: whole rounds of at most `cap` warps
int fix_warps(int units, int cap) {
  const int rounds = (units + cap - 1) / cap;
  return (units + rounds - 1) / rounds;
}

}  // namespace

cudaError_t fix_mode_multi(const ModeArgs<double>* jobs, int njobs, cudaStream_t s) {
  FixBatch fb{};
  fb.njobs = njobs;
  const int target = jobs[0].block > 0 ? std::min(jobs[0].block, 512) : 512;
  int nt = 1, ks = 1;
  for (int j = 0; j < njobs; ++j) {
    const ModeArgs<double>& m = jobs[j];
    if (!m.fx.fw.frag || m.eo_he < 1 || m.m != m.in.get(m.axis) || m.ld != m.m ||
        m.plain != jobs[0].plain || (m.lam1 && !m.invd))
      return cudaErrorInvalidValue;
    nt = std::max(nt, m.fx.fw.nt);
    ks = std::max(ks, m.fx.fw.ks);
  }
  constexpr int lb = 16;
  const int smem = fix_frag_size(1, ks, jobs[0].plain ? 1 : 2) * (int)sizeof(uint4);
  int blocks = 0;
  double flops = 0, bytes = 0;
  bool i32 = true;
  for (int j = 0; j < njobs; ++j) {
    const ModeArgs<double>& m = jobs[j];
    FixJob& J = fb.job[j];
    const Dims in = m.in;
    J.X = m.X;
    J.Y = m.Y;
    J.op = fix_op(m.fx, m.U, m.m, m.eo_he,
                  m.plain ? kFixPlain : (m.trans ? kFixForward : kFixBackward));
    J.L = m.axis == 1 ? 1 : (m.axis == 2 ? in.n1 : (int64_t)in.n1 * in.n2);
    J.R = m.axis == 1 ? (int64_t)in.n2 * in.n3 : (m.axis == 2 ? in.n3 : 1);
    J.invd = m.invd;
    J.post = m.post;
    J.has_post = J.post != 1.0;
    fb.first[j] = blocks;
    blocks += (int)((J.L * J.R + lb - 1) / lb);
    flops += (double)(J.L * J.R) * (m.plain ? 2.0 * m.m * m.m : eo_flops(m.m, m.eo_he));
    bytes += 2.0 * (double)in.size() * sizeof(double);
    if (in.size() + 1024 >= ((int64_t)1 << 31)) i32 = false;
  }
  fb.first[njobs] = blocks;
  const int threads = 32 * std::min(10, fix_warps(nt, std::max(4, target / 32)));
  static std::atomic<int> a32{0}, a64{0};
  const cudaError_t e = i32 ? raise_smem_limit(k_fix_mode<int>, a32, smem + 1024)
                            : raise_smem_limit(k_fix_mode<int64_t>, a64, smem + 1024);
  if (e != cudaSuccess) return e;
  const int cls = jobs[0].plain ? kClassLine : kClassMode;
  launch_begin(cls, s);
  const cudaError_t l = i32 ? launch_k(k_fix_mode<int>, blocks, threads, smem, s, fb)
                            : launch_k(k_fix_mode<int64_t>, blocks, threads, smem, s, fb);
  launch_end(cls, s, flops, bytes);
  return l;
}

bool fix_plane_multi(const FdPlaneArgs* jobs, int njobs, int fwd, int block, int cluster,
                    cudaStream_t s) {
  if (cluster != 1 && cluster != 2 && cluster != 4) return false;
  FixPlaneBatch pb{};
  pb.njobs = njobs;
  pb.fwd = fwd;
  int planes = 0, frag = 0, raw = 0;
  double flops = 0, bytes = 0;
  for (int j = 0; j < njobs; ++j) {
    const FdPlaneArgs& a = jobs[j];
    if (fd_plane_smem(a.in) == 0 || a.eo1 < 1 || a.eo2 < 1 || !a.fx1.fw.frag || !a.fx2.fw.frag)
      return false;
    FixPlaneJob& J = pb.job[j];
    J.X = a.X;
    J.Y = a.Y;
    J.n1 = a.in.n1;
    J.n2 = a.in.n2;
    J.post = a.post;
    J.has_post = a.post != 1.0;
    const int use = fwd ? kFixForward : kFixBackward;
    const FixOp o1 = fix_op(a.fx1, a.U1, a.in.n1, a.eo1, use);
    const FixOp o2 = fix_op(a.fx2, a.U2, a.in.n2, a.eo2, use);
    J.first = fwd ? o1 : o2;
    J.second = fwd ? o2 : o1;
    const int sa = fix_slice(fwd ? a.in.n2 : a.in.n1, cluster);
    const int sb = fix_slice(fwd ? a.in.n1 : a.in.n2, cluster);
    frag = std::max(frag, std::max(fix_frag_size(fix_mts(sa), J.first.t.ks),
                                   fix_frag_size(fix_mts(sb), J.second.t.ks)));
    raw = std::max(raw, J.second.K * (sb | 1));
    pb.first[j] = planes;
    planes += a.in.n3;
    flops += (double)a.in.n3 *
             (a.in.n2 * eo_flops(a.in.n1, a.eo1) + a.in.n1 * eo_flops(a.in.n2, a.eo2));
    bytes += 2.0 * (double)a.in.size() * sizeof(double);
  }
  pb.first[njobs] = planes;
  pb.raw_off = frag;
  const int smem = frag * (int)sizeof(uint4) + raw * (int)sizeof(double);
  // (the largest planes need the operands spread over more blocks than asked for)
  if (smem > 220 * 1024)
    return cluster < 4 && fix_plane_multi(jobs, njobs, fwd, block, 2 * cluster, s);
  const int threads = std::max(128, block > 0 ? std::min(block, 512) : 512);
  static std::atomic<int> attr{0};
  if (raise_smem_limit(k_fix_plane, attr, smem + 2048) != cudaSuccess) return false;
  launch_begin(kClassMode, s);
  launch_kc(k_fix_plane, planes * cluster, threads, smem, s, cluster, pb);
  launch_end(kClassMode, s, flops, bytes);
  return true;
}

bool fix_line3_multi(const FdLineArgs* jobs, int njobs, int block, cudaStream_t s) {
  FixLineBatch fb{};
  fb.njobs = njobs;
  int ks = 1, K = 1;
  for (int j = 0; j < njobs; ++j) {
    if (jobs[j].eo3 < 1 || !jobs[j].fx3.fw.frag || !jobs[j].invd) return false;
    ks = std::max(ks, jobs[j].fx3.fw.ks);
    K = std::max(K, jobs[j].in.n3);
  }
  constexpr int lb = 16;
  fb.raw_off = fix_frag_size(1, ks);
  int blocks = 0;
  double flops = 0, bytes = 0;
  for (int j = 0; j < njobs; ++j) {
    const FdLineArgs& a = jobs[j];
    FixLineJob& J = fb.job[j];
    J.X = a.X;
    J.Y = a.Y;
    J.fwd = fix_op(a.fx3, a.U3, a.in.n3, a.eo3, kFixForward);
    J.bwd = fix_op(a.fx3, a.U3, a.in.n3, a.eo3, kFixBackward);
    J.L = (int64_t)a.in.n1 * a.in.n2;
    J.n1 = a.in.n1;
    J.invd = a.invd;
    J.post = a.post;
    J.has_post = a.post != 1.0;
    fb.first[j] = blocks;
    blocks += (int)((J.L + lb - 1) / lb);
    flops += 2.0 * (double)J.L * eo_flops(a.in.n3, a.eo3);
    bytes += 2.0 * (double)a.in.size() * sizeof(double);
  }
  fb.first[njobs] = blocks;
  const int smem = fb.raw_off * (int)sizeof(uint4) + K * (lb + 1) * (int)sizeof(double);
  if (smem > 220 * 1024) return false;
  const int threads = std::max(128, block > 0 ? std::min(block, 512) : 512);
  static std::atomic<int> attr{0};
  if (raise_smem_limit(k_fix_line3, attr, smem + 1024) != cudaSuccess) return false;
  launch_begin(kClassMode, s);
  launch_k(k_fix_line3, blocks, threads, smem, s, fb);
  launch_end(kClassMode, s, flops, bytes);
  return true;
}

}  // namespace shp
