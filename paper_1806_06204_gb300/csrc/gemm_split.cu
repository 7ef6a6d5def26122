// Split-precision FP64 GEMM on the tensor cores (tcgen05 + TMEM + TMA), the Ozaki
// scheme: every FP64 operand row (of op(A)) / column (of op(B)) is scaled by a
// power of two 2^e so that its entries lie in [-1/2, 1/2], rounded to the
// fixed-point integer N = round(x 2^(bS - e)) and written in S balanced base-2^b
// digits,
//     x 2^-e = sum_{s=1..S} d_s 2^{-bs} (+ rounding below 2^{-bS-1}),
//     |d_s| <= 2^(b-1),
// each stored as the integer it is, which the slice type holds exactly (BF16 up
// to 256, FP16 up to 2048, E4M3 up to 16).  A product is the sum over digit pairs
// (s, t) with s + t <= top of tensor-core GEMMs, one TMEM accumulator per level
// s + t, whose sums of integers are exact in FP32 while p k 2^(2b-2) <= 2^24 (p
// pairs in the level, k terms).  Balanced digits make the dropped pairs and the
// rounding zero-mean (truncated digits bias every term of a Gram diagonal the
// same way).
//
//   BF16 form  b = 8, S = 7 (56 bits), levels 2..9: 34 pairs (zolo_dgemm's
//              slices = 9); S = 6 (48 bits), levels 2..8: 26 pairs (slices = 8)
//   FP16 form  b = 8, S = 7, levels 2..8: 28 pairs
//   FP8 form   b = 5, S = 11 (55 bits), levels 2..13: 76 pairs at the doubled rate
//
// The leading levels (2..6 of the 8-bit digits, 2..9 of the 5-bit ones) are exact
// over a K-chunk of 192 (4096) terms and are added to an int64 in units of 2^-48
// after every chunk; the levels below go to one float in units of 2^-56 (2^-65),
// whose FP32 rounding lies 2^-64 below the leading level.  At the end the two are joined in
// integers, rounded once to FP64 and
// scaled by 2^(e_i + f_j) through the exponent field.  The digit width was
// measured on the CPU against exact products (rms error over row and column
// maxima, K = 512, N(0,1) / Gram / operands graded over eight decades): 34 pairs
// of 8-bit digits 0.7 / 0.8 / 0.4 e-16, the 53 pairs of nine 6-bit digits they
// replace 4.2 / 4.6 / 1.5 e-16; 28 pairs 4.2 / 4.6 / 4.1 e-16, the 36 pairs of
// eight 7-bit digits they replace 4.7 / 8.1 / 4.5 e-16.  A K block of the FP8 form
// is 128 one-byte elements, the same 128-byte swizzled rows as the 16-bit forms,
// and one MMA takes K = 32 (32 bytes), so the shared-memory layout and
// descriptors are the same byte for byte.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_fp8.h>

#include <climits>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <algorithm>
#include <mutex>

#include <cooperative_groups.h>

#include "tc_ptx.cuh"
#include "zolo_internal.h"

namespace zolo {
namespace {

constexpr int kTileM = 128;
constexpr int kRowBytes = 128;     // one 128-byte swizzle row of K per tile row
// The slice forms: digit width, element bytes (K elements per 128-byte row), the
// chunk of K whose leading level sums are exact, tile width BN, the last level
// (1-based) that goes to the int64, and the largest 0-based s + t kept.
template <int FORM> struct Form;
template <> struct Form<kFormBF16> {
  static constexpr int kBits = 8, kElem = 2, kChunkK = 192, kIntTop = 6, kLo = 8;
  __host__ __device__ static constexpr int top(int S) { return S; }
};
template <> struct Form<kFormFP16> {
  static constexpr int kBits = 8, kElem = 2, kChunkK = 192, kIntTop = 6, kLo = 8;
  __host__ __device__ static constexpr int top(int S) { return S - 1; }
};
template <> struct Form<kFormFP8> {
  static constexpr int kBits = 5, kElem = 1, kChunkK = 4096, kBN = 32, kIntTop = 9, kLo = 17;
  __host__ __device__ static constexpr int top(int S) { return S; }
};
template <int FORM> __host__ __device__ constexpr int form_bk() { return kRowBytes / Form<FORM>::kElem; }
constexpr int kARing = 7;
constexpr int kGroupM = 8;         // tile rows per group of tiles (L2 reuse of the A slices)
constexpr int kEpiWarps = 16;      // four per TMEM lane quarter, each owning a quarter of the columns
constexpr int kThreads = 64 + 32 * kEpiWarps;   // warp 0 TMA, warp 1 MMA, the rest epilogue

// ----------------------------------------------------------------- slicing
// One batch entry per blockIdx.z; operand b starts at X + b * strideX.
// Row i of op(X) (rows x K):  trans = 0: X[i + k ldx] (rows contiguous),
//                             trans = 1: X[k + i ldx] (row contiguous along k).

// e with |x| < 2^(e - 1) (0 for a zero).  Integer arithmetic on the FP64 bit patterns
// (|x| orders like its magnitude bits); no FP64 pipe work.
__device__ __forceinline__ int exp_above(unsigned long long mag) {
  if (mag == 0) return 0;
  const int ef = (int)(mag >> 52);
  return ef ? ef - 1021 : -1021;   // normal: |x| < 2^(ef-1022); subnormal: < 2^-1022
}

// ek[k] = the exponent bound of column k of the (rows x K) view of op(X)
// (0 for a zero column or k >= K): scaling that column by 2^-ek[k] puts its
// largest magnitude in [1/4, 1/2).
__global__ void col_exp_kernel(const double* __restrict__ X, int64_t ldx, int64_t strideX, int trans,
                               int rows, int K, int* __restrict__ ek, int K_pad) {
  __shared__ unsigned long long red[8][33];
  const double* Xb = X + blockIdx.z * strideX;
  const int tx = threadIdx.x, ty = threadIdx.y;   // 32 x 8
  const unsigned long long kMag = 0x7FFFFFFFFFFFFFFFull;
  const int k0 = blockIdx.x * 32;
  if (trans) {    // element (i, k) = X[k + i ldx]: threads along k, rows split over ty
    unsigned long long mx = 0;
    const int k = k0 + tx;
    if (k < K)
      for (int i = ty; i < rows; i += 8) {
        const unsigned long long b = (unsigned long long)__double_as_longlong(Xb[k + (int64_t)i * ldx]) & kMag;
        mx = b > mx ? b : mx;
      }
    red[ty][tx] = mx;
  } else {        // element (i, k) = X[i + k ldx]: one warp per column, lanes along i
    for (int kk = ty; kk < 32; kk += 8) {
      unsigned long long mx = 0;
      const int k = k0 + kk;
      if (k < K)
        for (int i = tx; i < rows; i += 32) {
          const unsigned long long b = (unsigned long long)__double_as_longlong(Xb[i + (int64_t)k * ldx]) & kMag;
          mx = b > mx ? b : mx;
        }
      for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long t = __shfl_xor_sync(0xffffffffu, mx, o);
        mx = t > mx ? t : mx;
      }
      if (tx == 0) red[0][kk] = mx;   // row 0 collects the columns
    }
    __syncthreads();
    if (ty == 0) {
      const int k = k0 + tx;
      if (k < K_pad) ek[blockIdx.z * K_pad + k] = (k < K) ? exp_above(red[0][tx]) : 0;
    }
    return;
  }
  __syncthreads();
  if (ty == 0) {
    unsigned long long mx = red[0][tx];
    for (int y = 1; y < 8; ++y) mx = red[y][tx] > mx ? red[y][tx] : mx;
    const int k = k0 + tx;
    if (k < K_pad) ek[blockIdx.z * K_pad + k] = (k < K) ? exp_above(mx) : 0;
  }
}

// e with |x| <= 2^(e - 1) from the high word of |x|, its low bit set where the low word is
// not zero (one where that is a subnormal below 2^-1042).  A power of two is its own bound:
// the leading digit takes +-2^(b-1), and a column of reflectors, whose largest entry is the 1
// of its diagonal, keeps one more bit of the others.
__device__ __forceinline__ int exp_bound(int nz) {
  const int b = nz >= 0x7FF00000 ? nz : nz - 1;   // Inf and NaN: 1026
  return b >> 20 ? (b >> 20) - 1021 : -1021;
}

// N = round(x 2^(bS - e)) from the bit pattern (|x| <= 2^(e-1), so |N| <= 2^(bS-1));
// ties round away from zero.  The mantissa is raised by 8 bits, so every exponent is one
// right shift (by 5 at least: a subnormal of a row of subnormals; what is shifted further
// than 62 is zero).
template <int BITS>
__device__ __forceinline__ long long fixed_point(double x, int e) {
  const int hi = __double2hiint(x);
  const int ef = (hi >> 20) & 0x7FF;
  const unsigned mh = ((unsigned)hi & 0xFFFFFu) | (ef ? 0x100000u : 0u);
  const unsigned long long M = ((unsigned long long)mh << 32 | (unsigned)__double2loint(x)) << 8;
  const int t = min(max(1083 - BITS + e - max(ef, 1), 1), 63);
  const long long F = (long long)((M + (1ull << (t - 1))) >> t);
  const long long m = hi >> 31;
  return (F ^ m) - m;
}

// The S balanced digits of two neighbouring entries, plane by plane, as one packed
// pair of the slice type: o(s, pair).  Adding half a unit to every digit but the
// leading one (a constant) turns the balanced digits into the plain ones plus that
// half, so the digits of N are fields of one 64-bit word; an integer below 2^10
// becomes FP16, and one below 2^23 FP32, by setting the exponent bits of 1024 (2^23)
// over it and subtracting that: no conversion instruction (16 lanes a clock) per digit.
template <int S, int FORM, class Put>
__device__ __forceinline__ void slice_pair(double x0, double x1, int e0, int e1, Put put) {
  constexpr int B = Form<FORM>::kBits;
  constexpr long long half = 1ll << (B - 1);
  constexpr long long bias = []() {
    long long t = 0;
    for (int s = 0; s < S - 1; ++s) t |= half << (B * s);
    return t;
  }();
  const long long n0 = fixed_point<B * S>(x0, e0) + bias, n1 = fixed_point<B * S>(x1, e1) + bias;
  // digit s (1-based, 1 leads) plus half; the fields of the 8-bit digits are bytes
  auto field = [&](long long n, int s) -> unsigned {
    const int sh = B * (S - s);
    return s == 1 ? (unsigned)((int)(n >> sh) + (int)half) : (unsigned)(n >> sh) & ((1u << B) - 1);
  };
  auto word = [](long long n, int byte) { return (unsigned)(n >> (byte & 4) * 8); };
#pragma unroll
  for (int s = 1; s <= S; ++s) {
    const int byte = S - s;
    if (FORM == kFormBF16) {
      auto biased = [&](long long n) -> float {
        return __uint_as_float(s == 1 ? 0x4B000000u | field(n, s)
                                      : __byte_perm(word(n, byte), 0x4B000000u, 0x7440 | (byte & 3)));
      };
      const float f0 = biased(n0) - (8388608.f + (float)half), f1 = biased(n1) - (8388608.f + (float)half);
      // a digit has at most 8 significant bits: its BF16 is the float's upper half
      put(s - 1, __byte_perm(__float_as_uint(f0), __float_as_uint(f1), 0x7632));
    } else {
      const unsigned t =
          FORM == kFormFP16 && s > 1
              ? (__byte_perm(word(n0, byte), word(n1, byte), 0x0400 | (byte & 3) | (byte & 3) << 8) & 0x00FF00FFu) |
                    0x64006400u
              : (field(n0, s) | field(n1, s) << 16) + 0x64006400u;
      const __half2 h = __hsub2(*reinterpret_cast<const __half2*>(&t),
                                __half2half2(__ushort_as_half((unsigned short)(0x6400 + half))));
      if (FORM == kFormFP16) {
        put(s - 1, *reinterpret_cast<const unsigned*>(&h));
      } else {   // |d| <= 16: exact in E4M3
        put(s - 1, (unsigned)__nv_cvt_halfraw2_to_fp8x2(*reinterpret_cast<const __half2_raw*>(&h),
                                                        __NV_SATFINITE, __NV_E4M3));
      }
    }
  }
}

// One operand of a slicing launch.
struct SliceOp {
  const double* X;
  int64_t ldx, strideX;
  int trans, rows, rows_pad, esign;
  int* e;                   // row exponents out (batch x rows_pad)
  uint8_t* out;             // slice planes
};

// Row exponents and slices of both operands of a product in one launch.  A cluster of
// `cl` CTAs takes 16 rows of op(A) (the first nblk_a clusters along x) or of op(B)^T,
// blockIdx.z the batch entry; each CTA has its share of the 64-wide tiles of K.  It
// brings the first `keep` of its tiles to shared memory (every load in flight at once),
// finds its share's largest magnitudes, the ranks exchange them through distributed
// shared memory, and then it slices the tiles it kept and, beyond those, the others read
// once more: S planes of rows_pad x K_pad elements, K contiguous, batch entry b at out + b
// S rows_pad K_pad, plane s at + s rows_pad K_pad elements.  Reads run along X's
// contiguous dimension, a warp writes a whole 128-byte line (FP8: 64) per plane.  With ek
// (the inner-index equilibration), element (i, k) counts as x 2^(esign ek[k]).
// Between HBM (8 bytes read, 14 written per element) and the integer work bound it: the
// digits of the 8-bit forms are bytes picked by permutes.  Measured, both operands: 4096^3
// 158 us (4.7 TB/s of those bytes), 196 us with 32 rows a CTA read twice and shifts for
// digits; 8192 x 4096 x 512 50 -> 35 us, 128 x 512 x 8192 73 -> 41, 1000 x 1537 x 777 27
// -> 18, 300^3 13.9 -> 9.8, 512 x 512 x 16384 FP8 153 -> 120 us.  Tiles kept: 4 at five
// CTAs an SM (with one tile ahead in place of three: 163 us at 4096^3, 172 with 2 kept, 160
// with 6 at four CTAs, but 36 and 128 us above).
constexpr int kSliceRows = 16, kSliceTile = kSliceRows * 65;   // doubles of a tile, rows padded
constexpr int kSliceKeep = 4;
template <int S, int FORM>
__global__ void __launch_bounds__(256, 5)
slice_kernel(const SliceOp a, const SliceOp b, int nblk_a, int K, int K_pad,
             const int* __restrict__ ek, int cl, int keep) {
  namespace cgrp = cooperative_groups;
  constexpr int kE = Form<FORM>::kElem, R = kSliceRows;
  extern __shared__ double xs[];
  __shared__ int mine[R], es[R];
  const int rank = blockIdx.x % cl, blk = blockIdx.x / cl;
  const bool on_b = blk >= nblk_a;
  const SliceOp o = on_b ? b : a;
  const int i0 = (on_b ? blk - nblk_a : blk) * R;
  const double* Xb = o.X + blockIdx.z * o.strideX;
  const int* ekb = ek ? ek + blockIdx.z * K_pad : nullptr;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int ntiles = K_pad / 64, per = (ntiles + cl - 1) / cl;
  const int t_lo = min(ntiles, rank * per), t_hi = min(ntiles, t_lo + per);
  const int t_keep = min(t_hi, t_lo + keep);
  // element u (of 4) of this thread in a tile: along X's contiguous dimension
  auto row_of = [&](int u) { return o.trans ? (tid >> 6) + 4 * u : tid & (R - 1); };
  auto col_of = [&](int u) { return o.trans ? tid & 63 : (tid >> 4) + 16 * u; };
  auto fetch = [&](int t, double* d) {
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int rr = row_of(u), c = col_of(u), i = i0 + rr, k = t * 64 + c;
      double* to = d + rr * 65 + c;
      if (i < o.rows && k < K) {
        const double* from = Xb + (o.trans ? k + (int64_t)i * o.ldx : i + (int64_t)k * o.ldx);
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(tc::smem_u32(to)), "l"(from) : "memory");
      } else {
        *to = 0.0;
      }
    }
  };
  for (int t = t_lo; t < t_keep; ++t) fetch(t, xs + (t - t_lo) * kSliceTile);
  // the row bound: the largest high word (its low bit set for a subnormal below 2^-1042),
  // or with the inner-index shifts the largest shifted exponent bound
  const int none = ekb ? INT_MIN : 0;
  auto take = [&](int& mx, double x, int k) {
    const int hi = __double2hiint(x) & 0x7FFFFFFF, nz = hi | (__double2loint(x) != 0);
    if (!ekb) mx = max(mx, nz);
    else if (nz != 0) mx = max(mx, exp_bound(nz) + o.esign * ekb[k]);
  };
  if (tid < R) mine[tid] = none;
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncthreads();
  {
    int mx = none;   // 16 threads per row
    for (int t = t_lo; t < t_keep; ++t) {
      const double* d = xs + (t - t_lo) * kSliceTile + (tid >> 4) * 65;
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int c = (tid & 15) + 16 * u;
        if (t * 64 + c < K) take(mx, d[c], t * 64 + c);
      }
    }
#pragma unroll
    for (int h = 8; h > 0; h >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, h));
    if ((tid & 15) == 0) atomicMax(&mine[tid >> 4], mx);
  }
  if (t_keep < t_hi) {
    int mx[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) mx[u] = none;
    for (int t = t_keep; t < t_hi; t += 2) {
      double v[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int i = i0 + row_of(u & 3), k = (t + (u >> 2)) * 64 + col_of(u & 3);
        v[u] = i < o.rows && k < K && t + (u >> 2) < t_hi
                   ? Xb[o.trans ? k + (int64_t)i * o.ldx : i + (int64_t)k * o.ldx] : 0.0;
      }
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int k = (t + (u >> 2)) * 64 + col_of(u & 3);
        if (k < K && t + (u >> 2) < t_hi) take(mx[u & 3], v[u], k);
      }
    }
    if (o.trans) {
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int w = __reduce_max_sync(0xffffffffu, mx[u]);
        if (lane == 0) atomicMax(&mine[row_of(u)], w);
      }
    } else {
      atomicMax(&mine[tid & (R - 1)], max(max(mx[0], mx[1]), max(mx[2], mx[3])));
    }
  }
  cgrp::cluster_group cluster = cgrp::this_cluster();
  if (cl > 1) cluster.sync();
  else __syncthreads();
  if (tid < R) {
    int mx = mine[tid];
    for (int q = 0; q < cl; ++q)
      if (q != rank) mx = max(mx, cluster.map_shared_rank(mine, q)[tid]);
    es[tid] = ekb ? (mx == INT_MIN ? 0 : mx) : (mx == 0 ? 0 : exp_bound(mx));
    if (rank == 0 && i0 + tid < o.rows_pad) o.e[blockIdx.z * o.rows_pad + i0 + tid] = es[tid];
  }
  if (cl > 1) cluster.sync();   // no rank leaves while another reads its maxima
  else __syncthreads();
  const size_t plane = (size_t)o.rows_pad * K_pad * kE;
  uint8_t* ob = o.out + (size_t)blockIdx.z * S * plane + (size_t)i0 * K_pad * kE;
  // rows beyond the operand are zero: their digits are too
  auto cut = [&](int t, const double* d) {
    const int k = t * 64 + 2 * lane;                // this thread's two K entries
    const int s0 = ekb ? o.esign * ekb[k] : 0, s1 = ekb ? o.esign * ekb[k + 1] : 0;
#pragma unroll
    for (int q = 0; q < R / 8; ++q) {
      const int rr = warp + 8 * q;
      const double* x = d + rr * 65 + 2 * lane;
      const unsigned at = (unsigned)(rr * K_pad + k) * kE;
      slice_pair<S, FORM>(x[0], x[1], es[rr] - s0, es[rr] - s1, [&](int s, unsigned pair) {
        uint8_t* w = ob + s * plane + at;
        if (kE == 2) *reinterpret_cast<unsigned*>(w) = pair;
        else *reinterpret_cast<unsigned short*>(w) = (unsigned short)pair;
      });
    }
  };
  for (int t = t_lo; t < t_keep; ++t) cut(t, xs + (t - t_lo) * kSliceTile);
  if (t_keep < t_hi) {              // the others through the tiles' places, three ahead
    static_assert(kSliceKeep == 4, "the places are a ring of four");
    __syncthreads();
    auto ahead = [&](int t) {
      if (t < t_hi) fetch(t, xs + ((t - t_keep) & 3) * kSliceTile);
      asm volatile("cp.async.commit_group;" ::: "memory");
    };
    for (int u = 0; u < 3; ++u) ahead(t_keep + u);
    for (int t = t_keep; t < t_hi; ++t) {
      asm volatile("cp.async.wait_group 2;" ::: "memory");
      __syncthreads();              // tile t is there, the place of t - 1 is free
      ahead(t + 3);
      cut(t, xs + ((t - t_keep) & 3) * kSliceTile);
    }
  }
}

// ----------------------------------------------------------------- GEMM
// The epilogue's conversions: FP64 instructions, and conversions of int64 or float
// to or from FP64, go through the FP64 units (2 lanes a clock), conversions of 32
// bits and leading-zero counts through a unit of 16, and the epilogue of a product
// with a short K has as much work per output as its MMAs.  So an output takes one
// FP64 conversion (and the addend's FMA), the rest is plain integer work: an
// all-integer conversion measured slower (45 more instructions per output).

// An output's value from its level sums, iacc in units of 2^-48 and fm in units of
// 2^-(48 + LO), as x 2^k with |x| < 2^63: the LO bits below iacc's unit are kept while
// they fit.  The FP8 form's 17 do not above 2^45: there x takes nine of them (or none,
// above 2^54) and has 55 bits and more, two below the last of FP64's 53, so the lowest
// one may stand for all that is cut (set when any of it is) and x's own rounding to FP64
// is the only one.  WIDE: fm may exceed 2^30.
struct Fixed {
  long long x;
  int k;
};
// whether hi is outside [-2^b, 2^b)
template <int B>
__device__ __forceinline__ bool beyond(long long hi) {
  return (unsigned)((int)(hi >> 32) + (1 << (B - 32))) >> (B - 31) != 0;
}
template <int LO, bool WIDE>
__device__ __forceinline__ Fixed split_fixed(long long iacc, float fm) {
  constexpr int kLow = LO > 8 ? 9 : 8;   // low bits kept below 2^54
  long long hi;
  int lo;
  if (WIDE) {
    const int fh = __float2int_rn(fm * 0x1p-16f);
    const long long f = (long long)fh * 65536 + __float2int_rn(fmaf(-65536.f, (float)fh, fm));
    hi = iacc + (f >> LO);
    lo = (int)f & ((1 << LO) - 1);
  } else {
    const int f = __float2int_rn(fm);
    hi = iacc + (f >> LO);
    lo = f & ((1 << LO) - 1);
  }
  Fixed r;
  if (LO > 8 && !beyond<62 - LO>(hi)) {
    r.x = (hi << LO) | lo;
    r.k = -48 - LO;
    return r;
  }
  if (LO > 8) lo = (lo >> (LO - kLow)) | ((lo & ((1 << (LO - kLow)) - 1)) != 0);
  const bool big = beyond<54>(hi);
  r.x = big ? (hi | (lo != 0)) : ((hi << kLow) | lo);
  r.k = big ? -48 : -48 - kLow;
  return r;
}

// q times 2^e, rounded to nearest (ties to even), for results in the normal range: e20 is
// e in the exponent field's place; flip toggles the sign bit (its high word).
__device__ __forceinline__ double fixed_scaled(const Fixed& q, int e20, unsigned flip) {
  const double d = (double)q.x;
  const int h = __double2hiint(d);
  return __hiloint2double((int)((unsigned)(h + (h != 0 ? e20 + q.k * (1 << 20) : 0)) ^ flip),
                          __double2loint(d));
}

// x 2^k, any range: powers of two applied in steps that are exact until the last one
// rounds.
__device__ __forceinline__ double scale_steps(long long x, int k) {
  double d = (double)x;
  for (int i = 0; i < 3 && k != 0; ++i) {
    const int s = k < -1000 ? -1000 : (k > 1000 ? 1000 : k);
    d *= __longlong_as_double((long long)(1023 + s) << 52);
    k -= s;
  }
  return d;
}

struct SplitEpi {
  double* C;                // output (column-major), per-batch stride
  int64_t ldc, strideC;
  const double* Cin;
  int64_t ldcin, strideCin;
  double beta;
  double alpha[kGemmMaxBatch];
  const int* ea;            // row exponents, batch-major (batch x Mpad)
  const int* eb;            // column exponents (batch x Npad)
  int M, N, K, Mpad, Npad;
  int batch, reduce, swap;  // swap: the tile computes C^T (rows of the tile are columns of C)
  int c_upper;              // only tiles that touch the upper triangle (square, no swap)
  int b_lower;              // op(B)[k][j] = 0 for k < j: a tile starts at K block n0 / BK (no swap)
  int ks;                   // CTAs (one cluster) that share the K of a tile from full on; 1: none
  int full;                 // the tiles before it are computed by one CTA each
  int tiles_z, tiles;       // tiles of one batch entry (of the reduced product), in all
  int* err;
  int stall;                // test hook: the MMA issuer first waits on a barrier nothing completes
  long long stall_ns;
  int nan_rows;             // an exponent of 1026 marks a row or column with an Inf or NaN
                            // (off with the inner-index equilibration, whose shifted
                            // exponents may exceed it)
};

template <int BN, int S, int FORM>
struct SmemLayout {
  static constexpr int kAcc = Form<FORM>::top(S) + 1;   // level accumulators
  static constexpr int kBTile = BN * 128;          // bytes of one B slice tile (BN rows of 128 bytes)
  static constexpr int kBStage = S * kBTile;
  static constexpr int kATile = kTileM * 128;      // 16 KB
  static constexpr int kOffB = 0;
  static constexpr int kOffA = 2 * kBStage;
  static constexpr int kOffBar = kOffA + kARing * kATile;
  // B full / empty, A full / empty, level full / empty, done, never completed
  static constexpr int kBars = 4 + 2 * kARing + 2 * kAcc + 2;
  static constexpr int kBytes = kOffBar + kBars * 8 + 16;
  static constexpr int kAlloc = kBytes + 1024;     // slack for 1024-byte alignment
  static_assert(kAlloc <= 232448, "shared memory of one CTA");
  static_assert(kOffBar >= kTileM * BN * 12, "the K split's partial tile reuses the operand stages");
};

// Tiles of one batch entry, in groups of kGroupM tile rows (their A slices stay
// in L2 while B streams); with c_upper a group starts at the first tile column
// its first row needs.  Host and device count alike.
template <int BN>
__host__ __device__ inline int split_tiles_z(int num_m, int num_n, int c_upper) {
  if (!c_upper) return num_m * num_n;
  int total = 0;
  for (int first = 0; first < num_m; first += kGroupM) {
    const int gm = num_m - first < kGroupM ? num_m - first : kGroupM;
    total += gm * (num_n - first * (kTileM / BN));
  }
  return total;
}

struct TilePos {
  int z, tm, tn;
  bool valid;               // false: a tile below the diagonal inside a group
};
template <int BN>
__device__ __forceinline__ TilePos split_tile(const SplitEpi& p, int idx) {
  constexpr int R = kTileM / BN;
  const int num_m = p.Mpad / kTileM, num_n = p.Npad / BN;
  TilePos t;
  t.z = idx / p.tiles_z;
  idx -= t.z * p.tiles_z;
  int first = 0, n_first = 0;
  if (!p.c_upper) {
    first = idx / (kGroupM * num_n) * kGroupM;
    idx -= first * num_n;
  } else {
    for (;; first += kGroupM) {
      const int gm = num_m - first < kGroupM ? num_m - first : kGroupM;
      const int cnt = gm * (num_n - first * R);
      if (idx < cnt) break;
      idx -= cnt;
    }
    n_first = first * R;
  }
  const int gm = num_m - first < kGroupM ? num_m - first : kGroupM;
  t.tm = first + idx % gm;
  t.tn = n_first + idx / gm;
  t.valid = !p.c_upper || t.tn >= t.tm * R;
  return t;
}

// The output of one entry, any alpha and range: an Inf or NaN in the row of op(A)
// or the column of op(B) leaves digits that carry no value, so the output is NaN (as
// the FP64 product gives NaN or Inf there).
template <int FORM>
__device__ __forceinline__ double split_value(const SplitEpi& p, long long iacc, float fm, int ei,
                                              int ej, double al) {
  const Fixed q = split_fixed<Form<FORM>::kLo, true>(iacc, fm);
  const int e = ei + ej;
  double v = e >= -900 && e <= 900 ? fixed_scaled(q, e * (1 << 20), 0u) : scale_steps(q.x, q.k + e);
  if (p.nan_rows && (ei >= 1026 || ej >= 1026)) v = __longlong_as_double(0x7FF8000000000000ll);
  return v * al;
}

// Persistent: CTA b takes the tiles b, b + gridDim.x, ... (with a K split, the last or only
// tile is its cluster's).  Warp 0 streams slice tiles by TMA (two B stages of S tiles, a ring
// of A tiles), warp 1 issues the MMAs, sixteen warps drain the level accumulators;
// the three run ahead of one another across K blocks, chunks and tiles, so a
// tile's loads, its epilogue and the next tile's MMAs overlap.
//
// An MMA of M = 128, N = 64 reads 6 KB of operands in 32 clocks, more than shared
// memory's 128 B a clock.  The levels are neighbours in TMEM and the B slices
// neighbours in shared memory, so A slice s times the B slices t .. t+3 is one MMA
// of N = 256 that adds to the levels s+t .. s+t+3: A is read once for four pairs.
//
// With the slices taken in order s = 1..S, level L is complete when s = L - 1 has
// met t = 1: each level has its own full / empty barriers, so its drain runs under
// the pairs that follow and only the last levels of a chunk are waited for.
template <int BN, int S, int FORM>
__global__ void __launch_bounds__(kThreads, 1)
split_gemm_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                  const SplitEpi p) {
  using L = SmemLayout<BN, S, FORM>;
  using F = Form<FORM>;
  constexpr int kBK = form_bk<FORM>();
  constexpr int kChunkB = F::kChunkK / kBK;      // K blocks per chunk
  constexpr int kAcc = L::kAcc;
  constexpr int kTop = F::top(S);                // largest s + t (0-based) kept
  constexpr int kG = 256 / BN;                   // B slices per MMA
  static_assert(kAcc * BN <= 512, "the level accumulators must fit in TMEM");
  extern __shared__ uint8_t smem_raw[];
  uint8_t* sm = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint8_t* sB = sm + L::kOffB;
  uint8_t* sA = sm + L::kOffA;
  uint64_t* bar = (uint64_t*)(sm + L::kOffBar);
  uint64_t* bfull = bar;
  uint64_t* bempty = bar + 2;
  uint64_t* afull = bar + 4;
  uint64_t* aempty = afull + kARing;
  uint64_t* lfull = aempty + kARing;
  uint64_t* lempty = lfull + kAcc;
  uint64_t* tdone = lempty + kAcc;
  uint64_t* never = tdone + 1;         // initialised, never arrived at (test hook)
  uint32_t* tslot = (uint32_t*)(bar + L::kBars);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rank = blockIdx.x % p.ks;
  // the tile of this CTA's turn b, b + gridDim.x, ...: whole tiles, then its cluster's shared
  // one (full is a multiple of the grid where there are any); -1: none is left
  auto tile_at = [&](int turn) -> int {
    if (turn < p.full) return turn;
    if (p.ks == 1 || turn - p.full >= (int)gridDim.x) return -1;
    const int t = p.full + blockIdx.x / p.ks;
    return t < p.tiles ? t : -1;
  };
  const int nkb_all = (p.K + kBK - 1) / kBK;
  // this CTA's K blocks of a tile: [lo, hi), the structurally zero ones skipped
  auto k_range = [&](int tn, bool split, int* lo, int* hi) {
    *lo = p.b_lower ? tn * BN / kBK : 0;
    *hi = nkb_all;
    if (split) {
      const int per = (nkb_all - *lo + p.ks - 1) / p.ks;
      *lo += rank * per;
      *hi = min(*hi, *lo + per);
    }
  };
  int* err = p.err;

  if (threadIdx.x == 0) {
    tc::prefetch_tmap(&tmA);
    tc::prefetch_tmap(&tmB);
    for (int i = 0; i < 2; ++i) { tc::mbar_init(&bfull[i], 1); tc::mbar_init(&bempty[i], 1); }
    for (int i = 0; i < kARing; ++i) { tc::mbar_init(&afull[i], 1); tc::mbar_init(&aempty[i], 1); }
    for (int i = 0; i < kAcc; ++i) {
      tc::mbar_init(&lfull[i], 1);
      tc::mbar_init(&lempty[i], kEpiWarps);
    }
    tc::mbar_init(tdone, 1);
    tc::mbar_init(never, 1);
    tc::fence_barrier_init();
  }
  if (warp == 1) tc::tmem_alloc<512>(tslot);
  __syncthreads();
  tc::tc_fence_after();
  const uint32_t tmem = *tslot;

  // the K split's partial tile: exact sums, then float parts (column-major, 128 rows)
  long long* part_i = reinterpret_cast<long long*>(sm);
  float* part_f = reinterpret_cast<float*>(sm + (size_t)kTileM * BN * 8);

  if (warp == 0 && lane == 0) {
    // ---------------- TMA producer
    int kbg = 0, ia = 0;
    bool ok = true;
    int kbg_armed = 0, ia_armed = 0;   // loads issued (for the error-path drain)
    for (int turn = blockIdx.x, idx; ok && (idx = tile_at(turn)) >= 0; turn += gridDim.x) {
      const bool split = turn >= p.full;
      const TilePos t = split_tile<BN>(p, idx);
      if (!t.valid) continue;
      int kb_lo, kb_hi;
      k_range(t.tn, split, &kb_lo, &kb_hi);
      const int b_first = p.reduce ? 0 : t.z, b_last = p.reduce ? p.batch : t.z + 1;
      for (int b = b_first; b < b_last && ok; ++b) {
        const int arow = b * S * p.Mpad + t.tm * kTileM, brow = b * S * p.Npad + t.tn * BN;
        for (int kb = kb_lo; kb < kb_hi && ok; ++kb, ++kbg) {
          const int sb = kbg & 1;
          if (kbg >= 2 && !(ok = tc::mbar_wait(&bempty[sb], ((kbg >> 1) & 1) ^ 1, err))) break;
          tc::mbar_arrive_expect_tx(&bfull[sb], L::kBStage);
          kbg_armed = kbg + 1;
          for (int s = 0; s < S; ++s, ++ia) {
            // the first A tile ahead of the B stage's: the MMAs start with both
            const int sa = ia % kARing;
            if (ia >= kARing && !(ok = tc::mbar_wait(&aempty[sa], ((ia / kARing) & 1) ^ 1, err))) {
              // the armed B stage still gets the tiles it expects
              if (s == 0)
                for (int u = 0; u < S; ++u)
                  tc::tma_load_2d(sB + sb * L::kBStage + u * L::kBTile, &tmB, &bfull[sb], kb * kBK,
                                  brow + u * p.Npad);
              break;
            }
            tc::mbar_arrive_expect_tx(&afull[sa], L::kATile);
            ia_armed = ia + 1;
            tc::tma_load_2d(sA + sa * L::kATile, &tmA, &afull[sa], kb * kBK, arow + s * p.Mpad);
            if (s == 0)
              for (int u = 0; u < S; ++u)
                tc::tma_load_2d(sB + sb * L::kBStage + u * L::kBTile, &tmB, &bfull[sb], kb * kBK,
                                brow + u * p.Npad);
          }
        }
      }
    }
    if (*(volatile int*)err) {
      // something failed: wait (bounded) until every load this thread issued has landed
      for (int k = kbg_armed > 2 ? kbg_armed - 2 : 0; k < kbg_armed; ++k)
        tc::mbar_wait_drain(&bfull[k & 1], (k >> 1) & 1);
      for (int k = ia_armed > kARing ? ia_armed - kARing : 0; k < ia_armed; ++k)
        tc::mbar_wait_drain(&afull[k % kARing], (k / kARing) & 1);
    }
  } else if (warp == 1 && lane == 0) {
    // ---------------- MMA issuer
    // One thread issues 4 MMAs (32 bytes of K each) per A slice and group of B
    // slices: the descriptors are formed once and advanced by adding to their
    // start-address field (address >> 4, 14 bits; shared addresses stay below
    // 256 KB so no carry leaves the field).
    const uint32_t idesc0 = FORM == kFormFP8    ? tc::idesc_e4m3_f32(kTileM, 0)
                            : FORM == kFormFP16 ? tc::idesc_f16_f32(kTileM, 0)
                                                : tc::idesc_bf16_f32(kTileM, 0);
    const uint64_t adesc0 = tc::sdesc_k128(tc::smem_u32(sA));
    const uint64_t bdesc0 = tc::sdesc_k128(tc::smem_u32(sB));
    int kbg = 0, ia = 0, cg = 0;       // K blocks, A tiles and chunks so far
    bool ok = true;
    if (p.stall) {
      tc::mbar_stall(never, err, p.stall_ns);
      ok = false;
    }
    for (int turn = blockIdx.x, idx; ok && (idx = tile_at(turn)) >= 0; turn += gridDim.x) {
      const bool split = turn >= p.full;
      const TilePos t = split_tile<BN>(p, idx);
      if (!t.valid) continue;
      int kb_lo, kb_hi;
      k_range(t.tn, split, &kb_lo, &kb_hi);
      const int entries = p.reduce ? p.batch : 1;
      for (int b = 0; b < entries && ok; ++b) {
        for (int kb = kb_lo; kb < kb_hi && ok; ++kb, ++kbg) {
          const int in_chunk = (kb - kb_lo) % kChunkB;
          const bool first = in_chunk == 0;                       // the levels start anew
          const bool last = in_chunk == kChunkB - 1 || kb == kb_hi - 1;   // and are complete
          const int sb = kbg & 1;
          if (!(ok = tc::mbar_wait(&bfull[sb], (kbg >> 1) & 1, err))) break;
          const uint64_t bd = bdesc0 + (uint64_t)((sb * L::kBStage) >> 4);
          // level l drained by the epilogue after the previous chunk
          auto drained = [&](int l) {
            if (first && cg > 0 && ok) ok = tc::mbar_wait(&lempty[l], (cg - 1) & 1, err);
          };
#pragma unroll
          for (int s = 0; s < S; ++s) {
            const int sa = ia % kARing;
            if (!ok || !(ok = tc::mbar_wait(&afull[sa], (ia / kARing) & 1, err))) break;
            ++ia;
            tc::tc_fence_after();
            const uint64_t ad = adesc0 + (uint64_t)((sa * L::kATile) >> 4);
            // B slices [t0, t0 + nt) in one MMA per 32 bytes of K, levels s + t0 ..
            auto group = [&](int t0, int nt, bool fresh) {
              const uint32_t d = tmem + (s + t0) * BN;
              const uint64_t bt = bd + (uint64_t)((t0 * L::kBTile) >> 4);
              const uint32_t idesc = idesc0 | ((uint32_t)(nt * BN >> 3) << 17);
#pragma unroll
              for (int kk = 0; kk < kRowBytes / 32; ++kk) {
                const uint32_t accum = (fresh && kk == 0) ? 0u : 1u;
                if (FORM == kFormFP8) tc::mma_f8(d, ad + 2 * kk, bt + 2 * kk, idesc, accum);
                else tc::mma_bf16(d, ad + 2 * kk, bt + 2 * kk, idesc, accum);
              }
            };
            constexpr int kTs0 = S;              // t of s = 0
            const int ts = kTop - s + 1 < S ? kTop - s + 1 : S;
            if (s == 0) {
              // every level up to S - 1 is first touched here
#pragma unroll
              for (int t0 = 0; t0 < kTs0; t0 += kG) {
                const int nt = kTs0 - t0 < kG ? kTs0 - t0 : kG;
                if (first) {
#pragma unroll
                  for (int u = 0; u < nt; ++u) drained(t0 + u);
                  tc::tc_fence_after();
                }
                if (ok) group(t0, nt, first);
              }
            } else if (s == 1 && kTop == S) {
              // the pair (1, S - 1) opens level S: alone in a chunk's first block
              const int te = first ? ts - 1 : ts;
              for (int t0 = 0; t0 < te; t0 += kG) group(t0, te - t0 < kG ? te - t0 : kG, false);
              if (first) {
                drained(S);
                tc::tc_fence_after();
                if (ok) group(ts - 1, 1, true);
              }
            } else {
#pragma unroll
              for (int t0 = 0; t0 < ts; t0 += kG) group(t0, ts - t0 < kG ? ts - t0 : kG, false);
            }
            // level s is complete once the slices 0..s have met t = 0 (the last
            // slice also completes level S)
            if (last) {
              tc::mma_commit(&lfull[s]);
              if (s == S - 1 && kTop == S) tc::mma_commit(&lfull[kTop]);
            }
            tc::mma_commit(&aempty[sa]);
          }
          if (!ok) break;
          tc::mma_commit(&bempty[sb]);
          if (last) ++cg;
        }
      }
    }
    tc::mma_commit(tdone);   // arrives once every MMA issued above has completed
  } else if (warp >= 2) {
    // ---------------- epilogue: drain the levels into an int64 and a float
    // (level L of a chunk is an integer below 2^24 times 2^-bL; the int64 in units
    // of 2^-48 has room for 600 chunks of 192, 28 of 4096, at the digit bounds, and
    // gemm_split cuts a longer K into several products)
    constexpr int HALF = BN / (kEpiWarps / 4);     // columns of this warp
    constexpr bool kWide = F::kLo > 8;             // the float parts may exceed 2^30
    const int q = warp & 3;
    const int half = (warp - 2) >> 2;              // which column slice
    const uint32_t lane_off = (uint32_t)(q * 32) << 16;
    int cg = 0;
    bool ok = true;
    long long iacc[HALF];
    float fm[HALF];
#pragma unroll
    for (int j = 0; j < HALF; ++j) {
      iacc[j] = 0;
      fm[j] = 0.f;
    }
    for (int turn = blockIdx.x, idx; ok && (idx = tile_at(turn)) >= 0; turn += gridDim.x) {
      const bool split = turn >= p.full;
      const TilePos t = split_tile<BN>(p, idx);
      if (!t.valid) continue;
      int kb_lo, kb_hi;
      k_range(t.tn, split, &kb_lo, &kb_hi);
      const int nchunks = kb_hi > kb_lo ? (kb_hi - kb_lo + kChunkB - 1) / kChunkB : 0;
      const int b_first = p.reduce ? 0 : t.z, b_last = p.reduce ? p.batch : t.z + 1;
      const int row = t.tm * kTileM + q * 32 + lane;   // tile row
      const int n0 = t.tn * BN;
      double* C = p.C + (int64_t)(p.reduce ? 0 : t.z) * p.strideC;
      const double* Cin = p.Cin ? p.Cin + (int64_t)(p.reduce ? 0 : t.z) * p.strideCin : nullptr;
      for (int b = b_first; b < b_last && ok; ++b) {
        // the addends (beta C_in for the first entry, the running sum in C for the
        // later ones of a reduced batch): their lines are brought to L2 before the
        // chunks are waited for.  The strides are made opaque here: hoisted out of
        // the loops, the columns' addresses would spill the accumulators.
        const bool first = b == b_first;
        const bool addend = !split && (!first || (Cin && p.beta != 0.0));
        const int col0 = n0 + half * HALF;
        const int jn = row < (p.swap ? p.N : p.M) ? (p.swap ? p.M : p.N) - col0 : 0;   // columns left
        const int64_t ldi = first ? p.ldcin : p.ldc;
        const double* ip0 = (first ? Cin : C) + (p.swap ? col0 + row * ldi : row + col0 * ldi);
        int64_t st_i = p.swap ? 1 : ldi;
        asm volatile("" : "+l"(st_i));
        if (addend && (lane & 15) == 0 && !p.swap) {
          const double* ip = ip0;
#pragma unroll 4
          for (int j = 0; j < HALF; ++j, ip += st_i)
            if (j < jn) asm volatile("prefetch.global.L2 [%0];" ::"l"(ip));
        }
        // the exponents, under the wait for the MMAs (lane l holds column l's)
        const int ei = p.ea[b * p.Mpad + row];
        const int ej_lane = __ldg(p.eb + b * p.Npad + col0 + (lane & (HALF - 1)));
        for (int c = 0; c < nchunks && ok; ++c, ++cg) {
#pragma unroll
          for (int a = 0; a < kAcc; ++a) {
            if (!ok || !(ok = tc::mbar_wait(&lfull[a], cg & 1, err))) break;
            tc::tc_fence_after();
            uint32_t v[HALF];
            tc::tmem_ld<HALF>(tmem + lane_off + a * BN + half * HALF, v);
            tc::tmem_wait<HALF>(v);
            // the level is free as soon as it is in registers: the next chunk's MMAs wait
            // for this, not for the conversions
            tc::tc_fence_before();
            __syncwarp();
            if (lane == 0) tc::mbar_arrive(&lempty[a]);
            const int lv = a + 2;
#pragma unroll
            for (int j = 0; j < HALF; ++j) {
              const float x = __uint_as_float(v[j]);
              // one 32 x 32 + 64 bit multiply-add per element
              if (lv <= F::kIntTop) {
                const int sh = 48 - F::kBits * lv;
                if (sh < 31) iacc[j] += (long long)__float2int_rn(x) * (long long)(1 << (sh < 31 ? sh : 0));
                else iacc[j] += (long long)__float2int_rn(x) << sh;
              } else {
                fm[j] += x * __int_as_float((127 + 48 + F::kLo - F::kBits * lv) << 23);
              }
            }
          }
          // 32 chunks keep the float parts below 2^30: what lies above the int64's unit moves
          if (!kWide && (c & 31) == 31) {
#pragma unroll
            for (int j = 0; j < HALF; ++j) {
              const int f = __float2int_rn(fm[j]);
              iacc[j] += f >> F::kLo;
              fm[j] = (float)(f & ((1 << F::kLo) - 1));
            }
          }
        }
        if (!ok) break;
        if (split) break;         // the CTA's last tile: joined over the cluster below
        // end of a batch entry: scale, combine with the addend, write, reset.  The fast
        // loop's FP64 work is one conversion and the addend's FMA (the sign of alpha =
        // +-1 is a bit, the scale an exponent); another alpha, an Inf or NaN operand or
        // exponents from which a result could leave the normal range take the general
        // loop instead, decided before the first output: nothing of the sums is kept for
        // a second look.  4096 x 4096, C += A B, K = 64 / 128: 172 / 183 -> 141 / 148 us;
        // 8192 x 4096, K = 512: 768 -> 700 us (BF16); 4096^3 2.74 -> 2.67 ms.
        const double al = p.alpha[b], bt = first ? p.beta : 1.0;
        const int emin = __reduce_min_sync(0xffffffffu, ej_lane), emax = __reduce_max_sync(0xffffffffu, ej_lane);
        const bool slow = __any_sync(0xffffffffu, (al != 1.0 && al != -1.0) || ei + emin < -900 || ei + emax > 900 ||
                                                      (p.nan_rows && max(ei, emax) >= 1026));
        int64_t st_c = p.swap ? 1 : p.ldc;
        asm volatile("" : "+l"(st_c));
        double* cp = C + (p.swap ? col0 + row * p.ldc : row + col0 * p.ldc);
        const double* ip = ip0;
        if (slow) {
#pragma unroll 1
          for (int j = 0; j < HALF; ++j) {
            long long xi = 0;
            float xf = 0.f;
#pragma unroll
            for (int u = 0; u < HALF; ++u)
              if (u == j) {
                xi = iacc[u];
                xf = fm[u];
              }
            double w = split_value<FORM>(p, xi, xf, ei, __shfl_sync(0xffffffffu, ej_lane, j), al);
            if (j < jn) {
              if (addend) w = fma(bt, *ip, w);
              *cp = w;
            }
            ip += st_i;
            cp += st_c;
          }
        } else {
          const unsigned flip = al < 0.0 ? 0x80000000u : 0u;
          const int e0 = ei * (1 << 20);
          const int ejs = ej_lane * (1 << 20);
          constexpr int kAdd = 4;
#pragma unroll
          for (int j0 = 0; j0 < HALF; j0 += kAdd) {
            // the addends of four outputs first (a load after a store to C could alias
            // it, so a plain loop waits for each; eight at a time spill the sums)
            double add[kAdd], v[kAdd];
            if (addend) {
#pragma unroll
              for (int jj = 0; jj < kAdd; ++jj) {
                add[jj] = j0 + jj < jn ? *ip : 0.0;
                ip += st_i;
              }
            }
#pragma unroll
            for (int jj = 0; jj < kAdd; ++jj) {
              const Fixed q = split_fixed<F::kLo, kWide>(iacc[j0 + jj], fm[j0 + jj]);
              v[jj] = fixed_scaled(q, e0 + __shfl_sync(0xffffffffu, ejs, j0 + jj), flip);
            }
#pragma unroll
            for (int jj = 0; jj < kAdd; ++jj) {
              if (addend) v[jj] = fma(bt, add[jj], v[jj]);
              if (j0 + jj < jn) *cp = v[jj];
              cp += st_c;
            }
          }
        }
#pragma unroll
        for (int j = 0; j < HALF; ++j) {
          iacc[j] = 0;
          fm[j] = 0.f;
        }
      }
    }
    if (p.ks > 1) {
      // the operand stages are free: every MMA of this CTA (the last levels'
      // barrier) and every load it consumed are done
#pragma unroll
      for (int j = 0; j < HALF; ++j) {
        part_i[(half * HALF + j) * kTileM + q * 32 + lane] = iacc[j];
        part_f[(half * HALF + j) * kTileM + q * 32 + lane] = fm[j];
      }
    }
  }
  if (p.ks > 1) {
    // K split: the ranks' exact sums are added as integers and their float parts in
    // rank order; rank r writes the columns r BN / ks ..  Every thread of every rank
    // reaches both barriers, on the error path too.
    namespace cgrp = cooperative_groups;
    cgrp::cluster_group cluster = cgrp::this_cluster();
    __syncthreads();
    cluster.sync();
    const int shared = p.full + blockIdx.x / p.ks;
    if (warp >= 2 && shared < p.tiles) {
      const TilePos t = split_tile<BN>(p, shared);
      if (t.valid && !*(volatile int*)err) {
        const int e = threadIdx.x - 64, r = e % kTileM, row = t.tm * kTileM + r;
        const int share = BN / p.ks;
        double* C = p.C + (int64_t)t.z * p.strideC;
        const double* Cin = p.Cin ? p.Cin + (int64_t)t.z * p.strideCin : nullptr;
        const int ei = p.ea[t.z * p.Mpad + row];
        for (int jc = e / kTileM; jc < share; jc += 32 * kEpiWarps / kTileM) {
          const int j = rank * share + jc, col = t.tn * BN + j;
          const int ci = p.swap ? col : row, cj = p.swap ? row : col;
          if (row >= (p.swap ? p.N : p.M) || col >= (p.swap ? p.M : p.N)) continue;
          long long si = 0;
          float sf = 0.f;
          for (int k = 0; k < p.ks; ++k) {
            si += cluster.map_shared_rank(part_i, k)[j * kTileM + r];
            sf += cluster.map_shared_rank(part_f, k)[j * kTileM + r];
          }
          double v = split_value<FORM>(p, si, sf, ei, __ldg(p.eb + t.z * p.Npad + col), p.alpha[t.z]);
          if (Cin && p.beta != 0.0) v = fma(p.beta, Cin[ci + (int64_t)cj * p.ldcin], v);
          C[ci + (int64_t)cj * p.ldc] = v;
        }
      }
    }
    cluster.sync();   // no rank leaves while another reads its partial tile
  }
  tc::tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    if (lane == 0) tc::mbar_wait_drain(tdone, 0);
    __syncwarp();
    tc::tc_fence_after();
    tc::tmem_dealloc<512>(tmem);
  }
}

// ----------------------------------------------------------------- host side
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*,
                                  const cuuint64_t*, const cuuint64_t*, const cuuint32_t*,
                                  const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* f = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &f, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = (EncodeTiledFn)f;
  });
  return fn;
}

// 2-D map over a (rows x K_pad) matrix of the form's slice type, K contiguous,
// box of one 128-byte row (64 16-bit or 128 one-byte elements) x box_rows,
// 128-byte swizzle
template <int FORM>
bool make_map(CUtensorMap* m, const void* base, int64_t rows, int64_t K_pad, int box_rows) {
  EncodeTiledFn enc = encode_fn();
  if (!enc) return false;
  cuuint64_t dims[2] = {(cuuint64_t)K_pad, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)K_pad * Form<FORM>::kElem};
  cuuint32_t box[2] = {(cuuint32_t)form_bk<FORM>(), (cuuint32_t)box_rows};
  cuuint32_t es[2] = {1, 1};
  const CUtensorMapDataType ty = FORM == kFormFP8    ? CU_TENSOR_MAP_DATA_TYPE_UINT8
                                 : FORM == kFormFP16 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT16
                                                     : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16;
  return enc(m, ty, 2,
             const_cast<void*>(base), dims, strides, box, es,
             CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
             CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

int64_t round_up(int64_t x, int64_t m) { return (x + m - 1) / m * m; }

constexpr int kSplitSMs = 152;

// CTAs per tile: with too few tiles for the SMs, K is cut over a cluster while
// every rank keeps two chunks of K blocks (entries > 1: a reduced batch runs its
// entries one after another into the same output and is not cut).  Clusters of
// eight find room on about 128 SMs, of four on 144.
int split_ks(int tiles, int entries, int nkb, int chunk) {
  if (entries > 1) return 1;
  int best = 1;
  for (int ks = 2; ks <= 8; ks *= 2) {
    if (tiles * ks > (ks == 8 ? 128 : ks == 4 ? 144 : kSplitSMs) || nkb < ks * std::min(2 * chunk, 8)) break;
    best = ks;
  }
  return best;
}

template <int BN, int S, int FORM>
cudaError_t run_split(const GemmArgs& g, SplitWork& w, cudaStream_t st) {
  constexpr int kE = Form<FORM>::kElem;
  // orientation: put the larger output dimension on the 128-row tile side
  const bool swap = g.M < kTileM && g.N > g.M;
  const int M = swap ? g.N : g.M, N = swap ? g.M : g.N, K = g.K;
  const int Mpad = (int)round_up(M, kTileM), Npad = (int)round_up(N, BN),
            Kpad = (int)round_up(K, form_bk<FORM>());
  const int nb = g.batch;
  const size_t need_a = (size_t)nb * S * Mpad * Kpad, need_b = (size_t)nb * S * Npad * Kpad;
  const bool keq = g.k_equilibrate != 0;
  // the workspace counts 16-bit units
  if ((need_a + need_b) * kE > w.slice_elems * 2 ||
      (size_t)nb * (Mpad + Npad + (keq ? Kpad : 0)) > w.exp_elems)
    return cudaErrorMemoryAllocation;
  uint8_t* sa = static_cast<uint8_t*>(w.slices);
  uint8_t* sb = sa + need_a * kE;
  int* ea = w.exps;
  int* eb = w.exps + (size_t)nb * Mpad;
  int* ek = keq ? eb + (size_t)nb * Npad : nullptr;
  cudaError_t err;
  // op(A) rows: M x K.  With swap the tile's A side is op(B)^T (rows = columns of op(B)).
  //   op(A) row i, col k:   transA = 0: A[i + k lda]   transA = 1: A[k + i lda]
  //   op(B)^T row j, col k: transB = 0: B[k + j ldb]   transB = 1: B[j + k ldb]
  const double* Xa = swap ? g.B : g.A;
  const double* Xb = swap ? g.A : g.B;
  const int64_t lda = swap ? g.ldb : g.lda, ldb = swap ? g.lda : g.ldb;
  const int64_t sta = swap ? g.strideB : g.strideA, stb = swap ? g.strideA : g.strideB;
  const int ta = swap ? (g.transB ? 0 : 1) : g.transA;
  const int tb = swap ? g.transA : (g.transB ? 0 : 1);
  // inner-index equilibration: op(B)'s rows k are the columns of the (rows x K)
  // view of the tile's B side (A side when swapped); they are scaled by 2^-ek[k]
  // and op(A)'s columns by 2^+ek[k]
  const int sign_a = swap ? -1 : 1;
  if (keq) {
    ProfScope ps(kProfSlice, st, 0.0, 8.0 * nb * (double)N * K);
    const double* Xo = swap ? Xa : Xb;
    ps.blocks((const void*)col_exp_kernel, dim3(32, 8), 0, dim3((unsigned)(Kpad / 32), 1, nb));
    col_exp_kernel<<<dim3((unsigned)(Kpad / 32), 1, nb), dim3(32, 8), 0, st>>>(
        Xo, swap ? lda : ldb, swap ? sta : stb, swap ? ta : tb, swap ? M : N, K, ek, Kpad);
    if ((err = cudaGetLastError()) != cudaSuccess) return err;
  }
  {
    const SliceOp oa{Xa, lda, sta, ta, M, Mpad, sign_a, ea, sa};
    const SliceOp ob{Xb, ldb, stb, tb, N, Npad, -sign_a, eb, sb};
    // CTAs per 16 rows: about four per SM while each has a tile of K, and as many as keep
    // their share; one with many lanes in flight (clusters wait for room: 48 matrices took
    // 117.0 ms with up to eight, 112.9 with two, 111.8 with one)
    const int nblk = (Mpad + Npad) / kSliceRows, ntiles = Kpad / 64;
    int cl = 1;
    while (cl < (w.throughput ? 1 : 8) && ntiles >= 2 * cl &&
           ((int64_t)nblk * nb * cl < 4 * kSplitSMs || ntiles > kSliceKeep * cl))
      cl *= 2;
    const int per = (ntiles + cl - 1) / cl, keep = std::min(per, kSliceKeep);
    const int smem = keep * kSliceTile * (int)sizeof(double);
    const auto slice = slice_kernel<S, FORM>;
    if ((err = smem_attr_once((const void*)slice, kSliceKeep * kSliceTile * (int)sizeof(double))) != cudaSuccess)
      return err;
    ProfScope ps(kProfSlice, st, 0.0, (16.0 + (double)kE * S) * nb * (double)(Mpad + Npad) * Kpad);
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)(nblk * cl), 1, nb);
    cfg.blockDim = dim3(256);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = cl;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = cl > 1 ? 1 : 0;
    ps.blocks((const void*)slice, dim3(256), smem, cfg.gridDim);
    const int* ekc = ek;
    if ((err = cudaLaunchKernelEx(&cfg, slice, oa, ob, Mpad / kSliceRows, K, Kpad, ekc, cl, keep)) !=
        cudaSuccess)
      return err;
  }
  CUtensorMap mA, mB;
  if (!make_map<FORM>(&mA, sa, (int64_t)nb * S * Mpad, Kpad, kTileM) ||
      !make_map<FORM>(&mB, sb, (int64_t)nb * S * Npad, Kpad, BN))
    return cudaErrorInvalidValue;
  SplitEpi p{};
  p.C = g.Cout; p.ldc = g.ldcout; p.strideC = g.strideCout;
  p.Cin = g.Cin; p.ldcin = g.ldcin; p.strideCin = g.strideCin; p.beta = g.beta;
  for (int b = 0; b < kGemmMaxBatch; ++b) p.alpha[b] = g.alpha[b];
  p.ea = ea; p.eb = eb;
  p.M = g.M; p.N = g.N; p.K = K; p.Mpad = Mpad; p.Npad = Npad;
  p.batch = nb; p.reduce = g.reduce; p.swap = swap ? 1 : 0;
  // structural zeros: c_upper is square (never swapped); b_lower's op(B) is the
  // tile's B side unless swapped
  p.c_upper = g.c_upper && !swap && g.M == g.N;
  p.b_lower = g.b_lower && !swap;
  const int nz = g.reduce ? 1 : nb;
  p.tiles_z = split_tiles_z<BN>(Mpad / kTileM, Npad / BN, p.c_upper);
  p.tiles = p.tiles_z * nz;
  p.ks = split_ks(p.tiles, g.reduce ? nb : 1, Kpad / form_bk<FORM>(), Form<FORM>::kChunkK / form_bk<FORM>());
  p.full = p.ks > 1 ? 0 : p.tiles;
  int ctas = p.ks > 1 ? p.tiles * p.ks : std::min(p.tiles, kSplitSMs);
  // A last wave that fills at most half the SMs has its tiles' K shared by pairs of CTAs:
  // 4096^3 BF16 (13 waves and 72 tiles) 2656 -> 2591 us, 2000^3 FP16 360 -> 324, 1300 x 1000
  // x 1000 110 -> 90, x 256 40 -> 38.5 us.  Below four blocks of K the join costs what it
  // saves; with many lanes in flight other kernels fill the SMs.
  const int tail = p.tiles % kSplitSMs;
  if (p.ks == 1 && !g.reduce && !w.throughput && p.tiles > kSplitSMs && tail > 0 && 2 * tail <= kSplitSMs &&
      Kpad / form_bk<FORM>() >= 4) {
    p.ks = 2;
    p.full = p.tiles - tail;
    ctas = kSplitSMs;
  }
  p.err = w.err;
  p.stall = w.stall;
  p.stall_ns = w.stall_ns;
  p.nan_rows = keq ? 0 : 1;
  using L = SmemLayout<BN, S, FORM>;
  const auto kernel = split_gemm_kernel<BN, S, FORM>;
  if ((err = smem_attr_once((const void*)kernel, L::kAlloc)) != cudaSuccess) return err;
  const dim3 grid((unsigned)ctas);
  ProfScope ps(kProfSplitGemm, st, gemm_flops(g), 0.0);
  ps.blocks((const void*)kernel, dim3(kThreads), L::kAlloc, grid);
  if (p.ks == 1) {
    kernel<<<grid, kThreads, L::kAlloc, st>>>(mA, mB, p);
    return cudaGetLastError();
  }
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = L::kAlloc;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = p.ks;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, mA, mB, p);
}

}  // namespace

cudaError_t gemm_split(const GemmArgs& g, SplitWork& w, cudaStream_t st) {
  if (g.M <= 0 || g.N <= 0 || g.batch <= 0) return cudaSuccess;
  if (g.K <= 0 || g.batch > kGemmMaxBatch) return gemm_f64(g, st);
  // The int64 that holds an output's exact level sums has room for a bounded
  // number of K-chunks at the digit bounds (8-bit digits: 2^53.6 per 192-chunk,
  // FP8: 2^58.1 per 4096-chunk); a longer K runs as consecutive products whose
  // partial results are added in FP64.
  const int64_t kmax = 28 * 4096;
  if (g.K > kmax) {
    for (int64_t k0 = 0; k0 < g.K; k0 += kmax) {
      GemmArgs h = g;
      h.K = (int)std::min<int64_t>(kmax, g.K - k0);
      h.A = g.A + (g.transA ? k0 : k0 * g.lda);   // op(A) columns k0..
      h.B = g.B + (g.transB ? k0 * g.ldb : k0);   // op(B) rows k0..
      if (k0 > 0) {
        h.Cin = g.Cout;
        h.ldcin = g.ldcout;
        h.strideCin = g.reduce ? 0 : g.strideCout;
        h.beta = 1.0;
      }
      const cudaError_t e = gemm_split(h, w, st);
      if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
  }
  // batch entries per launch that the slice workspace and the exponent array hold
  const size_t per = split_slice_elems(g.M, g.N, g.K, 1, w.slices_s, w.form);
  const size_t rows = split_exp_elems(g.M, g.N, g.K, 1, g.k_equilibrate, w.form);
  int gs = (int)std::min<size_t>(g.batch, w.slice_elems / std::max<size_t>(per, 1));
  gs = (int)std::min<size_t>((size_t)gs, w.exp_elems / std::max<size_t>(rows, 1));
  if (gs < 1) return cudaErrorMemoryAllocation;
  auto run = [&](const GemmArgs& h) {
    if (w.form == kFormFP8) return run_split<Form<kFormFP8>::kBN, 11, kFormFP8>(h, w, st);
    if (w.form == kFormFP16) return run_split<64, 7, kFormFP16>(h, w, st);
    return w.slices_s == 9 ? run_split<64, 7, kFormBF16>(h, w, st)
                           : run_split<64, 6, kFormBF16>(h, w, st);
  };
  if (gs >= g.batch) return run(g);
  for (int b0 = 0; b0 < g.batch; b0 += gs) {
    GemmArgs h = g;
    h.batch = std::min(gs, g.batch - b0);
    h.A = g.A + b0 * g.strideA;
    h.B = g.B + b0 * g.strideB;
    for (int b = 0; b < h.batch; ++b) h.alpha[b] = g.alpha[b0 + b];
    if (g.reduce) {
      if (b0 > 0) { h.Cin = g.Cout; h.ldcin = g.ldcout; h.strideCin = 0; h.beta = 1.0; }
    } else {
      h.Cout = g.Cout + b0 * g.strideCout;
      if (g.Cin) h.Cin = g.Cin + b0 * g.strideCin;
    }
    cudaError_t e = run(h);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

template <int BN, int S, int FORM>
static void prepare_form() {
  smem_attr_once((const void*)split_gemm_kernel<BN, S, FORM>, SmemLayout<BN, S, FORM>::kAlloc);
  smem_attr_once((const void*)slice_kernel<S, FORM>, kSliceKeep * kSliceTile * (int)sizeof(double));
}

void split_prepare() {
  prepare_form<64, 6, kFormBF16>();
  prepare_form<64, 7, kFormBF16>();
  prepare_form<64, 7, kFormFP16>();
  prepare_form<Form<kFormFP8>::kBN, 11, kFormFP8>();
  encode_fn();
}

thread_local SplitWork* t_split = nullptr;

void set_split_engine(SplitWork* w) { t_split = w; }
SplitWork* get_split_engine() { return t_split; }

// Estimated seconds on GB300 of one call on the FP64 pipe and on the split
// tensor-core path (slicing traffic + output traffic + slice-pair products +
// launch latency).
// Slice planes of a form: zolo_dgemm's `slices` of 9 and 8 six-bit digits (54 and 48
// bits) are held as 7 and 6 eight-bit ones, the FP16 form's 8 seven-bit ones as 7.
int split_planes(int slices, int form) {
  if (form == kFormFP8) return slices;
  return form == kFormFP16 || slices == 9 ? 7 : 6;
}

bool split_preferred(const GemmArgs& g, const SplitWork& w) { return split_time_ratio(g, w) < 1.0; }

namespace {
// The padded tile sides, slice bytes per element and slice-pair products (in
// 16-bit-MMA equivalents: FP8 runs at twice the rate) of one call in a form.
struct SplitShape {
  double ra, rb, kp, elem_bytes, pairs;
};
SplitShape split_shape(const GemmArgs& g, const SplitWork& w) {
  const bool swap = g.M < kTileM && g.N > g.M;
  const bool fp8 = w.form == kFormFP8;
  SplitShape sh;
  sh.ra = (double)round_up(swap ? g.N : g.M, kTileM);
  sh.rb = (double)round_up(swap ? g.M : g.N, fp8 ? Form<kFormFP8>::kBN : 64);
  sh.kp = (double)round_up(g.K, fp8 ? form_bk<kFormFP8>() : form_bk<kFormBF16>());
  sh.elem_bytes = fp8 ? 1.0 : 2.0;
  const double P = split_planes(w.slices_s, w.form);
  // slice pairs: s + t <= P + 2 (BF16, FP8), s + t <= P + 1 (FP16)
  const double pairs = w.form == kFormFP16 ? P * (P + 1) / 2 : P * (P + 1) / 2 + (P - 1);
  sh.pairs = fp8 ? pairs / 2 : pairs;
  return sh;
}
}  // namespace

double split_time_ratio(const GemmArgs& g, const SplitWork& w) {
  const SplitShape sh = split_shape(g, w);
  const double S = split_planes(w.slices_s, w.form);
  const double slice_bytes = g.batch * (8.0 + sh.elem_bytes * S) * (sh.ra + sh.rb) * sh.kp;
  const double out_bytes = (g.reduce ? 1 : g.batch) * 8.0 * g.M * (double)g.N * (g.beta != 0.0 ? 2 : 1);
  const double products = sh.pairs * 2.0 * sh.ra * sh.rb * sh.kp * g.batch;
  if (w.throughput) {
    // GPU-seconds of each path when other calls fill the rest of the chip: the
    // FP64 pipe at its measured 1.2 TFLOP/s, the slice-pair products at 1.7 PFLOP/s
    // of BF16 issue, the slicing and output traffic at 6 TB/s
    return ((slice_bytes + out_bytes) / 6e12 + products / 1.7e15) / (gemm_flops(g) / 1.2e12);
  }
  const double t64 = gemm_flops(g) / 0.9e12;
  const double tsplit = slice_bytes / 4e12 + out_bytes / 5e12 + products / 0.7e15 + 30e-6;
  return tsplit / t64;
}

// Exponents run_split writes: one per padded tile row and column of every batch
// entry, plus one per padded inner index with the equilibration.
size_t split_exp_elems(int64_t M, int64_t N, int64_t K, int batch, int k_equilibrate, int form) {
  const bool swap = M < kTileM && N > M;
  const bool fp8 = form == kFormFP8;
  const int64_t rows = swap ? N : M, cols = swap ? M : N;
  const int64_t bk = fp8 ? form_bk<kFormFP8>() : form_bk<kFormBF16>();
  return (size_t)batch * (size_t)(round_up(rows, kTileM) + round_up(cols, fp8 ? Form<kFormFP8>::kBN : 64) +
                                  (k_equilibrate ? round_up(K, bk) : 0));
}

// Slice planes of one call, in 16-bit units (two FP8 slices per unit).
size_t split_slice_elems(int64_t M, int64_t N, int64_t K, int batch, int S, int form) {
  const bool swap = M < kTileM && N > M;
  const bool fp8 = form == kFormFP8;
  const int64_t rows = swap ? N : M, cols = swap ? M : N;
  const int64_t bk = fp8 ? form_bk<kFormFP8>() : form_bk<kFormBF16>();
  const size_t elems = (size_t)batch * split_planes(S, form) *
                       (round_up(rows, kTileM) + round_up(cols, fp8 ? Form<kFormFP8>::kBN : 64)) *
                       round_up(K, bk);
  return fp8 ? (elems + 1) / 2 : elems;
}

}  // namespace zolo
