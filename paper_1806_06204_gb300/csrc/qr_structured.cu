// Structured Householder QR of the stacked matrix [X; sqrt(c) I] (Section 3.1,
// Eq. 12) and the explicit thin Q = [Q1; Q2] (the structured ORGQR).
//
// Layout: the stacked (m+n) x n matrix is stored densely, column-major with
// ld = m + n (top block rows 0..m-1, bottom block rows m..m+n-1).  The bottom
// block starts diagonal; Householder vector c (column c) is non-zero only on
// top rows c..m-1 and bottom rows 0..c, i.e. on the CONTIGUOUS stored rows
// c..m+c: m+1 entries instead of m+n-c (the paper's "at most m+1 nonzero
// elements").  A set of columns [c0, c0 + w) therefore lives in the row window
// [c0, c0 + m + w), and its compact-WY update (I - V T V^T) touches only that
// window: every step costs O((m + w) w n) whatever n is.
//
// Levels of blocking.  Panels of NB = 32 columns are factored by one kernel and applied
// at once only to the rest of their block of NBb = 128 columns.  The block's reflectors
// are then merged into one compact-WY factor T_b (from the Gram matrix V_b^T V_b,
// below) and applied with three GEMMs whose inner dimension is the block width.  On the
// FP64 pipe the block goes to all later columns.  On the tensor cores a product with an
// inner dimension of 128 is bound by its outputs (their epilogue and the trailing
// matrix's traffic) and the trailing matrix is sliced for every one, so blocks are
// applied within a super-block of 512 columns (from n = 2048), whose merged reflectors
// go to everything to its right: the trailing matrix is sliced, read and written once
// per 512 columns.  The explicit Q applies the same (super-)block reflectors in reverse
// order.  4096^2 at r = 8: 272 -> 242 ms; no gain at 256 columns for n = 512 .. 1024.  The
// products over a super-block use the 34-pair slices in both 16-bit forms (28 pairs
// would raise the FP16 form's backward error at 2048^2 from 5.6e-15 to 8.2e-15; so it
// falls to 3.1e-15); the FP8 form, more accurate than those, keeps 128-column blocks.
//
// Q2 (the bottom block of Q) stays exactly upper triangular: the explicit V
// holds exact zeros outside each reflector's support, so every product that the
// structure makes zero is an exact zero in floating point too.
#include <cooperative_groups.h>

#include <algorithm>
#include <atomic>
#include <cmath>

#include "fp64_scalar.cuh"
#include "zolo_internal.h"

namespace zolo {
namespace {

constexpr int kPanelCluster = 8;            // CTAs per shift in the global-memory panel
constexpr int64_t kClusterPanelMinRows = 512;

// Reduce-scatter of 32 per-lane partial sums across a warp: on return lane q
// holds the warp's total of value q.  Each step keeps the half of the values
// selected by one lane bit and adds the partner's copy of that half: 16 + 8 +
// 4 + 2 + 1 = 31 adds per lane, where one butterfly per value costs 5 x 32 (the
// FP64 adds, not the shuffles, bound the panel on this part).
__device__ __forceinline__ double warp_reduce_scatter32(double (&a)[32], int lane) {
#pragma unroll
  for (int h = 16; h >= 1; h >>= 1) {
    const bool up = (lane & h) != 0;
#pragma unroll
    for (int j = 0; j < h; ++j) {
      const double send = up ? a[j] : a[j + h];
      const double keep = up ? a[j + h] : a[j];
      a[j] = keep + __shfl_xor_sync(0xffffffffu, send, h);
    }
  }
  return a[0];
}

// Cluster form of the panel factorisation: CG CTAs per shift (one thread-block
// cluster), each owning a contiguous slice of the panel's row window.  Per
// column, every CTA reduces its rows' part of the norm (and the owner of the
// diagonal row contributes alpha), the partials are exchanged through
// distributed shared memory, every CTA forms the same beta/tau from the same
// ordered sum, scales its rows of v, and the same exchange gives the dot
// products for the update and for T.  Two hardware cluster barriers per
// column; the partial buffers alternate between columns so that no third
// barrier is needed before they are rewritten.  All rows a CTA reads or writes
// in W and V are its own, so the only cross-CTA traffic is the partials.
template <int NB, int CG, int KT>
__global__ void __cluster_dims__(CG, 1, 1) __launch_bounds__(KT)
qr_panel_cluster_kernel(double* W, int64_t strideW, int64_t ldw, int64_t m, int64_t c0, int nbp,
                        double* V, int64_t strideV, int64_t ldv, double* T, int64_t strideT,
                        int* status) {
  namespace cgrp = cooperative_groups;
  cgrp::cluster_group cluster = cgrp::this_cluster();
  constexpr int kT = KT, kWarps = kT / 32;
  __shared__ double part[2][NB + 2];        // [0, NB): dots, NB: norm^2, NB+1: alpha
  __shared__ double red[kWarps][NB + 2];
  __shared__ double dots[NB];
  __shared__ double cf[NB];                // -tau dots[q]: the update's coefficients
  __shared__ double Ts[NB][NB + 1];
  __shared__ double s_tau, s_scal, s_beta;

  const int rank = (int)cluster.block_rank();
  const int shift = blockIdx.x / CG;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  double* Wj = W + shift * strideW;
  double* Vp = V + shift * strideV + c0 * ldv;
  double* Tp = T + shift * strideT + (c0 / NB) * (int64_t)(NB * NB);
  const int64_t height = m + NB;
  const int64_t chunk = (height + CG - 1) / CG;
  const int64_t lo = c0 + rank * chunk;                   // my window rows [lo, hi)
  const int64_t hi = lo + chunk < c0 + height ? lo + chunk : c0 + height;

  for (int e = tid; e < NB * (NB + 1); e += kT) (&Ts[0][0])[e] = 0.0;

  for (int i = 0; i < nbp; ++i) {
    const int64_t c = c0 + i;
    const int buf = i & 1;
    double* col = Wj + c * ldw;
    const int64_t r0 = lo > c ? lo : c;                  // my part of the support [c, m + c]
    const int64_t r1 = hi < m + c + 1 ? hi : m + c + 1;
    // ---- 1. partial norm of the tail (rows > c) and alpha from the owner of row c
    double ss = 0.0;
    for (int64_t r = (r0 > c + 1 ? r0 : c + 1) + tid; r < r1; r += kT) {
      const double v = col[r];
      ss = fma(v, v, ss);
    }
    // the block's partials are summed by warp 0 (kWarps - 1 + 5 FP64 warp
    // instructions; a butterfly in every warp would take 5 per warp, and an FP64
    // instruction costs its unit a whole warp slot however few lanes it uses)
    double* flat = &red[0][0];
    flat[tid] = ss;
    __syncthreads();
    if (warp == 0) {
      double t = flat[lane];
#pragma unroll
      for (int w = 1; w < kWarps; ++w) t += flat[lane + 32 * w];
      for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
      if (lane == 0) {
        part[buf][NB] = t;
        part[buf][NB + 1] = (c >= lo && c < hi) ? col[c] : 0.0;
      }
    }
    cluster.sync();
    if (tid == 0) {
      double s = 0.0, alpha = 0.0;
      for (int rk = 0; rk < CG; ++rk) {
        const double* rp = cluster.map_shared_rank(&part[buf][0], rk);
        s += rp[NB];
        alpha += rp[NB + 1];
      }
      double beta, tau, scal;
      if (s == 0.0) {
        beta = alpha; tau = 0.0; scal = 0.0;
      } else {
        beta = -copysign(sqrt(fma(alpha, alpha, s)), alpha);
        tau = (beta - alpha) / beta;
        scal = 1.0 / (alpha - beta);
      }
      if (rank == 0 && (!isfinite(beta) || !isfinite(tau))) atomicOr(status + kStatNonFinite, 1);
      s_beta = beta; s_tau = tau; s_scal = scal;
    }
    __syncthreads();
    const double tau = s_tau, scal = s_scal;
    // ---- 2. my rows of v, and of the explicit reflector (zeros outside the support)
    double* Vcol = Vp + (int64_t)i * ldv;
    for (int64_t r = lo + tid; r < hi; r += kT) {
      double v;
      if (r < c || r > m + c) {
        v = 0.0;
      } else if (r == c) {
        v = 1.0;
      } else {
        v = col[r] * scal;
        col[r] = v;
      }
      Vcol[r - c0] = v;
    }
    __syncthreads();
    if (tid == 0 && c >= lo && c < hi) col[c] = s_beta;
    // ---- 3. partial dots of v with the later panel columns and the earlier reflectors
    double acc[NB];
#pragma unroll
    for (int q = 0; q < NB; ++q) acc[q] = 0.0;
    for (int64_t r = r0 + tid; r < r1; r += kT) {
      const double v = Vcol[r - c0];
#pragma unroll
      for (int q = 0; q < NB; ++q) {
        if (q < nbp && q != i) {
          const double o = q > i ? Wj[r + (c0 + q) * ldw] : Vp[(r - c0) + (int64_t)q * ldv];
          acc[q] = fma(v, o, acc[q]);
        }
      }
    }
    static_assert(NB == 32, "one dot product per lane");
    red[warp][lane] = warp_reduce_scatter32(acc, lane);
    __syncthreads();
    if (tid < NB) {
      double t = 0.0;
      for (int w = 0; w < kWarps; ++w) t += red[w][tid];
      part[buf][tid] = t;
    }
    cluster.sync();
    if (tid < NB) {
      double t = 0.0;
      for (int rk = 0; rk < CG; ++rk) t += cluster.map_shared_rank(&part[buf][0], rk)[tid];
      dots[tid] = t;
      cf[tid] = -tau * t;
    }
    __syncthreads();
    // ---- 4. my rows of the later panel columns: W[:, q] -= tau * dots[q] * v
    //         (the coefficients formed once above: the stores through pq may
    //         alias shared memory for the compiler, so a product written here
    //         would be redone for every row)
    for (int64_t r = r0 + tid; r < r1; r += kT) {
      const double v = Vcol[r - c0];
#pragma unroll
      for (int q = 0; q < NB; ++q) {
        if (q > i && q < nbp) {
          double* pq = Wj + r + (c0 + q) * ldw;
          *pq = fma(cf[q], v, *pq);
        }
      }
    }
    // ---- 5. T(0:i, i) = -tau T(0:i, 0:i) V^T v_i (same in every CTA)
    if (tid < i) {
      double t = 0.0;
      for (int pc = tid; pc < i; ++pc) t = fma(Ts[tid][pc], dots[pc], t);
      Ts[tid][i] = -tau * t;
    }
    if (tid == 0) Ts[i][i] = tau;
    __syncthreads();
  }
  if (rank == 0)
    for (int e = tid; e < NB * NB; e += kT) Tp[e] = Ts[e % NB][e / NB];
  cluster.sync();   // no CTA leaves while another may still read its partials
}

// T_b of one block: its panel factors on the 32 x 32 diagonal blocks, zero
// elsewhere (leading dimension ld).  Grid (ceil(nbb^2 / 256), r).
__global__ void tb_init_kernel(const double* __restrict__ T, int64_t strideT, double* __restrict__ Tb,
                               int64_t strideTb, int ld, int panel0, int nbb) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= nbb * nbb) return;
  const int i = e % nbb, j = e / nbb;
  double v = 0.0;
  if (i / kQrNB == j / kQrNB)
    v = T[blockIdx.y * strideT + (int64_t)(panel0 + i / kQrNB) * kQrNB * kQrNB + (i % kQrNB) +
          (j % kQrNB) * kQrNB];
  Tb[blockIdx.y * strideTb + i + (int64_t)j * ld] = v;
}

// One merge level of the block factor: for each pair of neighbouring diagonal
// blocks [a, a+h) and [a+h, a+h+w) of T_b (already merged up to width h),
//     T_b[a:a+h, a+h:a+h+w] = -T_11 (V_1^T V_2) T_22,
// which makes (I - V_1 T_11 V_1^T)(I - V_2 T_22 V_2^T) = I - V T V^T.  One CTA
// per column j of the right block, per pair and per shift; thread i owns row i.
__global__ void __launch_bounds__(kQrBlock / 2)
tb_merge_kernel(const double* __restrict__ G, int64_t strideG, double* __restrict__ Tb,
                int64_t strideTb, int ld, int nbb, int h) {
  __shared__ double x[kQrBlock / 2];
  const int j = blockIdx.x, i = threadIdx.x;
  const int a = blockIdx.y * 2 * h, b0 = a + h;
  const int w = nbb - b0 < h ? nbb - b0 : h;
  if (w <= 0 || j >= w) return;
  const double* Gs = G + blockIdx.z * strideG;
  double* T = Tb + blockIdx.z * strideTb;
  if (i < h) {
    double t = 0.0;
    for (int k = 0; k <= j; ++k) t = fma(Gs[(a + i) + (int64_t)(b0 + k) * ld], T[(b0 + k) + (int64_t)(b0 + j) * ld], t);
    x[i] = t;
  }
  __syncthreads();
  if (i < h) {
    double t = 0.0;
    for (int k = i; k < h; ++k) t = fma(T[(a + i) + (int64_t)(a + k) * ld], x[k], t);
    T[(a + i) + (int64_t)(b0 + j) * ld] = -t;
  }
}

// ------------------------------------------------- register-resident panel
// The panel factorisation with the panel's rows held in registers: lane q of every
// warp owns column q, a warp owns rows, and the rows are dealt cyclically over NG =
// RANKS x WARPS x SUB groups (RANKS CTAs of one cluster, WARPS warps each, SUB groups
// per warp): group g holds the window's rows g, g + NG, g + 2 NG, ..., so the panel's
// diagonal rows are row 0 of groups 0..31 (static register indices).
//
// What bounds a panel is the chain of one column to the next: FP64 instructions (64
// clocks of a sub-partition's unit per warp, however few lanes are active) and the
// exchanges between them.  So a column costs one pass, one reduction and one
// exchange: the pass applies the previous reflector to a row, takes the row's new
// entry x of column i by a shuffle and adds x a_q to every column's sum, which gives
// x^T x and x^T a_q of the tail together (the lanes q < i, which hold finished
// reflectors, yield V^T v for T at no cost).  With the tail sums s_q and the pivot
// row's entries a_cq exchanged at once,
//     beta = -sign(alpha) sqrt(alpha^2 + s_i),  tau = (beta - alpha) / beta,
//     scal = 1 / (alpha - beta),   v^T a_q = a_cq + scal s_q,
// and the update a_q -= tau (v^T a_q) v is -tau scal (v^T a_q) x below the pivot: the
// reflectors stay unscaled until they are written.  Four warps, one on each FP64 unit,
// form the scalars; with eight the others wait for theirs (two warps on a unit took twice
// as long, 35 us a panel).  The four share the sum over the ranks.
// The groups' sums are added in a fixed tree (4 groups, then the 8 fours), the same
// for 8 CTAs x 4 warps x 1 group and for 1 CTA x 8 warps x 4 groups: the one-CTA form
// of a batch and the cluster form of a single call give the same bits.
// Measured, 32 columns of 256 / 1024 / 4096 / 8192 rows at r = 6: 98 / 125 / 231 / 375
// us, against 325 / 285 / 440 / 1480 us of a panel in shared memory (one CTA under 512
// rows, else eight; the global-memory one at 8192); 400 rows on one CTA 231 us.
template <int N>
__device__ __forceinline__ double tree_sum(const double (&v)[N]) {
  double t[N];
#pragma unroll
  for (int i = 0; i < N; ++i) t[i] = v[i];
#pragma unroll
  for (int h = 1; h < N; h *= 2)
#pragma unroll
    for (int i = 0; i + h < N; i += 2 * h) t[i] += t[i + h];
  return t[0];
}

template <int RANKS, int WARPS, int SUB, int KMAX>
__global__ void __launch_bounds__(WARPS * 32)
qr_panel_reg_kernel(double* W, int64_t strideW, int64_t ldw, int64_t m, int64_t c0, int nbp,
                    double* V, int64_t strideV, int64_t ldv, double* T, int64_t strideT,
                    int* status, int kr) {
  constexpr int NB = 32, NG = RANKS * WARPS * SUB;
  static_assert(NG >= NB, "the diagonal rows are row 0 of their groups");
  namespace cgrp = cooperative_groups;
  cgrp::cluster_group cluster = cgrp::this_cluster();
  constexpr int LW = 4;                // the warps that form the scalars, one per sub-partition
  static_assert(WARPS >= LW && (RANKS < LW || RANKS % LW == 0), "equal shares");
  __shared__ double red[2][WARPS][NB];
  __shared__ double part[2][RANKS][NB];
  __shared__ double quarter[LW][NB];
  __shared__ double piv[2][NB];
  __shared__ double next[2][NB], next_scalar[2];   // f and cf, beta and scal, for the other warps
  __shared__ double Gs[NB][NB + 1], Ts[NB][NB + 1], Ys[NB][NB + 1];
  __shared__ double taus[NB];
  const int rank = RANKS > 1 ? (int)cluster.block_rank() : 0;
  const int shift = blockIdx.x / RANKS;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int g0 = (rank * WARPS + warp) * SUB;          // this warp's groups g0 .. g0 + SUB - 1
  double* Wj = W + shift * strideW + c0 + (c0 + lane) * ldw;
  double* Vp = V + shift * strideV + (c0 + lane) * ldv;
  const int64_t H = m + NB;                            // window rows
  const int64_t rows = ldw - c0 < H ? ldw - c0 : H;    // those that exist in W

  double a[SUB][KMAX];
#pragma unroll
  for (int s = 0; s < SUB; ++s)
#pragma unroll
    for (int k = 0; k < KMAX; ++k) {
      const int64_t r = g0 + s + (int64_t)NG * k;
      a[s][k] = (k < kr && lane < nbp && r < rows) ? Wj[r] : 0.0;
    }
  // f: what the pivot row of the previous column adds to this lane's column; cf: the
  // factor of the rows below it; scal_q: the scale of this lane's own reflector
  double f = 0.0, cf = 0.0, scal_q = 0.0, beta = 0.0;
  for (int e = threadIdx.x; e < NB * (NB + 1); e += WARPS * 32) (&Ts[0][0])[e] = (&Gs[0][0])[e] = 0.0;
  // no rank writes to another's shared memory before that one runs
  if constexpr (RANKS > 1) cluster.sync();
  else __syncthreads();

  for (int i = 0; i < nbp; ++i) {
    const int buf = i & 1;
    double acc[SUB];
#pragma unroll
    for (int s = 0; s < SUB; ++s) {
      const int g = g0 + s;
      double t = 0.0;
      {
        double v = a[s][0];
        const double xo = __shfl_sync(0xffffffffu, v, i > 0 ? i - 1 : 0);
        if (i > 0) {
          if (g > i - 1) v = fma(cf, xo, v);
          else if (g == i - 1) v = lane == i - 1 ? beta : v + f;
          a[s][0] = v;
        }
        const double x = __shfl_sync(0xffffffffu, v, i);
        if (g > i) t = x * v;
        if (g == i) {   // the pivot row goes to every rank
          if constexpr (RANKS > 1) {
            for (int q = 0; q < RANKS; ++q) cluster.map_shared_rank(&piv[buf][0], q)[lane] = v;
          } else {
            piv[buf][lane] = v;
          }
        }
      }
#pragma unroll
      for (int k = 1; k < KMAX; ++k) {
        if (k < kr) {
          double v = a[s][k];
          const double xo = __shfl_sync(0xffffffffu, v, i > 0 ? i - 1 : 0);
          v = fma(cf, xo, v);
          a[s][k] = v;
          t = fma(__shfl_sync(0xffffffffu, v, i), v, t);
        }
      }
      acc[s] = t;
    }
    red[buf][warp][lane] = tree_sum(acc);
    __syncthreads();
    double total = 0.0;
    if (warp < LW) {
      double w[WARPS];
#pragma unroll
      for (int q = 0; q < WARPS; ++q) w[q] = red[buf][q][lane];
      total = tree_sum(w);
    }
    if constexpr (RANKS > 1) {
      constexpr int PER = RANKS < LW ? RANKS : RANKS / LW;
      if (warp < LW)
        for (int q = warp; q < RANKS; q += LW)
          cluster.map_shared_rank(&part[buf][rank][0], q)[lane] = total;
      cluster.sync();
      if (warp < LW) {
        double w[PER], x[LW];
#pragma unroll
        for (int q = 0; q < PER; ++q) w[q] = part[buf][RANKS < LW ? q : warp * PER + q][lane];
        total = tree_sum(w);
        if constexpr (RANKS >= LW) {
          quarter[warp][lane] = total;
          asm volatile("bar.sync 1, %0;" ::"n"(LW * 32) : "memory");
#pragma unroll
          for (int q = 0; q < LW; ++q) x[q] = quarter[q][lane];
          total = tree_sum(x);
        }
      }
    }
    double scal = 0.0;
    if (warp < LW) {
      const double pv = piv[buf][lane];
      const double alpha = __shfl_sync(0xffffffffu, pv, i), ss = __shfl_sync(0xffffffffu, total, i);
      double tau = 0.0;
      if (ss == 0.0) {
        beta = alpha;
      } else {
        const double n2 = fma(alpha, alpha, ss);
        double nrm, inv;
        if (n2 > 1e-280 && n2 < 1e280) {
          root_pair(n2, &nrm, &inv);
          beta = -copysign(nrm, alpha);
          tau = fma(fabs(alpha), inv, 1.0);   // (beta - alpha) / beta with beta = -sign(alpha) nrm
          scal = reciprocal(alpha - beta);
        } else {   // near the ends of the range, or not finite
          beta = -copysign(sqrt(n2), alpha);
          tau = (beta - alpha) / beta;
          scal = 1.0 / (alpha - beta);
        }
      }
      const double dot = fma(scal, total, pv);   // v^T a_q; unscaled x_q^T v for q < i
      f = lane > i ? -tau * dot : 0.0;
      cf = f * scal;
      if (rank == 0 && warp == 0) {
        if (lane < i) Gs[lane][i] = scal_q * dot;
        if (lane == i) {
          taus[i] = tau;
          if (!isfinite(beta) || !isfinite(tau)) atomicOr(status + kStatNonFinite, 1);
        }
      }
      if (WARPS > LW && warp == 0) {
        next[0][lane] = f;
        next[1][lane] = cf;
        if (lane == 0) {
          next_scalar[0] = beta;
          next_scalar[1] = scal;
        }
      }
    }
    if constexpr (WARPS > LW) {
      __syncthreads();
      if (warp >= LW) {
        f = next[0][lane];
        cf = next[1][lane];
        beta = next_scalar[0];
        scal = next_scalar[1];
      }
    }
    if (lane == i) scal_q = scal;
  }
  // ---- the explicit reflectors (unit diagonal, exact zeros above it) and R's rows
#pragma unroll
  for (int s = 0; s < SUB; ++s) {
    const int g = g0 + s;
    if (lane < nbp) {
      double v = a[s][0];
      if (g == nbp - 1 && lane == nbp - 1) v = beta;
      if (g < NB && g <= lane && g < rows) Wj[g] = v;
      if (g < H) Vp[g] = g < lane ? 0.0 : (g == lane ? 1.0 : scal_q * v);
#pragma unroll
      for (int k = 1; k < KMAX; ++k) {
        const int64_t r = g + (int64_t)NG * k;
        if (k < kr && r < H) Vp[r] = scal_q * a[s][k];
      }
    }
  }
  if (rank != 0) return;
  // ---- T: 8 x 8 diagonal blocks row by row (T_ij = -tau_j sum_p T_ip G_pj), then
  //      pairs merged as -T_11 (G_12 T_22), 8 -> 16 -> 32
  __syncthreads();
  if (warp == 0) {
    const int b0 = lane & 24;
    double t[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int c = b0 + j;
      const double tj = c < nbp ? taus[c] : 0.0;
      double sum = 0.0;
#pragma unroll
      for (int q = 0; q < 8; ++q)
        if (q < j && b0 + q >= lane) sum = fma(t[q], Gs[b0 + q][c], sum);
      t[j] = c == lane ? tj : (c > lane ? -tj * sum : 0.0);
      Ts[lane][c] = t[j];
    }
  }
  __syncthreads();
#pragma unroll
  for (int h = 8; h < NB; h *= 2) {
    const int outs = (NB / (2 * h)) * h * h;
    for (int e = threadIdx.x; e < outs; e += WARPS * 32) {
      const int pr = e / (h * h), x = e % (h * h), r = pr * 2 * h + x % h, c = pr * 2 * h + h + x / h;
      double y = 0.0;   // (G_12 T_22)(r, c)
#pragma unroll
      for (int q = 0; q < h; ++q) y = fma(Gs[r][pr * 2 * h + h + q], Ts[pr * 2 * h + h + q][c], y);
      Ys[r][c] = y;
    }
    __syncthreads();
    for (int e = threadIdx.x; e < outs; e += WARPS * 32) {
      const int pr = e / (h * h), x = e % (h * h), r = pr * 2 * h + x % h, c = pr * 2 * h + h + x / h;
      double y = 0.0;
#pragma unroll
      for (int q = 0; q < h; ++q) y = fma(Ts[r][pr * 2 * h + q], Ys[pr * 2 * h + q][c], y);
      Ts[r][c] = -y;
    }
    __syncthreads();
  }
  double* Tp = T + shift * strideT + (c0 / NB) * (int64_t)(NB * NB);
  for (int e = threadIdx.x; e < NB * NB; e += WARPS * 32) Tp[e] = Ts[e % NB][e / NB];
}

struct PanelArgs {
  double* W; int64_t strideW, ldw, m, c0; int nbp;
  double* V; int64_t strideV, ldv; double* T; int64_t strideT; int* status;
};

template <int RANKS, int WARPS, int SUB, int KMAX>
cudaError_t launch_panel_reg(const PanelArgs& p, int r, double flops, double bytes, cudaStream_t st) {
  const auto kernel = qr_panel_reg_kernel<RANKS, WARPS, SUB, KMAX>;
  constexpr int NG = RANKS * WARPS * SUB;
  const int kr = (int)((p.m + kQrNB + NG - 1) / NG);
  if (kr > KMAX) return cudaErrorInvalidValue;
  ProfScope ps(kProfPanel, st, flops, bytes);
  ps.blocks((const void*)kernel, dim3(WARPS * 32), 0, dim3(r * RANKS));
  if (RANKS == 1) {
    kernel<<<r, WARPS * 32, 0, st>>>(p.W, p.strideW, p.ldw, p.m, p.c0, p.nbp, p.V, p.strideV, p.ldv,
                                     p.T, p.strideT, p.status, kr);
    return cudaGetLastError();
  }
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(r * RANKS);
  cfg.blockDim = dim3(WARPS * 32);
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = RANKS;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, p.W, p.strideW, p.ldw, p.m, p.c0, p.nbp, p.V, p.strideV,
                            p.ldv, p.T, p.strideT, p.status, kr);
}

// The products the block reflectors' T factors and a panel's own update hang on: in
// FP64, or for the 16-bit forms on the tensor cores with the more accurate slices (the
// BF16 form's 34 pairs), where the router expects a gain.  4096^2 at r = 8: 31.0 -> 4.2
// ms of FP64 work for 5 ms of split products.  Error of a product over its Frobenius norm in
// units of 2^-53, digits against FP64, over reflectors of geometric, uniform and shifted
// spectra: V^T V 0.7 .. 1.3 and 1.3 .. 4.8 (K = 128 .. 2128), a panel's V^T C 0.8 .. 1.4 and
// 1.4 .. 3.2 (K = 332 .. 2532).  The FP8 form, whose decompositions' errors grew by 2 to 9%
// with these products in digits, keeps FP64.
SplitWork fine_engine(const SplitWork& w) {
  SplitWork f = w;
  f.form = kFormBF16;
  f.slices_s = 9;
  return f;
}
bool gemm_fine_splits(const GemmArgs& g) {
  const SplitWork* w = get_split_engine();
  return w && w->form != kFormFP8 && split_preferred(g, fine_engine(*w));
}
cudaError_t gemm_fine(const GemmArgs& g, cudaStream_t st) {
  SplitWork* w = get_split_engine();
  if (!gemm_fine_splits(g)) return gemm_f64(g, st);
  SplitWork f = fine_engine(*w);
  return gemm_split(g, f, st);
}

// C <- (I - V op(T) V^T) C for r shifts, on the row window of C, as
// W1 = V^T C, W2 = op(T) W1, C -= V W2 (transT = 1 applies Q^T, the
// factorisation's update; transT = 0 applies Q, the explicit-Q build).
cudaError_t apply_block(const QrBuffers& b, const double* Vw, int64_t ldv, const double* Tw,
                        int ldt, int64_t strideT, double* C, int64_t ldw, int64_t rows, int w,
                        int64_t ncols, int r, int transT, cudaStream_t st) {
  cudaError_t err;
  GemmArgs g;
  g.M = w; g.N = (int)ncols; g.K = (int)rows; g.transA = 1; g.transB = 0;
  g.A = Vw; g.lda = ldv; g.strideA = b.strideV;
  g.B = C; g.ldb = ldw; g.strideB = b.strideW;
  g.Cout = b.W1; g.ldcout = b.sb; g.strideCout = b.strideW1;
  g.batch = r;
  for (int j = 0; j < r; ++j) g.alpha[j] = 1.0;
  // over a super-block the later reflectors meet columns that the earlier ones have
  // not been taken off: the cancellation that follows wants the finer slices
  err = w <= kQrNB || w > kQrBlock ? gemm_fine(g, st) : gemm_any(g, st);
  if (err != cudaSuccess) return err;
  GemmArgs h = g;
  h.K = w; h.transA = transT;
  h.A = Tw; h.lda = ldt; h.strideA = strideT;
  h.B = b.W1; h.ldb = b.sb; h.strideB = b.strideW1;
  h.Cout = b.W2; h.ldcout = b.sb; h.strideCout = b.strideW2;
  // the rows of W1 decay like the singular values across the reflectors; over a
  // super-block one scale per column would cost the small ones their precision
  h.k_equilibrate = w > kQrBlock;
  if ((err = w > kQrBlock ? gemm_fine(h, st) : gemm_any(h, st)) != cudaSuccess) return err;
  GemmArgs u = g;
  u.M = (int)rows; u.N = (int)ncols; u.K = w; u.transA = 0; u.transB = 0;
  u.A = Vw; u.lda = ldv; u.strideA = b.strideV;
  u.B = b.W2; u.ldb = b.sb; u.strideB = b.strideW2;
  u.Cin = C; u.ldcin = ldw; u.strideCin = b.strideW; u.beta = 1.0;
  u.Cout = C; u.ldcout = ldw; u.strideCout = b.strideW;
  for (int j = 0; j < r; ++j) u.alpha[j] = -1.0;
  // the rows of W2 follow the trailing matrix, whose size decays across the
  // block's reflectors like the singular values: equilibrate them
  u.k_equilibrate = 1;
  return w > kQrBlock ? gemm_fine(u, st) : gemm_any(u, st);
}

// The factor of a super-block from its blocks' factors, merged pairwise (128 -> 256 ->
// 512): T_12 = -T_11 (V_1^T V_2) T_22, V^T V in one product (upper tiles).  The
// products read T in full: what lies below its diagonal blocks is zero.  (V_1^T V_2) T_22
// stays on the FP64 pipe: its sums are short, and the digits' error over its Frobenius norm
// is twice the FP64 one (1.6 .. 2.2 against 0.6 .. 1.1 in units of 2^-53), where the other two
// products' is below it (T_11 Y 1.6 .. 2.2 against 1.8 .. 2.6); 4096^2 at r = 8: 2 of 205 ms.
cudaError_t merge_super(const QrBuffers& b, const double* Vs, int64_t ldv, double* Ts, int ldt,
                        int64_t rows, int sw, int r, cudaStream_t st) {
  cudaError_t err;
  GemmArgs g;
  g.M = g.N = sw; g.K = (int)rows; g.transA = 1;
  g.A = g.B = Vs; g.lda = g.ldb = ldv; g.strideA = g.strideB = b.strideV;
  g.Cout = b.G; g.ldcout = ldt; g.strideCout = b.strideG;
  g.batch = r; g.c_upper = 1;
  for (int j = 0; j < r; ++j) g.alpha[j] = 1.0;
  if ((err = gemm_fine(g, st)) != cudaSuccess) return err;
  for (int h = kQrBlock; h < sw; h *= 2)
    for (int a = 0; a + h < sw; a += 2 * h) {
      const int w = sw - a - h < h ? sw - a - h : h;
      GemmArgs y;   // Y = (V_1^T V_2) T_22, into W2
      y.M = h; y.N = w; y.K = w;
      y.A = b.G + a + (int64_t)(a + h) * ldt; y.lda = ldt; y.strideA = b.strideG;
      y.B = Ts + (a + h) + (int64_t)(a + h) * ldt; y.ldb = ldt; y.strideB = b.strideTb;
      y.Cout = b.W2; y.ldcout = ldt; y.strideCout = b.strideW2;
      y.batch = r;
      for (int j = 0; j < r; ++j) y.alpha[j] = 1.0;
      if ((err = gemm_f64(y, st)) != cudaSuccess) return err;
      GemmArgs t = y;   // T_12 = -T_11 Y
      t.M = h; t.N = w; t.K = h;
      t.A = Ts + a + (int64_t)a * ldt; t.lda = ldt; t.strideA = b.strideTb;
      t.B = b.W2; t.ldb = ldt; t.strideB = b.strideW2;
      t.Cout = Ts + a + (int64_t)(a + h) * ldt; t.ldcout = ldt; t.strideCout = b.strideTb;
      for (int j = 0; j < r; ++j) t.alpha[j] = -1.0;
      if ((err = gemm_fine(t, st)) != cudaSuccess) return err;
    }
  return cudaSuccess;
}

}  // namespace

namespace {

// The register panel that serves m rows, or kRegNone: kReg<CTAs>x<rows a thread> with four
// warps a CTA, ...w... with eight.  Below 512 rows a single call takes a cluster of 8 CTAs
// and a batch one CTA (the same bits).  From there a single call takes 16 CTAs; seven
// clusters of 16 find room at once and eight of 12, so eight shifts take 12 (4096 rows:
// 275 us, 403 in two rounds of 16, 397 with the former 8 CTAs; 1024 rows 131 and 178 us).
// A thread's rows beyond those there are cost a predicate each (4096 rows at r <= 7: 231
// us with 33, 244 with 65), hence the steps of 16.  With many problems in flight (narrow)
// the fewest CTAs that hold the rows cost the GPU least: 96 problems of 1024 / 2048 / 4096
// rows take 0.77 / 1.12 / 2.54 ms, against 0.93 / 1.45 / 3.53 of panels in shared memory
// (600 rows: 0.51 against 0.47, but 0.28 against 0.47 ms for a few problems alone).
enum PanelKind { kRegNone, kReg1x17, kReg2x17, kReg4x33, kReg8x17, kReg8x97, kReg8w65, kReg12w17, kReg12w33,
                 kReg12w49, kReg12w65, kReg12w97, kReg16w17, kReg16w33, kReg16w49, kReg16w65, kReg16w97 };
// Clusters of 12 and 16 CTAs are beyond the portable size of 8 and a partition of the GPU
// may have no room for them: `most` is the largest there is, and without 12 the clusters of
// 8 serve what they hold.
PanelKind panel_kind(int64_t m, int r, bool narrow, int most) {
  const int64_t H = m + kQrNB;
  if (m < kClusterPanelMinRows) return narrow ? kReg1x17 : kReg8x17;
  if (narrow || most < 12) {
    if (narrow && H <= 64 * 17) return kReg2x17;
    if (narrow && H <= 64 * 33) return kReg4x33;
    if (H <= 32 * 97) return kReg8x97;
    if (H <= 64 * 65) return kReg8w65;
  }
  if (most >= 12 && (r > 7 || narrow || most < 16)) {
    if (H <= 96 * 17) return kReg12w17;
    if (H <= 96 * 33) return kReg12w33;
    if (H <= 96 * 49) return kReg12w49;
    if (H <= 96 * 65) return kReg12w65;
    if (H <= 96 * 97) return kReg12w97;
  }
  if (most >= 16) {
    if (H <= 128 * 17) return kReg16w17;
    if (H <= 128 * 33) return kReg16w33;
    if (H <= 128 * 49) return kReg16w49;
    if (H <= 128 * 65) return kReg16w65;
    if (H <= 128 * 97) return kReg16w97;
  }
  return kRegNone;
}

// Allows the kernel its cluster; whether there is room for one (an error of the query: no,
// and *asked stays false).
template <int RANKS, int KMAX>
bool allow_cluster(bool* asked) {
  const auto kernel = qr_panel_reg_kernel<RANKS, 8, 1, KMAX>;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(RANKS);
  cfg.blockDim = dim3(256);
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = RANKS;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  int clusters = 0;
  if (cudaFuncSetAttribute((const void*)kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) !=
          cudaSuccess ||
      cudaOccupancyMaxActiveClusters(&clusters, kernel, &cfg) != cudaSuccess) {
    cudaGetLastError();
    *asked = false;
  }
  return clusters > 0;
}
template <int RANKS>
bool allow_clusters(bool* asked) {
  return allow_cluster<RANKS, 17>(asked) && allow_cluster<RANKS, 33>(asked) && allow_cluster<RANKS, 49>(asked) &&
         allow_cluster<RANKS, 65>(asked) && allow_cluster<RANKS, 97>(asked);
}

thread_local int t_cluster_limit = 16;

// The largest of 16, 12 and 8 CTAs whose panel kernels the current device has room for,
// asked once per device.
int largest_cluster() {
  static std::atomic<uint64_t> done{0}, has12{0}, has16{0};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev >= 64) return 8;
  const uint64_t bit = 1ull << dev;
  if (!(done.load() & bit)) {
    bool asked = true;
    if (allow_clusters<12>(&asked)) has12.fetch_or(bit);
    if (allow_clusters<16>(&asked)) has16.fetch_or(bit);
    if (asked) done.fetch_or(bit);
  }
  return std::min(t_cluster_limit, has16.load() & bit ? 16 : has12.load() & bit ? 12 : 8);
}

cudaError_t launch_panel(PanelKind k, const PanelArgs& p, int r, double fl, double by, cudaStream_t st) {
  switch (k) {
    case kReg1x17: return launch_panel_reg<1, 8, 4, 17>(p, r, fl, by, st);
    case kReg2x17: return launch_panel_reg<2, 8, 4, 17>(p, r, fl, by, st);
    case kReg4x33: return launch_panel_reg<4, 8, 2, 33>(p, r, fl, by, st);
    case kReg8x17: return launch_panel_reg<8, 4, 1, 17>(p, r, fl, by, st);
    case kReg8x97: return launch_panel_reg<8, 4, 1, 97>(p, r, fl, by, st);
    case kReg8w65: return launch_panel_reg<8, 8, 1, 65>(p, r, fl, by, st);
    case kReg12w17: return launch_panel_reg<12, 8, 1, 17>(p, r, fl, by, st);
    case kReg12w33: return launch_panel_reg<12, 8, 1, 33>(p, r, fl, by, st);
    case kReg12w49: return launch_panel_reg<12, 8, 1, 49>(p, r, fl, by, st);
    case kReg12w65: return launch_panel_reg<12, 8, 1, 65>(p, r, fl, by, st);
    case kReg12w97: return launch_panel_reg<12, 8, 1, 97>(p, r, fl, by, st);
    case kReg16w17: return launch_panel_reg<16, 8, 1, 17>(p, r, fl, by, st);
    case kReg16w33: return launch_panel_reg<16, 8, 1, 33>(p, r, fl, by, st);
    case kReg16w49: return launch_panel_reg<16, 8, 1, 49>(p, r, fl, by, st);
    case kReg16w65: return launch_panel_reg<16, 8, 1, 65>(p, r, fl, by, st);
    case kReg16w97: return launch_panel_reg<16, 8, 1, 97>(p, r, fl, by, st);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace

void qr_prepare() { largest_cluster(); }

PanelClusterScope::PanelClusterScope(int limit) : prev(t_cluster_limit) {
  if (limit > 0) t_cluster_limit = limit;
}
PanelClusterScope::~PanelClusterScope() { t_cluster_limit = prev; }

int qr_super_width(int64_t n) { return n >= 2048 ? 512 : kQrBlock; }

cudaError_t structured_qr_q(const QrBuffers& b, int64_t m, int64_t n, int r, int* status,
                            cudaStream_t st, bool explicit_q, bool narrow_panels) {
  constexpr int NB = kQrNB, NBb = kQrBlock;
  const int64_t ldw = m + n;
  // On the tensor cores the blocks of a super-block are applied to its own columns
  // one by one and to everything to its right together (see the file's head).
  const SplitWork* eng = get_split_engine();
  const int SB = eng && eng->form != kFormFP8 ? b.sb : NBb;
  const int ldt = SB;
  const int64_t ldv = m + SB;
  cudaError_t err;
  // the register panel where there is one, else the global-memory cluster kernel
  const PanelKind reg = panel_kind(m, r, narrow_panels, largest_cluster());
  // every V entry outside the rows a panel writes must be an exact zero
  if ((err = cudaMemsetAsync(b.V, 0, sizeof(double) * r * b.strideV, st)) != cudaSuccess) return err;
  if (SB > NBb &&
      (err = cudaMemsetAsync(b.Tb, 0, sizeof(double) * r * b.strideTb, st)) != cudaSuccess)
    return err;
  // ---------------- factorisation (structured GEQRF)
  for (int64_t c0b = 0; c0b < n; c0b += NBb) {
    const int64_t s0 = c0b / SB * SB;                              // the super-block
    const int sw = (int)(n - s0 < SB ? n - s0 : SB);
    const int off = (int)(c0b - s0);
    const int nbb = (int)(n - c0b < NBb ? n - c0b : NBb);
    for (int p = 0; p * NB < nbb; ++p) {
      const int64_t c0 = c0b + (int64_t)p * NB;
      const int nbp = nbb - p * NB < NB ? nbb - p * NB : NB;
      // V rows are relative to the super-block: this panel's window starts there
      double* Vpan = b.V + off + (int64_t)p * NB;
      const double pf = 3.0 * r * (double)(m + 1) * nbp * nbp, pb = 16.0 * r * (double)(m + NB) * nbp;
      if (reg != kRegNone) {
        const PanelArgs pa{b.W, b.strideW, ldw, m, c0, nbp, Vpan, b.strideV, ldv, b.T, b.strideT, status};
        if ((err = launch_panel(reg, pa, r, pf, pb, st)) != cudaSuccess) return err;
      } else {
        ProfScope ps(kProfPanel, st, pf, pb);
        ps.blocks((const void*)qr_panel_cluster_kernel<NB, kPanelCluster, 512>, dim3(512), 0,
                  dim3(r * kPanelCluster));
        // 512 threads per CTA halve each thread's share of the rows on the serial chain
        // of every column
        qr_panel_cluster_kernel<NB, kPanelCluster, 512><<<r * kPanelCluster, 512, 0, st>>>(
            b.W, b.strideW, ldw, m, c0, nbp, Vpan, b.strideV, ldv, b.T, b.strideT, status);
      }
      if ((err = cudaGetLastError()) != cudaSuccess) return err;
      // the rest of this block's columns
      const int64_t nin = c0b + nbb - (c0 + nbp);
      if (nin > 0) {
        const double* Vp = Vpan + c0 * ldv;
        const double* Tp = b.T + (c0 / NB) * (int64_t)(NB * NB);
        if ((err = apply_block(b, Vp, ldv, Tp, NB, b.strideT, b.W + c0 + (c0 + nbp) * ldw, ldw,
                               m + nbp, nbp, nin, r, 1, st)) != cudaSuccess)
          return err;
      }
    }
    // ---- the block factor T_b: panel factors on the diagonal, merged pairwise
    const double* Vb = b.V + off + c0b * ldv;
    double* Ts = b.Tb + s0 / SB * (int64_t)ldt * ldt;              // the super-block's factor
    double* Tb = Ts + off + (int64_t)off * ldt;
    {
      ProfScope ps(kProfOther, st);
      ps.blocks((const void*)tb_init_kernel, dim3(256), 0, dim3((nbb * nbb + 255) / 256, r));
      tb_init_kernel<<<dim3((nbb * nbb + 255) / 256, r), 256, 0, st>>>(b.T, b.strideT, Tb,
                                                                      b.strideTb, ldt, (int)(c0b / NB), nbb);
    }
    if ((err = cudaGetLastError()) != cudaSuccess) return err;
    if (nbb > NB) {
      // G = V_b^T V_b for the merges (they read the blocks [0,32)x[32,64),
      // [64,96)x[96,128) and [0,64)x[64,128)): small next to the columns' norms, and
      // T_b carries its error into every update.  On the FP64 pipe those three blocks
      // alone; on the tensor cores one product.
      static_assert(kQrBlock == 4 * kQrNB, "the merge levels assume four panels per block");
      GemmArgs g;
      g.M = g.N = nbb; g.K = (int)(m + nbb); g.transA = 1;
      g.A = g.B = Vb; g.lda = g.ldb = ldv; g.strideA = g.strideB = b.strideV;
      g.Cout = b.G; g.ldcout = ldt; g.strideCout = b.strideG;
      g.batch = r; g.c_upper = 1;
      for (int j = 0; j < r; ++j) g.alpha[j] = 1.0;
      if (gemm_fine_splits(g)) {
        if ((err = gemm_fine(g, st)) != cudaSuccess) return err;
      } else {
        g.c_upper = 0;
        auto gram = [&](int i0, int j0, int mt, int nt, int inner) {
          GemmArgs q = g;
          q.M = mt; q.N = nt;
          q.A = Vb + i0 * ldv;
          q.B = Vb + j0 * ldv;
          q.Cout = b.G + i0 + j0 * ldt;
          q.inner = inner;
          q.innerA = q.innerB = 2 * NB * ldv; q.innerC = 2 * NB + 2 * NB * ldt;
          return gemm_f64(q, st);
        };
        const int n01 = nbb - NB < NB ? nbb - NB : NB, n23 = nbb - 3 * NB;
        // the two 32-wide pairs in one launch when both are whole
        if ((err = gram(0, NB, NB, n01, n23 >= NB ? 2 : 1)) != cudaSuccess) return err;
        if (n23 > 0 && n23 < NB && (err = gram(2 * NB, 3 * NB, NB, n23, 1)) != cudaSuccess) return err;
        if (nbb > 2 * NB && (err = gram(0, 2 * NB, 2 * NB, nbb - 2 * NB, 1)) != cudaSuccess) return err;
      }
      for (int h = NB; h < nbb; h *= 2) {
        const int pairs = (nbb + 2 * h - 1) / (2 * h);
        {
          ProfScope ps(kProfOther, st);
          ps.blocks((const void*)tb_merge_kernel, dim3(NBb / 2), 0, dim3(h, pairs, r));
          tb_merge_kernel<<<dim3(h, pairs, r), NBb / 2, 0, st>>>(b.G, b.strideG, Tb, b.strideTb,
                                                                 ldt, nbb, h);
        }
        if ((err = cudaGetLastError()) != cudaSuccess) return err;
      }
    }
    // ---- the rest of the super-block's columns, or (its last block) its merged
    //      factor and all later columns
    const int64_t nsup = s0 + sw - c0b - nbb;
    if (nsup > 0) {
      if ((err = apply_block(b, Vb, ldv, Tb, ldt, b.strideTb, b.W + c0b + (c0b + nbb) * ldw, ldw,
                             m + nbb, nbb, nsup, r, 1, st)) != cudaSuccess)
        return err;
      continue;
    }
    const double* Vs = b.V + s0 * ldv;
    if (sw > NBb && (err = merge_super(b, Vs, ldv, Ts, ldt, m + sw, sw, r, st)) != cudaSuccess)
      return err;
    const int64_t ntr = n - s0 - sw;
    if (ntr > 0 &&
        (err = apply_block(b, Vs, ldv, Ts, ldt, b.strideTb, b.W + s0 + (s0 + sw) * ldw, ldw,
                           m + sw, sw, ntr, r, 1, st)) != cudaSuccess)
      return err;
  }
  if (!explicit_q) return cudaSuccess;
  // ---------------- explicit Q (structured ORGQR), overwriting W
  if ((err = init_q_identity(b.W, b.strideW, m, n, r, st)) != cudaSuccess) return err;
  for (int64_t s0 = (n - 1) / SB * SB; s0 >= 0; s0 -= SB) {
    const int sw = (int)(n - s0 < SB ? n - s0 : SB);
    if ((err = apply_block(b, b.V + s0 * ldv, ldv, b.Tb + s0 / SB * (int64_t)ldt * ldt, ldt,
                           b.strideTb, b.W + s0 + s0 * ldw, ldw, m + sw, sw, n - s0, r, 0, st)) !=
        cudaSuccess)
      return err;
  }
  return cudaSuccess;
}

}  // namespace zolo
