// Eigendecomposition of H for Zolo-SVD (Algorithm 2, step 2; ELPA in the paper).
//
// H = R^T R (Cholesky, upper R).  One-sided Jacobi rotations from the right on
// X = R^T make its columns mutually orthogonal: X Z = W diag(s) with W
// orthonormal, so H = X X^T = W diag(s^2) W^T.  The eigenvectors are the
// normalised columns of the converged X and the eigenvalues are taken as the
// Rayleigh quotients w_i^T H w_i (the squared column norms carry the rounding
// of every rotation applied to the column).  On the geometric spectra of this
// workload two-sided Jacobi on H converges only linearly in the absolute
// off-diagonal norm; the Cholesky factor restores quadratic convergence.
//
// Mixed precision.  FP32 runs 58x faster than FP64 on this part, so the sweeps
// that only need to bring the columns close to orthogonal run in FP32 on a copy
// X32 = R^T with the rotations accumulated in Z32, as block Jacobi on 16-column
// blocks (one cooperative dataflow launch per sweep).  Z is then made
// orthonormal in FP64 (Cholesky QR), X = R^T Z is formed in FP64, and FP64
// sweeps (one cooperative dataflow launch per sweep, one CTA per column pair at
// a time) finish from cosines ~1e-4 in a few quadratically convergent sweeps.
// FP32 sweeps stop when fewer than n rotations (cosines above 8e-6) were needed
// in a sweep (25 sweeps at most): the FP64 sweeps start from cosines of about
// 1e-4 whatever the last FP32 sweeps do, since Z's FP32 rounding, times R^T,
// sets them.  The FP32 sweeps' Gram entries and the FP64 sweeps' FP32 cosines and angles
// are of the size of H's eigenvalues, so X is R^T times a power of two that puts the
// largest diagonal entry of H in [2^90, 2^92): their range then holds eigenvalues down to
// 1e-50 of the largest, whatever the matrix's own scale (V and the Rayleigh quotients do
// not see it).  FP64 sweeps stop when no pair has |x_p . x_q| > 8 eps ||x_p||
// ||x_q||, or after a sweep in which every cosine was below sqrt(n) eps (the
// rounding level of an n-term dot product): its rotations were of that size,
// so the next sweep would find the same rounding-level cosines again.  Pairs are
// rotated down to 2 eps all the same, at no cost in time: the cosines that the
// last sweeps leave alone are what V's orthogonality consists of.
#include <algorithm>
#include <cmath>
#include <cstdlib>
#include <cstring>
#include <vector>

#include <cooperative_groups.h>

#include "fp64_scalar.cuh"
#include "zolo_internal.h"

namespace zolo {
namespace {

constexpr int kJacThreads = 256;
constexpr double kEps = 2.220446049250313e-16;

__device__ __forceinline__ double warp_sum(double v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Per-column round counters of the FP64 sweep: acquire/release at GPU scope.
__device__ __forceinline__ int ld_acquire(const int* p) {
  int v;
  asm volatile("ld.acquire.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_release(int* p, int v) {
  asm volatile("st.release.gpu.global.b32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

__device__ __forceinline__ void add_release(int* p, int v) {
  asm volatile("red.release.gpu.global.add.s32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// Waits until *ver >= want, two seconds at most (by the global timer), giving up
// at once when another block has set the error flag; false (and *err set) on
// time-out.
__device__ bool wait_round(const int* ver, int want, int* err) {
  if (ld_acquire(ver) >= want) return true;
  uint64_t t0;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t0));
  for (unsigned k = 0;; ++k) {
    if (ld_acquire(ver) >= want) return true;
    if ((k & 63u) == 63u) {
      if (*(volatile int*)err) return false;
      uint64_t t;
      asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
      if (t - t0 > 2000000000ull) break;
    }
    if (k > 15u) __nanosleep(32);
  }
  atomicExch(err, 1);
  return false;
}

// One FP64 sweep (the n_even - 1 rounds of the round-robin ordering, n_even / 2
// column pairs each) in one cooperative launch, as a dataflow: pair (round k, i)
// is work item k * n_even / 2 + i, block b takes the items b, b + gridDim.x, ...
// in order, and an item starts as soon as the two items of round k - 1 that
// held its columns are done (per-column round counters, acquire / release),
// instead of after a launch boundary that waits for the whole round.  Every
// block is resident (cooperative launch) and takes its items in increasing
// order, and an item waits only for lower-numbered items, so the lowest
// unfinished item can always run.  Columns are read through L2 (__ldcg): this
// SM's L1 may hold a column from an earlier round.
//
// Per pair: the squared column norms are tracked in nrm2 (formed afresh at the
// start of every sweep): a rotation with t = tan(theta) changes them exactly to
// a - t g and b + t g, so only the cross product of the pair is formed.  The
// rotations are the scaled ("fast") form: column j is held as dsc[j] * x~_j, the
// cosine goes into the scales (dsc_p <- c dsc_p, dsc_q <- c dsc_q) and each
// stored column takes one FMA, x~_p -= t (dsc_q / dsc_p) x~_q and
// x~_q += t (dsc_p / dsc_q) x~_p: three FP64 operations per row and pair instead
// of five (the FP64 pipe is the bound).  Near convergence c = 1 - O(t^2), so the
// scales stay within rounding of 1 over a sweep; the caller folds them into the
// columns between sweeps.
//
// What bounds an item below n of a few thousand is its chain: wait, load, dot product,
// rotation, update, publish.  So the two columns stay in registers between the dot
// product and the update (RPT rows a thread; 0: too long, read again), the block has as
// many threads as the length warrants, the scale ratios are formed while the columns
// are in flight, and only what the update needs (t times the ratios) lies on the chain;
// cosine, norms and scales follow it.  An FP64 instruction occupies its sub-partition's
// FP64 unit for a whole warp slot (64 clocks) however few lanes are active, so the
// partial dot products are summed by one warp, which changes with the item.  A sweep
// (events): n = 256 1.12 ms (1.71 with the columns read twice by 256 threads and the
// whole rotation formed in one chain), n = 512 2.9 (3.3), n = 1024 7.0 (7.3); from n =
// 2048 the FP64 units bound it (3 n^3 / 2 FMA: 25.5 ms a sweep, 167 at 4096; 24.9 and 164).
// A rotation is made for cosines above tol and counted above 4 tol.
template <int NT, int RPT>
__global__ void __launch_bounds__(NT, RPT == 0 ? 1536 / NT : 1)
jacobi_sweep_kernel(double* X, int64_t ldx, int64_t m, int n_even, int n_real, double tol,
                    int* status, double* nrm2, double* dsc, int* ver, int* err, int stall,
                    long long stall_ns) {
  __shared__ double part[NT];
  __shared__ double s_al, s_be, s_t;
  __shared__ int s_rot, s_ok[2], never;
  const int npairs = n_even / 2;
  const int64_t items = (int64_t)(n_even - 1) * npairs;
  if (stall && blockIdx.x == 0) {
    // test hook of the error exit: item 0 first waits, bounded, on a flag that
    // nothing sets; the blocks whose items need its columns leave on the flag
    if (threadIdx.x == 0) {
      never = 0;
      long long t0;
      asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t0));
      for (;;) {
        if (*(volatile int*)&never) break;
        long long t;
        asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
        if (t - t0 > stall_ns) break;
        __nanosleep(256);
      }
      atomicExch(err, 1);
    }
    __syncthreads();
    return;
  }
  constexpr int kWarps = NT / 32;
  const int tid = threadIdx.x, l = tid & 31, warp = tid >> 5;
  for (int64_t it = blockIdx.x; it < items; it += gridDim.x) {
    const int round = (int)(it / npairs), i = (int)(it - (int64_t)round * npairs);
    auto elem = [&](int pos) { return pos == 0 ? 0 : 1 + (pos - 1 + round) % (n_even - 1); };
    int p = elem(i), q = elem(n_even - 1 - i);
    if (p > q) { const int t = p; p = q; q = t; }
    const bool real = q < n_real;      // the pair with the padding column is no work
    if (tid < 2)
      s_ok[tid] = !*(volatile int*)err && ((tid == 1 && !real) || wait_round(ver + (tid ? q : p), round, err));
    __syncthreads();
    if (!s_ok[0] || !s_ok[1]) return;
    if (real) {
      double* xp = X + p * ldx;
      double* xq = X + q * ldx;
      double u[RPT > 0 ? RPT : 1], v[RPT > 0 ? RPT : 1];
      double g = 0.0;
      const int lead = (int)(it % kWarps);   // the warp that forms the rotation
      double dp = 1.0, dq = 1.0, sa = 0.0, sb = 0.0;
      if (RPT > 0) {
#pragma unroll
        for (int k = 0; k < RPT; ++k) {
          const int r = tid + k * NT;
          u[k] = r < m ? __ldcg(xp + r) : 0.0;
          v[k] = r < m ? __ldcg(xq + r) : 0.0;
        }
      }
      if (warp == lead) {
        dp = __ldcg(dsc + p);
        dq = __ldcg(dsc + q);
        sa = __ldcg(nrm2 + p);
        sb = __ldcg(nrm2 + q);
      }
      if (RPT > 0) {
        double h = 0.0;
#pragma unroll
        for (int k = 0; k < RPT; ++k) {
          if (k & 1) h = fma(u[k], v[k], h);
          else g = fma(u[k], v[k], g);
        }
        if (RPT > 1) g += h;
      } else {
        for (int64_t r = tid; r < m; r += NT) g = fma(__ldcg(xp + r), __ldcg(xq + r), g);
      }
      part[tid] = g;
      // what does not need the dot product: the scales' product and ratios, and the
      // FP32 operands of the cosine test and of the angle's first approximation
      double dd = 1.0, r1 = 1.0, r2 = 1.0, sg = 0.0;
      float fa = 0.f, fb = 0.f, fd = 0.f;
      if (warp == lead) {
        dd = dp * dq;
        r1 = dq * reciprocal(dp);
        r2 = dp * reciprocal(dq);
        fa = (float)sa;
        fb = (float)sb;               // below float range: left as converged
        fd = (float)(sb - sa);
      }
      __syncthreads();
      if (warp == lead) {
        sg = part[l];
#pragma unroll
        for (int k = 1; k < kWarps; ++k) sg += part[l + 32 * k];
        sg = warp_sum(sg) * dd;                         // cross product of the true columns
        const float fg = (float)sg;
        const float cosv = (fa > 0.f && fb > 0.f) ? fabsf(fg) * rsqrtf(fa) * rsqrtf(fb) : 0.f;
        // (a cross product below FLT_MIN: left as converged)
        const int rot = fabsf(fg) >= 0x1p-126f && cosv > (float)tol ? (cosv > 4.f * (float)tol ? 2 : 1) : 0;
        const float zeta = __fdividef(0.5f * fd, fg), az = fabsf(zeta);
        const float z1 = fmaf(az, az, 1.f);
        const float tf = copysignf(az > 1e18f ? __fdividef(0.5f, az) : __fdividef(1.f, az + z1 * rsqrtf(z1)), zeta);
        // one Newton step of g (t^2 - 1) + (s_q - s_p) t = 0 in FP64: the pair's next
        // cosine is the angle's error times this one
        const double t0 = (double)tf;
        const double res = fma(sg, fma(t0, t0, -1.0), (sb - sa) * t0);
        const double t = t0 - (double)__fdividef((float)res, fmaf(2.f * fg, tf, fd));
        if (l == 0) {
          s_al = t * r1;
          s_be = t * r2;
          s_t = t;
          s_rot = rot;
          atomicMax(status + kStatJacobiMaxCos, __float_as_int(cosv));
        }
      }
      __syncthreads();
      if (s_rot) {
        const double al = s_al, be = s_be;
        if (RPT > 0) {
#pragma unroll
          for (int k = 0; k < RPT; ++k) {
            const int r = tid + k * NT;
            if (r < m) {
              xp[r] = fma(-al, v[k], u[k]);
              xq[r] = fma(be, u[k], v[k]);
            }
          }
        } else {
          for (int64_t r = tid; r < m; r += NT) {
            const double a = __ldcg(xp + r), c = __ldcg(xq + r);
            xp[r] = fma(-al, c, a);
            xq[r] = fma(be, a, c);
          }
        }
        if (warp == lead) {
          // c = (1 + t^2)^(-1/2) for the t actually applied, in FP64
          const double t = s_t, x = fma(t, t, 1.0);
          double root, c;
          root_pair(x, &root, &c);
          if (l == 0) {
            nrm2[p] = fma(-t, sg, sa);
            nrm2[q] = fma(t, sg, sb);
            dsc[p] = c * dp;
            dsc[q] = c * dq;
            if (s_rot == 2) atomicAdd(status + kStatJacobiRot, 1);
          }
        }
      }
    }
    // publish: the block barrier orders every thread's stores before the releases of
    // the columns' round counters (a release at GPU scope covers what happens before
    // it in the block), which the next pair's acquire pairs with
    __syncthreads();
    if (tid == 0) st_release(ver + p, round + 1);
    if (tid == 1 && real) st_release(ver + q, round + 1);
  }
}

__global__ void fill_kernel(double* d, int64_t n, double v) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) d[i] = v;
}

// One FP32 sweep of block Jacobi: the columns are grouped in blocks of kJB, the blocks
// paired by the round-robin ordering, and each block pair of a round is a work item of
// `split` CTAs (one cluster), each on its share of the rows: they form the Gram matrix G
// = C^T C of the pair's 2 kJB columns (partial sums exchanged through distributed shared
// memory and added in rank order, so every rank continues with the same bits), run one
// cyclic Jacobi sweep on G in shared memory (the rotation from the 2x2 Gram entries of a
// column pair is the one-sided rotation of those two columns; J^T G J keeps G current),
// and apply the accumulated rotation Q to their rows of the pair's columns of X32 and
// Z32.  A rotation is counted when |g_pq| > tol sqrt(g_pp g_qq).
//
// Latency bounds it below n of a few thousand (the flops of a 1024^2 sweep take 0.2 ms),
// so rows are shared until a CTA has 128, items start as soon as the previous items that
// held their two blocks are done (per-block counters, acquire / release, as the FP64
// sweep's) instead of after a grid barrier, and a step of the inner sweep is one phase:
// thread (t1, t2) owns the 2x2 block of G at the rows of rotation t1 and the columns of
// t2, forms both rotations itself, and writes to the other copy of G.
// A sweep (events): n = 256 0.35 ms (0.51 with two phases a step, a grid barrier a round
// and at most two CTAs a pair), n = 1024 2.1 (3.0), n = 2048 7.9 (8.9); from n = 3000 the
// products take over (26.6 and 25.4 ms, n = 4096 45.9 and 42.9).
constexpr int kJB = 16;                // columns per block
constexpr int kJW = 2 * kJB;           // columns of a block pair
// rows per staged chunk: 128, or 256 where a CTA has several; the chunk's leading
// dimension has 16-byte rows and no bank conflicts
constexpr int kJRows = 128;
template <int ROWS>
constexpr int jac32_smem() {
  return (kJW * (ROWS + 4) + 4 * kJW * kJW) * (int)sizeof(float);
}

template <int ROWS>
__global__ void __launch_bounds__(kJacThreads, 2)
jacobi32_block_sweep_kernel(float* X, float* Z, int64_t ld, int64_t m, int nb_even, int n_real,
                            float tol, int* status, int* ver, int* err, int stall,
                            long long stall_ns, int split, int vec) {
  static_assert(kJacThreads == 256 && kJW == 32 && (ROWS == 128 || ROWS == 256), "thread mapping below");
  constexpr int kJLd = ROWS + 4;
  constexpr int kCols = kJW * ROWS / kJacThreads;   // columns a thread loads
  namespace cgrp = cooperative_groups;
  cgrp::cluster_group cluster = cgrp::this_cluster();
  extern __shared__ __align__(16) float jac_smem[];
  float* Ct = jac_smem;                // chunk, column-major: Ct[j * kJLd + r]
  float* fold = jac_smem + kJW * kJLd; // four warps' partial Gram matrices
  __shared__ float Gb[2][kJW][kJW + 1];
  __shared__ __align__(16) float Q4[kJW][kJW];
  __shared__ float part[2][kJW * kJW];
  __shared__ int s_ok[2], s_alive[2], s_rot, never;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int npairs = nb_even / 2;
  const int rank = blockIdx.x % split, first = blockIdx.x / split, step_items = gridDim.x / split;
  const int64_t mh = ((m + split - 1) / split + 3) / 4 * 4;
  const int64_t row_lo = rank * mh < m ? rank * mh : m;
  const int64_t row_hi = row_lo + mh < m ? row_lo + mh : m;
  const bool single = row_hi - row_lo <= ROWS;
  if (tid == 0) s_rot = 0;
  int buf = 0;
  bool alive = true;
  if (stall && blockIdx.x == 0) {
    // test hook of the error exit: wait, bounded, on a flag that nothing sets
    if (tid == 0) {
      never = 0;
      long long t0;
      asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t0));
      for (;;) {
        if (*(volatile int*)&never) break;
        long long t;
        asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
        if (t - t0 > stall_ns) break;
        __nanosleep(256);
      }
      atomicExch(err, 1);
    }
    alive = false;
  }
  for (int64_t it = first; it < (int64_t)(nb_even - 1) * npairs; it += step_items, buf ^= 1) {
    const int round = (int)(it / npairs), pi = (int)(it - (int64_t)round * npairs);
    auto elem = [&](int pos) { return pos == 0 ? 0 : 1 + (pos - 1 + round) % (nb_even - 1); };
    int P = elem(pi), Qb = elem(nb_even - 1 - pi);
    if (P > Qb) { const int t = P; P = Qb; Qb = t; }
    auto col = [&](int j) { return j < kJB ? P * kJB + j : Qb * kJB + (j - kJB); };
    // both blocks' previous items done, by all their ranks
    if (tid < 2)
      s_ok[tid] = alive && !*(volatile int*)err && wait_round(ver + (tid ? Qb : P), split * round, err);
    __syncthreads();
    const bool ok = s_ok[0] && s_ok[1];
    // chunk loader: thread = row and half of the columns (256 rows: all); the next chunk is fetched into
    // registers while the current one is used (through L2: other SMs wrote it)
    const int lr = tid & (ROWS - 1), lj = tid / ROWS * kCols;
    float pf[kCols];
    auto fetch = [&](const float* M, int64_t r0) {
      const int64_t r = r0 + lr;
#pragma unroll
      for (int j = 0; j < kCols; ++j) {
        const int c = col(lj + j);
        pf[j] = (c < n_real && r < row_hi) ? __ldcg(M + (int64_t)c * ld + r) : 0.f;
      }
    };
    auto stage = [&]() {
#pragma unroll
      for (int j = 0; j < kCols; ++j) Ct[(lj + j) * kJLd + lr] = pf[j];
    };
    if (ok) {
      // ---- 1. Gram G = C^T C: 16 row groups; thread owns the 8x8 block (bi, bj) of G
      //         over the rows r = g (mod 16) of each chunk
      const int g = tid >> 4, t = tid & 15, bi = t >> 2, bj = t & 3;
      float acc[8][8];
#pragma unroll
      for (int a = 0; a < 8; ++a)
#pragma unroll
        for (int b = 0; b < 8; ++b) acc[a][b] = 0.f;
      fetch(X, row_lo);
      for (int64_t r0 = row_lo; r0 < row_hi; r0 += ROWS) {
        stage();
        __syncthreads();
        if (r0 + ROWS < row_hi) fetch(X, r0 + ROWS);
#pragma unroll 2
        for (int r = g; r < ROWS; r += 16) {
          float va[8], vb[8];
#pragma unroll
          for (int a = 0; a < 8; ++a) va[a] = Ct[(8 * bi + a) * kJLd + r];
#pragma unroll
          for (int b = 0; b < 8; ++b) vb[b] = Ct[(8 * bj + b) * kJLd + r];
#pragma unroll
          for (int a = 0; a < 8; ++a)
#pragma unroll
            for (int b = 0; b < 8; ++b) acc[a][b] = fmaf(va[a], vb[b], acc[a][b]);
        }
        __syncthreads();
      }
      // one chunk: X stays staged and Z is on its way during the inner sweep
      if (single) fetch(Z, row_lo);
      // groups 2w and 2w+1 share warp w (lanes l and l ^ 16): fold them, then the warps'
      // partials through shared memory, four at a time
#pragma unroll
      for (int a = 0; a < 8; ++a)
#pragma unroll
        for (int b = 0; b < 8; ++b) acc[a][b] += __shfl_xor_sync(0xffffffffu, acc[a][b], 16);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        if (lane < 16 && (warp >> 2) == h)
#pragma unroll
          for (int a = 0; a < 8; ++a)
#pragma unroll
            for (int b = 0; b < 8; ++b)
              fold[(warp & 3) * kJW * kJW + (8 * bi + a) * kJW + (8 * bj + b)] = acc[a][b];
        __syncthreads();
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int e = tid + kJacThreads * u;
          const float sum = (fold[e] + fold[kJW * kJW + e]) + (fold[2 * kJW * kJW + e] + fold[3 * kJW * kJW + e]);
          part[buf][e] = h ? part[buf][e] + sum : sum;
        }
        __syncthreads();
      }
    }
    if (tid == 0) s_alive[buf] = ok;
    if (split > 1) cluster.sync();   // the ranks' partial sums (and whether all go on)
    else __syncthreads();
    bool all = true;
    if (split == 1) all = ok;
    else for (int k = 0; k < split; ++k) all = all && cluster.map_shared_rank(s_alive, k)[buf] != 0;
    if (!all) break;                 // every rank of the cluster leaves here
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int e = tid + kJacThreads * u, i = e >> 5, jj = e & 31;
      float sum = 0.f;
      if (split == 1) sum = part[buf][e];
      else for (int k = 0; k < split; ++k) sum += cluster.map_shared_rank(&part[0][0], k)[buf * kJW * kJW + e];
      Gb[0][i][jj] = sum;
      Q4[i][jj] = i == jj ? 1.f : 0.f;
    }
    __syncthreads();
    // ---- 2. cyclic Jacobi on G (round-robin over the 32 indices, 16 disjoint
    //         rotations per step); Q accumulates the rotations
    int nrot = 0;
    {
      const int t1 = tid >> 4, t2 = tid & 15;
      for (int step = 0; step < kJW - 1; ++step) {
        float (*G)[kJW + 1] = Gb[step & 1];
        float (*Gn)[kJW + 1] = Gb[(step & 1) ^ 1];
        auto pair = [&](int k, int* a, int* b) {
          auto e2 = [&](int pos) { return pos == 0 ? 0 : 1 + (pos - 1 + step) % (kJW - 1); };
          const int x = e2(k), y = e2(kJW - 1 - k);
          *a = x < y ? x : y;
          *b = x < y ? y : x;
        };
        int a1, b1, a2, b2;
        pair(t1, &a1, &b1);
        pair(t2, &a2, &b2);
        // rotation t2 (each half-warp has all sixteen); t1's comes from its lane
        float c2 = 1.f, n2 = 0.f;
        {
          const float ga = G[a2][a2], gb = G[b2][b2], gab = G[a2][b2];
          auto quotient = [](float n, float d) {
            const float r = __fdividef(1.f, d), q = n * r;
            return fmaf(r, fmaf(-d, q, n), q);
          };
          if (col(b2) < n_real && fabsf(gab) >= 0x1p-126f && ga > 0.f && gb > 0.f &&
              fabsf(gab) * rsqrtf(ga) * rsqrtf(gb) > tol) {
            // approximations polished to FP32 rounding by one Newton step each (a wrong
            // angle leaves its error times the cosine to the next sweep)
            const float zeta = quotient(0.5f * (gb - ga), gab), az = fminf(fabsf(zeta), 1e18f);
            const float z1 = fmaf(az, az, 1.f), ri = rsqrtf(z1), rt = z1 * ri;
            const float root = fmaf(0.5f * ri, fmaf(-rt, rt, z1), rt);
            const float t = copysignf(quotient(1.f, az + root), zeta);
            const float x = fmaf(t, t, 1.f);
            c2 = rsqrtf(x);
            c2 = c2 * fmaf(-0.5f * x * c2, c2, 1.5f);
            n2 = c2 * t;
            if (t1 == t2) ++nrot;
          }
        }
        const float c1 = __shfl_sync(0xffffffffu, c2, t1), n1 = __shfl_sync(0xffffffffu, n2, t1);
        // rows a1, b1 (J^T G), then columns a2, b2 (G J) of the 2x2 block
        const float x0 = G[a1][a2], x1 = G[a1][b2], y0 = G[b1][a2], y1 = G[b1][b2];
        const float p0 = c1 * x0 - n1 * y0, p1 = c1 * x1 - n1 * y1;
        const float q0 = fmaf(n1, x0, c1 * y0), q1 = fmaf(n1, x1, c1 * y1);
        Gn[a1][a2] = c2 * p0 - n2 * p1;
        Gn[a1][b2] = fmaf(n2, p0, c2 * p1);
        Gn[b1][a2] = c2 * q0 - n2 * q1;
        Gn[b1][b2] = fmaf(n2, q0, c2 * q1);
        // columns a2, b2 of Q: rows t1 and t1 + 16
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          const int k = t1 + 16 * u;
          const float qx = Q4[k][a2], qy = Q4[k][b2];
          Q4[k][a2] = c2 * qx - n2 * qy;
          Q4[k][b2] = fmaf(n2, qx, c2 * qy);
        }
        __syncthreads();
      }
    }
    if (nrot) atomicAdd(&s_rot, nrot);
    const int any = __syncthreads_or(nrot);
    // ---- 3. this rank's rows of the pair's X and Z columns times Q (skipped when
    //         nothing rotated): thread computes rows 4 rt .. + 3, columns 4 ct .. + 3
    if (any) {
      const int rt = tid >> 3, ct = tid & 7;
      for (int which = 0; which < 2; ++which) {
        float* M = which ? Z : X;
        if (!single) fetch(M, row_lo);
        for (int64_t r0 = row_lo; r0 < row_hi; r0 += ROWS) {
          if (!single || which) {
            stage();
            __syncthreads();
          }
          if (r0 + ROWS < row_hi) fetch(M, r0 + ROWS);
#pragma unroll
          for (int h = 0; h < ROWS / 128; ++h) {
            float o[4][4];
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
              for (int b = 0; b < 4; ++b) o[a][b] = 0.f;
#pragma unroll 8
            for (int k = 0; k < kJW; ++k) {
              const float4 q = *reinterpret_cast<const float4*>(&Q4[k][4 * ct]);
              const float4 x = *reinterpret_cast<const float4*>(&Ct[k * kJLd + 128 * h + 4 * rt]);
              const float xv[4] = {x.x, x.y, x.z, x.w}, qv[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
              for (int a = 0; a < 4; ++a)
#pragma unroll
                for (int b = 0; b < 4; ++b) o[a][b] = fmaf(xv[a], qv[b], o[a][b]);
            }
            const int64_t r = r0 + 128 * h + 4 * rt;
#pragma unroll
            for (int b = 0; b < 4; ++b) {
              const int c = col(4 * ct + b);
              if (c >= n_real) continue;
              float* d = M + (int64_t)c * ld + r;
              if (vec && r + 4 <= row_hi) {
                *reinterpret_cast<float4*>(d) = make_float4(o[0][b], o[1][b], o[2][b], o[3][b]);
              } else {
#pragma unroll
                for (int a = 0; a < 4; ++a)
                  if (r + a < row_hi) d[a] = o[a][b];
              }
            }
          }
          __syncthreads();   // the chunk is refilled
        }
      }
    }
    // publish: as the FP64 sweep's, one count per rank
    __syncthreads();
    if (tid < 2) add_release(ver + (tid ? Qb : P), 1);
  }
  if (split > 1) cluster.sync();   // no rank leaves while another reads its partial sums
  __syncthreads();
  if (tid == 0 && rank == 0 && s_rot) atomicAdd(status + kStatJacobiRot, s_rot);
}

__global__ void to_f32_kernel(const double* __restrict__ X, float* __restrict__ Y, int64_t n) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n;
       e += (int64_t)gridDim.x * blockDim.x)
    Y[e] = (float)X[e];
}

__global__ void to_f64_kernel(const float* __restrict__ X, double* __restrict__ Y, int64_t n) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n;
       e += (int64_t)gridDim.x * blockDim.x)
    Y[e] = (double)X[e];
}

__global__ void identity_f32_kernel(float* Z, int64_t n) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n * n;
       e += (int64_t)gridDim.x * blockDim.x)
    Z[e] = (e % n) == (e / n) ? 1.f : 0.f;
}

__global__ void column_norms_kernel(const double* __restrict__ X, int64_t ldx, int64_t m,
                                    double* __restrict__ out) {
  __shared__ double red[kJacThreads / 32];
  const double* x = X + blockIdx.x * ldx;
  double s = 0.0;
  for (int64_t r = threadIdx.x; r < m; r += kJacThreads) s = fma(x[r], x[r], s);
  s = warp_sum(s);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int k = 0; k < kJacThreads / 32; ++k) t += red[k];
    out[blockIdx.x] = sqrt(t);
  }
}

__global__ void column_dots_kernel(const double* __restrict__ A, int64_t lda,
                                   const double* __restrict__ B, int64_t ldb, int64_t m,
                                   double* __restrict__ out) {
  __shared__ double red[kJacThreads / 32];
  const double* a = A + blockIdx.x * lda;
  const double* b = B + blockIdx.x * ldb;
  double s = 0.0;
  for (int64_t r = threadIdx.x; r < m; r += kJacThreads) s = fma(a[r], b[r], s);
  s = warp_sum(s);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int k = 0; k < kJacThreads / 32; ++k) t += red[k];
    out[blockIdx.x] = t;
  }
}

__global__ void scale_columns_kernel(double* X, int64_t ldx, int64_t m, const double* s, int invert) {
  const double f = invert ? (s[blockIdx.y] > 0.0 ? 1.0 / s[blockIdx.y] : 1.0) : s[blockIdx.y];
  double* x = X + blockIdx.y * ldx;
  for (int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; r < m;
       r += (int64_t)gridDim.x * blockDim.x)
    x[r] *= f;
}

__global__ void gather_columns_kernel(const double* __restrict__ X, int64_t ldx, double* __restrict__ Y,
                                      int64_t ldy, int64_t m, const int* __restrict__ perm,
                                      const double* __restrict__ sign) {
  const int j = blockIdx.y;
  const double f = sign ? sign[j] : 1.0;
  const double* x = X + perm[j] * ldx;
  double* y = Y + j * ldy;
  for (int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; r < m;
       r += (int64_t)gridDim.x * blockDim.x)
    y[r] = f * x[r];
}

// *scale = 2^k with 4^k times the largest diagonal entry of H in [2^90, 2^92) (1 where that
// entry is not a positive number).  One block.
__global__ void eig_scale_kernel(const double* __restrict__ H, int64_t ldh, int64_t n, double* scale) {
  __shared__ double red[kJacThreads / 32];
  double mx = 0.0;
  for (int64_t i = threadIdx.x; i < n; i += kJacThreads) mx = fmax(mx, H[i + i * ldh]);
  for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = mx;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int k = 0; k < kJacThreads / 32; ++k) mx = fmax(mx, red[k]);
    *scale = mx > 0.0 && isfinite(mx) ? ldexp(1.0, (91 - ilogb(mx)) >> 1) : 1.0;
  }
}

// X = scale R^T, the strictly upper part zero.
__global__ void transpose_lower_kernel(const double* __restrict__ R, int64_t ldr, double* __restrict__ X,
                                       int64_t ldx, int64_t n, const double* __restrict__ scale) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n * n;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = e % n, j = e / n;
    X[i + j * ldx] = i >= j ? *scale * R[j + i * ldr] : 0.0;
  }
}

unsigned rows_grid(int64_t m) {
  const int64_t b = (m + 255) / 256;
  return (unsigned)std::min<int64_t>(std::max<int64_t>(b, 1), 64);
}

}  // namespace

cudaError_t column_norms(const double* X, int64_t ldx, int64_t m, int64_t n, double* out,
                         cudaStream_t st) {
  ProfScope ps(kProfOther, st);
  ps.blocks((const void*)column_norms_kernel, dim3(kJacThreads), 0, dim3((unsigned)n));
  column_norms_kernel<<<(unsigned)n, kJacThreads, 0, st>>>(X, ldx, m, out);
  return cudaGetLastError();
}

cudaError_t column_dots(const double* A, int64_t lda, const double* B, int64_t ldb, int64_t m,
                        int64_t n, double* out, cudaStream_t st) {
  ProfScope ps(kProfOther, st);
  ps.blocks((const void*)column_dots_kernel, dim3(kJacThreads), 0, dim3((unsigned)n));
  column_dots_kernel<<<(unsigned)n, kJacThreads, 0, st>>>(A, lda, B, ldb, m, out);
  return cudaGetLastError();
}

cudaError_t scale_columns(double* X, int64_t ldx, int64_t m, int64_t n, const double* s, int invert,
                          cudaStream_t st) {
  ProfScope ps(kProfOther, st);
  ps.blocks((const void*)scale_columns_kernel, dim3(256), 0, dim3(rows_grid(m), (unsigned)n));
  scale_columns_kernel<<<dim3(rows_grid(m), (unsigned)n), 256, 0, st>>>(X, ldx, m, s, invert);
  return cudaGetLastError();
}

cudaError_t gather_columns(const double* X, int64_t ldx, double* Y, int64_t ldy, int64_t m,
                           int64_t n, const int* perm, const double* sign, cudaStream_t st) {
  ProfScope ps(kProfOther, st);
  ps.blocks((const void*)gather_columns_kernel, dim3(256), 0, dim3(rows_grid(m), (unsigned)n));
  gather_columns_kernel<<<dim3(rows_grid(m), (unsigned)n), 256, 0, st>>>(X, ldx, Y, ldy, m, perm,
                                                                         sign);
  return cudaGetLastError();
}

cudaError_t transpose_lower(const double* R, int64_t ldr, double* X, int64_t ldx, int64_t n,
                            const double* scale, cudaStream_t st) {
  const int64_t b = std::min<int64_t>((n * n + 255) / 256, 4096);
  ProfScope ps(kProfOther, st);
  ps.blocks((const void*)transpose_lower_kernel, dim3(256), 0,
            dim3((unsigned)std::max<int64_t>(b, 1)));
  transpose_lower_kernel<<<(unsigned)std::max<int64_t>(b, 1), 256, 0, st>>>(R, ldr, X, ldx, n, scale);
  return cudaGetLastError();
}

// One FP64 sweep: n_even - 1 rounds of n_even / 2 pairs (ProfScope: 6 flops and
// 32 bytes per row and pair).
template <int NT, int RPT>
static cudaError_t launch_sweep(double* X, int64_t ldx, int64_t m, int64_t n_even, int64_t n_real,
                                double tol, int* status, double* nrm2, double* dsc, int* ver, int* err,
                                int stall, long long stall_ns, cudaStream_t st) {
  const void* kernel = (const void*)jacobi_sweep_kernel<NT, RPT>;
  int occ = 0, dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kernel, NT, 0) != cudaSuccess)
    return cudaErrorUnknown;
  const int64_t items = (n_even - 1) * (n_even / 2);
  // short columns: blocks further ahead than the next round only poll, and the polls
  // cost the others (n = 256: 1.1 ms a sweep with one round's 128 blocks, 1.6 with four;
  // n = 512: 2.8 and 3.5; n = 1024: 6.2 with one and a half rounds' 768, 7.8 with 512)
  const int64_t npairs = n_even / 2;
  const int64_t want = RPT == 0 ? items : m <= 512 ? npairs : npairs + npairs / 2;
  const int grid = (int)std::max<int64_t>(1, std::min<int64_t>(std::min(want, items),
                                                               (int64_t)std::max(1, occ) * sms));
  if (cudaMemsetAsync(ver, 0, sizeof(int) * n_even, st) != cudaSuccess) return cudaErrorUnknown;
  ProfScope ps(kProfJacobi, st, 6.0 * (double)m * (double)items, 32.0 * (double)m * (double)items);
  ps.blocks(kernel, dim3(NT), 0, dim3(grid));
  int ne = (int)n_even, nr = (int)n_real;
  void* args[] = {&X, &ldx, &m, &ne, &nr, &tol, &status, &nrm2, &dsc, &ver, &err, &stall, &stall_ns};
  return cudaLaunchCooperativeKernel(kernel, grid, NT, args, 0, st);
}

cudaError_t jacobi_sweep(double* X, int64_t ldx, int64_t m, int64_t n_even, int64_t n_real,
                         double tol, int* status, double* nrm2, double* dsc, int* ver, int* err,
                         int stall, long long stall_ns, cudaStream_t st) {
  // up to 1024 rows in registers; longer columns are bound by the FP64 units and want
  // six blocks an SM (4096 rows: 161 ms a sweep, 237 with 16 rows a thread held)
  const auto launch = m <= 256    ? launch_sweep<128, 2>
                      : m <= 512  ? launch_sweep<128, 4>
                      : m <= 1024 ? launch_sweep<256, 4>
                                  : launch_sweep<256, 0>;
  return launch(X, ldx, m, n_even, n_real, tol, status, nrm2, dsc, ver, err, stall, stall_ns, st);
}

// Full driver.  Returns 0; 1 = CUDA error, 2 = no convergence, 3 = a bounded
// wait expired.  lam_out (host, n) receives the eigenvalues in the order of V's
// columns (descending |lambda|).
int eig_sym_jacobi(const double* H, int64_t ldh, int64_t n, double* V, int64_t ldv, double* lam_out,
                   const EigWork& w, int* sweeps, cudaStream_t st) {
  // ---- Cholesky H = R^T R (shifted by 10 n eps ||H||_F if it breaks down)
  CholBuffers cb{w.R, 0, w.Rinv, 0};
  int hstat[kStatSlots] = {0, 0, 0, 0};
  double shift = 0.0;
  for (int attempt = 0; attempt < 2; ++attempt) {
    if (cudaMemsetAsync(w.status, 0, sizeof(int) * kStatSlots, st) != cudaSuccess) return 1;
    if (copy_matrix(H, ldh, w.R, n, n, n, st) != cudaSuccess) return 1;
    if (shift != 0.0 && init_shifted(w.R, w.R, 0, n, &shift, 1, st) != cudaSuccess) return 1;
    if (cholesky_upper_batched(cb, n, 1, w.status, st) != cudaSuccess) return 1;
    if (cudaMemcpyAsync(hstat, w.status, sizeof(hstat), cudaMemcpyDeviceToHost, st) != cudaSuccess)
      return 1;
    if (cudaStreamSynchronize(st) != cudaSuccess) return 1;
    if (!hstat[kStatCholFail]) break;
    if (attempt == 1) return 2;
    if (frob_norm2(H, ldh, n, n, w.HV, w.lam, st) != cudaSuccess) return 1;
    double nrm2 = 0.0;
    if (cudaMemcpyAsync(&nrm2, w.lam, sizeof(double), cudaMemcpyDeviceToHost, st) != cudaSuccess)
      return 1;
    if (cudaStreamSynchronize(st) != cudaSuccess) return 1;
    shift = 10.0 * (double)n * kEps * sqrt(nrm2);
  }
  const int64_t nn = n * n;
  const unsigned eg = (unsigned)std::min<int64_t>((nn + 255) / 256, 4096);
  const int64_t n_even = n + (n & 1);
  int total_sweeps = 0;
  // ---- FP32 phase on X32 = R^T, rotations accumulated in Z32
  if (cudaMemsetAsync(w.err, 0, sizeof(int), st) != cudaSuccess) return 1;
  double* scale = w.lam;   // free until the FP64 sweeps
  {
    ProfScope ps(kProfOther, st);
    ps.blocks((const void*)eig_scale_kernel, dim3(kJacThreads), 0, dim3(1));
    eig_scale_kernel<<<1, kJacThreads, 0, st>>>(H, ldh, n, scale);
  }
  if (transpose_lower(w.R, n, w.X, n, n, scale, st) != cudaSuccess) return 1;
  {
    ProfScope ps(kProfOther, st);
    ps.blocks((const void*)to_f32_kernel, dim3(256), 0, dim3(eg));
    to_f32_kernel<<<eg, 256, 0, st>>>(w.X, w.X32, nn);
  }
  {
    ProfScope ps(kProfOther, st);
    ps.blocks((const void*)identity_f32_kernel, dim3(256), 0, dim3(eg));
    identity_f32_kernel<<<eg, 256, 0, st>>>(w.Z32, n);
  }
  if (n > 1) {
    const bool wide = n >= 2048;
    const auto kern = wide ? jacobi32_block_sweep_kernel<256> : jacobi32_block_sweep_kernel<128>;
    const void* kernel = (const void*)kern;
    const int smem = wide ? jac32_smem<256>() : jac32_smem<128>();
    if (smem_attr_once(kernel, smem) != cudaSuccess) return 1;
    const int nb = (int)((n + kJB - 1) / kJB);
    const int nb_even = nb + (nb & 1), npairs = nb_even / 2;
    // CTAs per block pair (one cluster): while each keeps 128 rows and all pairs of a
    // round fit on the GPU at once
    int split = 8, grid = 0;
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute at[2];
    for (;; split /= 2) {
      cfg.blockDim = dim3(kJacThreads);
      cfg.dynamicSmemBytes = smem;
      cfg.gridDim = dim3((unsigned)(npairs * split));
      cfg.stream = st;
      at[0].id = cudaLaunchAttributeCooperative;
      at[0].val.cooperative = 1;
      at[1].id = cudaLaunchAttributeClusterDimension;
      at[1].val.clusterDim.x = split;
      at[1].val.clusterDim.y = 1;
      at[1].val.clusterDim.z = 1;
      cfg.attrs = at;
      cfg.numAttrs = split > 1 ? 2 : 1;
      if (split == 1) break;
      int clusters = 0;
      if ((n + split - 1) / split < kJRows) continue;
      if (cudaOccupancyMaxActiveClusters(&clusters, kernel, &cfg) != cudaSuccess) return 1;
      if (clusters >= npairs) break;
    }
    if (split == 1) {
      int occ = 0, dev = 0, sms = 0;
      if (cudaGetDevice(&dev) != cudaSuccess ||
          cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
          cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kernel, kJacThreads, smem) != cudaSuccess)
        return 1;
      cfg.gridDim = dim3((unsigned)std::min<int64_t>(npairs, (int64_t)std::max(1, occ) * sms));
    }
    grid = (int)cfg.gridDim.x;
    const float tol32 = 8e-6f;
    for (int sw = 0; sw < 25; ++sw) {
      if (cudaMemsetAsync(w.status + kStatJacobiRot, 0, sizeof(int), st) != cudaSuccess) return 1;
      if (cudaMemsetAsync(w.ver, 0, sizeof(int) * nb_even, st) != cudaSuccess) return 1;
      {
        // Gram and two products with Q per block pair: 6 (2 kJB)^2 m flops
        ProfScope ps(kProfJacobi32, st,
                     6.0 * kJW * kJW * (double)n * (double)npairs * (double)(nb_even - 1));
        ps.blocks(kernel, dim3(kJacThreads), smem, dim3(grid));
        if (cudaLaunchKernelEx(&cfg, kern, w.X32, w.Z32, n, n, nb_even, (int)n,
                               tol32, w.status, w.ver, w.err, sw == 0 ? w.stall : 0, w.stall_ns, split,
                               (int)(n % 4 == 0)) != cudaSuccess)
          return 1;
      }
      int rot = 0, herr = 0;
      if (cudaMemcpyAsync(&rot, w.status + kStatJacobiRot, sizeof(int), cudaMemcpyDeviceToHost, st) !=
              cudaSuccess ||
          cudaMemcpyAsync(&herr, w.err, sizeof(int), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
          cudaStreamSynchronize(st) != cudaSuccess)
        return 1;
      if (herr) return 3;
      ++total_sweeps;
      if (rot < n) break;
    }
  }
  // ---- Z orthonormal in FP64 (Cholesky QR: Z^T Z = R_z^T R_z, Z <- Z R_z^{-1})
  {
    ProfScope ps(kProfOther, st);
    ps.blocks((const void*)to_f64_kernel, dim3(256), 0, dim3(eg));
    to_f64_kernel<<<eg, 256, 0, st>>>(w.Z32, w.Z, nn);
  }
  {
    GemmArgs g;
    g.M = g.N = (int)n; g.K = (int)n; g.transA = 1;
    g.A = w.Z; g.lda = n; g.B = w.Z; g.ldb = n; g.Cout = w.HV; g.ldcout = n; g.c_upper = 1;
    g.alpha[0] = 1.0;
    if (gemm_f64(g, st) != cudaSuccess) return 1;
    CholBuffers cz{w.HV, 0, w.Rinv, 0};
    if (cudaMemsetAsync(w.status, 0, sizeof(int) * kStatSlots, st) != cudaSuccess) return 1;
    if (cholesky_upper_batched(cz, n, 1, w.status, st) != cudaSuccess) return 1;
    if (trsm_right_upper_batched(w.Z, n, cz, w.X, 0, w.tmp, 0, n, n, 1, st) != cudaSuccess) return 1;
  }
  // ---- X = R^T Z in FP64 (w.Z <- R^T, scaled as before, w.HV <- R^T Z)
  if (transpose_lower(w.R, n, w.Z, n, n, scale, st) != cudaSuccess) return 1;
  {
    GemmArgs g;
    g.M = g.N = g.K = (int)n;
    g.A = w.Z; g.lda = n; g.B = w.X; g.ldb = n; g.Cout = w.HV; g.ldcout = n;
    g.alpha[0] = 1.0;
    if (gemm_f64(g, st) != cudaSuccess) return 1;
  }
  double* X = w.HV;
  // ---- FP64 sweeps
  // ||V^T V - I||_F / sqrt(n) with rotations down to 2 eps and down to 8 eps: n = 256
  // 1.2e-15 and 4.8e-15, n = 1024 2.7e-15 and 5.2e-15, n = 4096 4.3e-15 and 1.1e-14
  const double tol_rot = 2.0 * kEps, tol_loose = sqrt((double)n) * kEps;
  bool converged = n == 1;
  for (int sw = 0; sw < 40 && !converged; ++sw) {
    if (cudaMemsetAsync(w.status + kStatJacobiRot, 0, 2 * sizeof(int), st) != cudaSuccess) return 1;
    // fold the previous sweep's column scales in, then the squared column norms
    // afresh (w.lam and w.tmp are free until the Rayleigh quotients)
    if (sw > 0 && scale_columns(X, n, n, n, w.tmp, 0, st) != cudaSuccess) return 1;
    {
      ProfScope ps(kProfOther, st);
      ps.blocks((const void*)fill_kernel, dim3(256), 0, dim3((unsigned)((n + 255) / 256)));
      fill_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(w.tmp, n, 1.0);
    }
    if (column_dots(X, n, X, n, n, n, w.lam, st) != cudaSuccess) return 1;
    if (jacobi_sweep(X, n, n, n_even, n, tol_rot, w.status, w.lam, w.tmp, w.ver, w.err,
                     sw == 0 ? w.stall64 : 0, w.stall_ns, st) != cudaSuccess)
      return 1;
    int rs[2] = {0, 0}, herr = 0;
    if (cudaMemcpyAsync(rs, w.status + kStatJacobiRot, sizeof(rs), cudaMemcpyDeviceToHost, st) !=
            cudaSuccess ||
        cudaMemcpyAsync(&herr, w.err, sizeof(int), cudaMemcpyDeviceToHost, st) != cudaSuccess)
      return 1;
    if (cudaStreamSynchronize(st) != cudaSuccess) return 1;
    if (herr) return 3;
    ++total_sweeps;
    float maxcos;
    memcpy(&maxcos, &rs[1], sizeof(float));
    if (rs[0] == 0) converged = true;
    else if (maxcos <= tol_loose) converged = true;
  }
  *sweeps = total_sweeps;
  if (!converged) return 2;
  if (n > 1 && scale_columns(X, n, n, n, w.tmp, 0, st) != cudaSuccess) return 1;
  // ---- eigenvectors (normalised columns) and Rayleigh quotients
  if (column_norms(X, n, n, n, w.lam, st) != cudaSuccess) return 1;
  if (scale_columns(X, n, n, n, w.lam, 1, st) != cudaSuccess) return 1;
  GemmArgs g;
  g.M = g.N = g.K = (int)n;
  g.A = H; g.lda = ldh; g.B = X; g.ldb = n; g.Cout = w.Z; g.ldcout = n;
  g.alpha[0] = 1.0;
  if (gemm_f64(g, st) != cudaSuccess) return 1;
  if (column_dots(X, n, w.Z, n, n, n, w.lam, st) != cudaSuccess) return 1;
  std::vector<double> lam(n);
  if (cudaMemcpyAsync(lam.data(), w.lam, sizeof(double) * n, cudaMemcpyDeviceToHost, st) !=
      cudaSuccess)
    return 1;
  if (cudaStreamSynchronize(st) != cudaSuccess) return 1;
  std::vector<int> perm(n);
  for (int64_t i = 0; i < n; ++i) perm[i] = (int)i;
  std::stable_sort(perm.begin(), perm.end(),
                   [&](int a, int b) { return std::fabs(lam[a]) > std::fabs(lam[b]); });
  for (int64_t i = 0; i < n; ++i) lam_out[i] = lam[perm[i]];
  if (cudaMemcpyAsync(w.perm, perm.data(), sizeof(int) * n, cudaMemcpyHostToDevice, st) !=
      cudaSuccess)
    return 1;
  if (gather_columns(X, n, V, ldv, n, n, w.perm, nullptr, st) != cudaSuccess) return 1;
  // the host vectors must outlive the async copy
  if (cudaStreamSynchronize(st) != cudaSuccess) return 1;
  return 0;
}

}  // namespace zolo
