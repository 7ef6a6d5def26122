// Cholesky form of one Zolo-PD iteration (Algorithm 1 step (d)):
//   Z_j = X^T X + c_{2j-1} I = R_j^T R_j   (upper R_j; the paper's "L = Chol(Z)"
//   with X L^{-1} L^{-*} is consistent only for this upper factor),
//   T_j = a_j (X R_j^{-1}) R_j^{-T}.
// Blocked right-looking Cholesky: the NB x NB diagonal block is factored in
// shared memory by one CTA per shift, which also inverts it; the row panel is
// R_kk^{-T} Z_k,rest and the trailing update a SYRK, both on the FP64 GEMM.
// The triangular solves are recursive: halve the columns, solve one half,
// update the other with one GEMM whose inner dimension is the half's width,
// solve it; 64-column leaves are products with the inverted diagonal block.
// Every column of the right-hand side is read by O(log n) GEMMs (the
// block-column-by-block-column form reads the solved part once per block, which
// on the split path re-slices it n/64 times).
#include <cmath>

#include "fp64_scalar.cuh"
#include "zolo_internal.h"

namespace zolo {
namespace {

constexpr int kDiagThreads = 256;

// Inverse of the NB x NB upper-triangular R in S (zero outside its first columns,
// reciprocal diagonal in Dinv), kept transposed in the strictly lower part of S: 8 x 8
// diagonal blocks by back substitution (one thread per column), then pairs merged as
// X_12 = -X_11 (R_12 X_22), h = 8, 16, 32: every sum's length is the same for a whole
// warp (lanes along the rows of R_12 X_22, then along the columns of X_11 Y), so the
// triangles' zeros cost nothing.  All threads of the block call it.
template <int NB>
__device__ void invert_upper(double (*S)[NB + 1], const double* Dinv, double (*Y)[NB / 2 + 1]) {
  static_assert(NB == 64 && kDiagThreads == 256, "thread mapping below");
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (warp < NB / 32) {
    const int c = 32 * warp + lane, b0 = c & ~7, j = c & 7;
    double x[8];
#pragma unroll
    for (int i = 7; i >= 0; --i) {
      double t = 0.0;
#pragma unroll
      for (int l = i + 1; l < 8; ++l)
        if (l <= j) t = fma(S[b0 + i][b0 + l], x[l], t);
      x[i] = i == j ? Dinv[c] : (i < j ? -t * Dinv[b0 + i] : 0.0);
    }
    __syncwarp();
#pragma unroll
    for (int i = 0; i < 8; ++i)
      if (i < j) S[c][b0 + i] = x[i];
  }
  __syncthreads();
#pragma unroll
  for (int h = 8; h < NB; h *= 2) {
    const int pr = lane / h, u = lane % h;      // pair (lanes cover 32 / h of them at a time)
    for (int p0 = 0; p0 < NB / (2 * h); p0 += 32 / h) {
      const int a = (p0 + pr) * 2 * h, b = a + h;
      for (int c = warp; c < h; c += kDiagThreads / 32) {   // (R_12 X_22)(u, c)
        double t = S[a + u][b + c] * Dinv[b + c];
        for (int l = 0; l < c; ++l) t = fma(S[a + u][b + l], S[b + c][b + l], t);
        Y[(pr * h + u)][c] = t;
      }
      __syncthreads();
      for (int r = warp; r < h; r += kDiagThreads / 32) {   // -(X_11 Y)(r, u)
        double t = Dinv[a + r] * Y[pr * h + r][u];
        for (int l = r + 1; l < h; ++l) t = fma(S[a + l][a + r], Y[pr * h + l][u], t);
        S[b + u][a + r] = -t;
      }
      __syncthreads();
    }
  }
}

// Cholesky of one 64 x 64 diagonal block and the inverse of its factor.  The chain of
// pivots is what bounds it: eight columns at a time, every warp that has work factors
// the 8 x 8 diagonal block in registers (lanes 0..7) together with 24 columns to its
// right (lanes 8..31, the same instructions), so a pivot costs one root, one scale and
// one update (about 650 clocks), and the rank-8 update of the rest runs on all warps
// with rows paired to equal lengths.
// Measured: 77 us per 64 x 64 block (factor and inverse), 143 us with one column per
// step and a division per pivot.
template <int NB>
__global__ void __launch_bounds__(kDiagThreads)
chol_diag_kernel(double* Z, int64_t strideZ, int64_t n, int64_t k0, int nbk, double* Rinv,
                 int64_t strideRinv, int* status) {
  // S holds R on and above the diagonal; the inverse R^{-1} (also upper) is
  // kept transposed in the strictly lower part, its diagonal in Dinv.
  __shared__ double S[NB][NB + 1];
  __shared__ double Y[NB / 2][NB / 2 + 1];
  __shared__ double Dinv[NB];
  __shared__ int s_fail;
  double* Zj = Z + blockIdx.x * strideZ;
  double* Ij = Rinv + blockIdx.x * strideRinv + (k0 / NB) * (int64_t)(NB * NB);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (tid == 0) s_fail = 0;
  if (tid < NB) Dinv[tid] = 0.0;
  for (int e = tid; e < NB * NB; e += kDiagThreads) {
    const int i = e % NB, k = e / NB;
    S[i][k] = (i <= k && k < nbk) ? Zj[(k0 + i) + (k0 + k) * n] : 0.0;
  }
  __syncthreads();
  for (int b0 = 0; b0 < nbk; b0 += 8) {
    if (warp == 0 || b0 + 8 + 24 * warp < nbk) {
      const int col = lane < 8 ? b0 + lane : b0 + 24 * warp + lane;
      const bool mine = col < nbk;
      double d[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) d[i] = mine ? S[b0 + i][col] : 0.0;
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        if (b0 + j < nbk) {
          const double pv = __shfl_sync(0xffffffffu, d[j], j);
          double sd = 1.0, rd = 1.0;
          if (!(pv > 0.0) || !isfinite(pv)) {
            if (lane == 0) s_fail = 1;
          } else if (pv > 1e-280 && pv < 1e280) {
            root_pair(pv, &sd, &rd);
          } else {
            sd = sqrt(pv);
            rd = 1.0 / sd;
          }
          d[j] = lane == j ? sd : d[j] * rd;
          if (warp == 0 && lane == j) Dinv[b0 + j] = rd;
#pragma unroll
          for (int i = j + 1; i < 8; ++i) d[i] = fma(-__shfl_sync(0xffffffffu, d[j], i), d[j], d[i]);
        }
      }
      // every warp read the diagonal block before warp 0 writes it
      __syncwarp();
      if (mine && (lane >= 8))
#pragma unroll
        for (int i = 0; i < 8; ++i) S[b0 + i][col] = d[i];
      if (warp == 0 && lane < 8 && mine) {
#pragma unroll
        for (int i = 0; i < 8; ++i)
          if (i <= lane) Y[i][lane] = d[i];
      }
    }
    __syncthreads();
    if (tid < 64 && (tid & 7) <= (tid >> 3) && b0 + (tid >> 3) < nbk)
      S[b0 + (tid & 7)][b0 + (tid >> 3)] = Y[tid & 7][tid >> 3];
    // rank-8 update of the rest: rows p and rest - 1 - p together have rest + 1 entries
    const int t0 = b0 + 8, rest = nbk - t0;
    for (int p = warp; 2 * p < rest; p += kDiagThreads / 32) {
      const int p2 = rest - 1 - p, len = p2 > p ? rest + 1 : rest - p;
      for (int e = lane; e < len; e += 32) {
        const int i = t0 + (e < rest - p ? p : p2), k = e < rest - p ? t0 + p + e : i + e - (rest - p);
        double t = S[i][k];
#pragma unroll
        for (int q = 0; q < 8; ++q) t = fma(-S[b0 + q][i], S[b0 + q][k], t);
        S[i][k] = t;
      }
    }
    __syncthreads();
  }
  invert_upper<NB>(S, Dinv, Y);
  for (int e = tid; e < NB * NB; e += kDiagThreads) {
    const int i = e % NB, k = e / NB;
    if (i < nbk && k < nbk && i <= k) Zj[(k0 + i) + (k0 + k) * n] = S[i][k];
    double inv = 0.0;
    if (i < nbk && k < nbk) inv = i == k ? Dinv[k] : (i < k ? S[k][i] : 0.0);
    Ij[e] = inv;
  }
  if (tid == 0 && s_fail) atomicOr(status + kStatCholFail, 1);
}

// Upper-triangular inverse of one NB x NB diagonal block of R (one CTA per block).
template <int NB>
__global__ void __launch_bounds__(kDiagThreads)
tri_inv_kernel(const double* __restrict__ R, int64_t n, double* __restrict__ Rinv, int* status) {
  __shared__ double S[NB][NB + 1];
  __shared__ double Y[NB / 2][NB / 2 + 1];
  __shared__ double Dinv[NB];
  const int64_t k0 = (int64_t)blockIdx.x * NB;
  const int nbk = n - k0 < NB ? (int)(n - k0) : NB;
  const int tid = threadIdx.x;
  for (int e = tid; e < NB * NB; e += kDiagThreads) {
    const int i = e % NB, k = e / NB;
    S[i][k] = (i <= k && k < nbk) ? R[(k0 + i) + (k0 + k) * n] : 0.0;
  }
  __syncthreads();
  if (tid < NB) {
    const double d = S[tid][tid];
    const bool bad = tid < nbk && !(d != 0.0);
    Dinv[tid] = tid < nbk && !bad ? 1.0 / d : 0.0;
    if (bad) atomicOr(status + kStatNonFinite, 1);
  }
  __syncthreads();
  invert_upper<NB>(S, Dinv, Y);
  double* Ij = Rinv + (k0 / NB) * (int64_t)(NB * NB);
  for (int e = tid; e < NB * NB; e += kDiagThreads) {
    const int i = e % NB, k = e / NB;
    double inv = 0.0;
    if (i < nbk && k < nbk) inv = i == k ? Dinv[k] : (i < k ? S[k][i] : 0.0);
    Ij[e] = inv;
  }
}

}  // namespace

cudaError_t tri_inv_diag_blocks(const double* R, int64_t n, double* Rinv, int* status,
                                cudaStream_t st) {
  ProfScope ps(kProfCholDiag, st);
  ps.blocks((const void*)tri_inv_kernel<kCholNB>, dim3(kDiagThreads), 0,
            dim3((unsigned)((n + kCholNB - 1) / kCholNB)));
  tri_inv_kernel<kCholNB><<<(unsigned)((n + kCholNB - 1) / kCholNB), kDiagThreads, 0, st>>>(
      R, n, Rinv, status);
  return cudaGetLastError();
}

cudaError_t cholesky_upper_batched(const CholBuffers& b, int64_t n, int r, int* status,
                                   cudaStream_t st) {
  constexpr int NB = kCholNB;
  cudaError_t err;
  // On the tensor cores a product with an inner dimension of 64 is bound by its outputs,
  // so what lies beyond an outer block of 256 rows is updated once per outer block and only
  // the block's own rows after every panel (4096^2 at r = 8: 211.0 -> 203.8 ms, 205.6 with
  // 128, 204.1 with 512; 48 matrices up to 1024^2: 104.1 -> 103.2 ms).  The FP64 pipe is
  // bound by its own work at 64 already.
  const int64_t OB = get_split_engine() ? 256 : NB;
  for (int64_t k0 = 0; k0 < n; k0 += NB) {
    const int64_t j0 = k0 / OB * OB, j1 = j0 + OB < n ? j0 + OB : n;   // the outer block
    const int nbk = (int)(n - k0 < NB ? n - k0 : NB);
    {
      ProfScope ps(kProfCholDiag, st, r * 2.0 / 3.0 * (double)nbk * nbk * nbk);
      ps.blocks((const void*)chol_diag_kernel<NB>, dim3(kDiagThreads), 0, dim3(r));
      chol_diag_kernel<NB><<<r, kDiagThreads, 0, st>>>(b.Z, b.strideZ, n, k0, nbk, b.Rinv,
                                                       b.strideRinv, status);
    }
    if ((err = cudaGetLastError()) != cudaSuccess) return err;
    const int64_t rest = n - k0 - nbk;
    if (rest <= 0) break;
    double* panel = b.Z + k0 + (k0 + nbk) * n;
    GemmArgs g;   // panel <- Rinv_kk^T panel (in place: each tile reads only its own columns)
    g.M = nbk; g.N = (int)rest; g.K = nbk; g.transA = 1; g.transB = 0;
    g.A = b.Rinv + (k0 / NB) * (int64_t)(NB * NB); g.lda = NB; g.strideA = b.strideRinv;
    g.B = panel; g.ldb = n; g.strideB = b.strideZ;
    g.Cout = panel; g.ldcout = n; g.strideCout = b.strideZ;
    g.batch = r;
    for (int j = 0; j < r; ++j) g.alpha[j] = 1.0;
    if ((err = gemm_any(g, st)) != cudaSuccess) return err;
    // the update of the outer block's rows, or after its last panel of all that follows
    // it (SYRK, upper tiles only)
    const int64_t c0 = k0 + nbk, top = c0 < j1 ? k0 : j0;
    GemmArgs u;
    u.M = (int)(c0 < j1 ? j1 - c0 : rest); u.N = (int)rest; u.K = (int)(c0 - top); u.transA = 1; u.transB = 0;
    u.A = u.B = b.Z + top + c0 * n; u.lda = u.ldb = n; u.strideA = u.strideB = b.strideZ;
    double* trail = b.Z + c0 + c0 * n;
    u.Cin = trail; u.ldcin = n; u.strideCin = b.strideZ; u.beta = 1.0;
    u.Cout = trail; u.ldcout = n; u.strideCout = b.strideZ;
    u.batch = r; u.c_upper = u.M == u.N;
    for (int j = 0; j < r; ++j) u.alpha[j] = -1.0;
    if ((err = gemm_any(u, st)) != cudaSuccess) return err;
  }
  return cudaSuccess;
}

namespace {

// dst_j[:, 0:w] = src_j[:, 0:w] for r matrices of m rows (column-major).
__global__ void copy_cols_kernel(const double* __restrict__ src, int64_t lds, int64_t strideS,
                                 double* __restrict__ dst, int64_t ldd, int64_t strideD, int64_t m,
                                 int w) {
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= m * w) return;
  const int64_t i = e % m, c = e / m;
  dst[blockIdx.y * strideD + i + c * ldd] = src[blockIdx.y * strideS + i + c * lds];
}

cudaError_t copy_cols(const double* src, int64_t lds, int64_t strideS, double* dst, int64_t ldd,
                      int64_t strideD, int64_t m, int w, int r, cudaStream_t st) {
  ProfScope ps(kProfOther, st, 0.0, 16.0 * m * w * r);
  ps.blocks((const void*)copy_cols_kernel, dim3(256), 0, dim3((unsigned)((m * w + 255) / 256), r));
  copy_cols_kernel<<<dim3((unsigned)((m * w + 255) / 256), r), 256, 0, st>>>(src, lds, strideS, dst,
                                                                             ldd, strideD, m, w);
  return cudaGetLastError();
}

struct TrsmCtx {
  const CholBuffers* b;
  double* Y; int64_t strideY;
  double* tmp; int64_t strideTmp;
  int64_t m, n;
  int r;
  cudaStream_t st;
};

// split point of [j0, j0 + w): a multiple of NB near the middle
int64_t half_of(int w) {
  const int nb = kCholNB;
  const int blocks = (w + nb - 1) / nb;
  return (int64_t)((blocks + 1) / 2) * nb;
}

// Y[:, j0:j0+w] R[j0:j0+w, j0:j0+w] = rhs[:, j0:j0+w]; rhs is X (shared by the
// shifts, stride strideR = 0) at the top and Y itself once updated.
cudaError_t fwd(const TrsmCtx& c, const double* rhs, int64_t ldr, int64_t strideR, int64_t j0, int w) {
  cudaError_t err;
  const CholBuffers& b = *c.b;
  if (w <= kCholNB) {
    const double* A = rhs + j0 * ldr;
    int64_t lda = ldr, strideA = strideR;
    if (rhs == c.Y) {   // in place: the product reads its own output, so copy first
      if ((err = copy_cols(rhs + j0 * ldr, ldr, strideR, c.tmp, c.m, c.strideTmp, c.m, w, c.r, c.st)) !=
          cudaSuccess)
        return err;
      A = c.tmp; lda = c.m; strideA = c.strideTmp;
    }
    GemmArgs h;   // Y_j = rhs_j Rinv_jj
    h.M = (int)c.m; h.N = w; h.K = w; h.transA = 0; h.transB = 0;
    h.A = A; h.lda = lda; h.strideA = strideA;
    h.B = b.Rinv + (j0 / kCholNB) * (int64_t)(kCholNB * kCholNB); h.ldb = kCholNB;
    h.strideB = b.strideRinv;
    h.Cout = c.Y + j0 * c.m; h.ldcout = c.m; h.strideCout = c.strideY;
    h.batch = c.r;
    for (int j = 0; j < c.r; ++j) h.alpha[j] = 1.0;
    return gemm_any(h, c.st);
  }
  const int64_t h1 = half_of(w);
  const int w2 = (int)(w - h1);
  if ((err = fwd(c, rhs, ldr, strideR, j0, (int)h1)) != cudaSuccess) return err;
  GemmArgs g;   // Y_2 = rhs_2 - Y_1 R_12
  g.M = (int)c.m; g.N = w2; g.K = (int)h1; g.transA = 0; g.transB = 0;
  g.A = c.Y + j0 * c.m; g.lda = c.m; g.strideA = c.strideY;
  g.B = b.Z + j0 + (j0 + h1) * c.n; g.ldb = c.n; g.strideB = b.strideZ;
  g.Cin = rhs + (j0 + h1) * ldr; g.ldcin = ldr; g.strideCin = strideR; g.beta = 1.0;
  g.Cout = c.Y + (j0 + h1) * c.m; g.ldcout = c.m; g.strideCout = c.strideY;
  g.batch = c.r;
  for (int j = 0; j < c.r; ++j) g.alpha[j] = -1.0;
  if ((err = gemm_any(g, c.st)) != cudaSuccess) return err;
  return fwd(c, c.Y, c.m, c.strideY, j0 + h1, w2);
}

// W[:, j0:j0+w] R[j0:j0+w, j0:j0+w]^T = Y[:, j0:j0+w], W overwriting Y.
cudaError_t bwd(const TrsmCtx& c, int64_t j0, int w) {
  cudaError_t err;
  const CholBuffers& b = *c.b;
  if (w <= kCholNB) {
    if ((err = copy_cols(c.Y + j0 * c.m, c.m, c.strideY, c.tmp, c.m, c.strideTmp, c.m, w, c.r, c.st)) !=
        cudaSuccess)
      return err;
    GemmArgs h;   // W_j = Y_j Rinv_jj^T
    h.M = (int)c.m; h.N = w; h.K = w; h.transA = 0; h.transB = 1;
    h.A = c.tmp; h.lda = c.m; h.strideA = c.strideTmp;
    h.B = b.Rinv + (j0 / kCholNB) * (int64_t)(kCholNB * kCholNB); h.ldb = kCholNB;
    h.strideB = b.strideRinv;
    h.Cout = c.Y + j0 * c.m; h.ldcout = c.m; h.strideCout = c.strideY;
    h.batch = c.r;
    for (int j = 0; j < c.r; ++j) h.alpha[j] = 1.0;
    return gemm_any(h, c.st);
  }
  const int64_t h1 = half_of(w);
  const int w2 = (int)(w - h1);
  if ((err = bwd(c, j0 + h1, w2)) != cudaSuccess) return err;
  GemmArgs g;   // Y_1 -= W_2 R_12^T
  g.M = (int)c.m; g.N = (int)h1; g.K = w2; g.transA = 0; g.transB = 1;
  g.A = c.Y + (j0 + h1) * c.m; g.lda = c.m; g.strideA = c.strideY;
  g.B = b.Z + j0 + (j0 + h1) * c.n; g.ldb = c.n; g.strideB = b.strideZ;
  g.Cin = c.Y + j0 * c.m; g.ldcin = c.m; g.strideCin = c.strideY; g.beta = 1.0;
  g.Cout = c.Y + j0 * c.m; g.ldcout = c.m; g.strideCout = c.strideY;
  g.batch = c.r;
  for (int j = 0; j < c.r; ++j) g.alpha[j] = -1.0;
  if ((err = gemm_any(g, c.st)) != cudaSuccess) return err;
  return bwd(c, j0, (int)h1);
}

}  // namespace

cudaError_t trsm_right_upper_batched(const double* X, int64_t ldx, const CholBuffers& b, double* Y,
                                     int64_t strideY, double* tmp, int64_t strideTmp, int64_t m,
                                     int64_t n, int r, cudaStream_t st) {
  if (n <= 0 || m <= 0) return cudaSuccess;
  TrsmCtx c{&b, Y, strideY, tmp, strideTmp, m, n, r, st};
  return fwd(c, X, ldx, 0, 0, (int)n);
}

cudaError_t trsm_pair_batched(const double* X, int64_t ldx, const CholBuffers& b, double* Y,
                              int64_t strideY, double* tmp, int64_t strideTmp, int64_t m,
                              int64_t n, int r, cudaStream_t st) {
  if (n <= 0 || m <= 0) return cudaSuccess;
  cudaError_t err;
  if ((err = trsm_right_upper_batched(X, ldx, b, Y, strideY, tmp, strideTmp, m, n, r, st)) !=
      cudaSuccess)
    return err;
  TrsmCtx c{&b, Y, strideY, tmp, strideTmp, m, n, r, st};
  return bwd(c, 0, (int)n);
}

}  // namespace zolo
