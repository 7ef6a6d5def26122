// FP64 GEMM on the FP64 FMA pipe (DFMA), batched or batch-reduced.
//
// On GB300 the FP64 rate is ~1.2 TFLOP/s (2 DFMA per clock per SM: a warp's DFMA
// holds its sub-partition's unit for 64 clocks) while HBM delivers ~6.7 TB/s, so
// every FP64 contraction here is bound by the FMA pipe, not by memory, and what
// decides a product's time is how evenly its outputs spread over the 152 SMs: a
// 64 x 64 x 256 tile holds one SM for 250 us.  The issue slots between two DFMAs
// are nearly free, so small tiles cost little, and the tile and a K split over a
// thread-block cluster are chosen per shape (gemm_f64_rule).  tcgen05 has no FP64
// kind, and the FP64 mma.sync path measured slower than DFMA on this part.
#include <cooperative_groups.h>

#include <algorithm>
#include <cmath>

#include "zolo_internal.h"

namespace zolo {
namespace {

constexpr int kBK = 16;

// One BM x BN output tile per cluster of `ks` CTAs (ks = 1: no cluster), each on
// one slice of K (whole kBK steps, so every step lies in exactly one slice); the
// ranks' partial tiles meet in distributed shared memory and are added in rank
// order (deterministic, no scratch).  The next step's operands are fetched into
// registers while the current one is multiplied from shared memory (two buffers,
// one barrier per step).  alpha scales op(A) as it is staged (one FP64 multiply
// per staged element, 1/BN of the FMAs) except for +-1, which cost nothing: the
// sign is applied to the result.
template <int BM, int BN, int TM, int TN>
__global__ void __launch_bounds__((BM / TM) * (BN / TN))
gemm_f64_kernel(const GemmArgs g, int ks) {
  constexpr int RT = BM / TM;           // threads along rows
  constexpr int CT = BN / TN;           // threads along columns
  constexpr int NT = RT * CT;
  constexpr int NA = BM * kBK / NT, NB = BN * kBK / NT;   // staged elements per thread
  static_assert(NA * NT == BM * kBK && NB * NT == BN * kBK, "whole staging rounds");
  constexpr int kStage = kBK * (BM + 1) + kBK * (BN + 1);
  constexpr int kSmem = 2 * kStage > BM * BN ? 2 * kStage : BM * BN;
  __shared__ double sm[kSmem];

  const int rank = blockIdx.x % ks;            // K slice (the cluster's CTAs are x-neighbours)
  int tm = blockIdx.y, tn = blockIdx.x / ks;
  if (g.b_lower) {
    // a tile's inner length is K - n0: the longest tiles start first
    const int lin = blockIdx.y * (gridDim.x / ks) + tn;
    tm = lin % gridDim.y;
    tn = lin / gridDim.y;
  }
  const int m0 = tm * BM, n0 = tn * BN;
  if (g.c_upper && m0 > n0 + BN - 1) return;   // tile strictly below the diagonal (all ranks)
  const int tid = threadIdx.x;
  const int tr = tid % RT;
  const int tc = tid / RT;

  double acc[TM][TN];
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN; ++j) acc[i][j] = 0.0;

  const int zb = blockIdx.z;                   // batch entry (output plane)
  const int zo = g.reduce ? 0 : zb / g.inner, zi = g.reduce ? 0 : zb % g.inner;
  const int bbeg = zo;
  const int nb = g.reduce ? g.batch : 1;
  int kbeg = g.b_lower ? (n0 / kBK) * kBK : 0;
  int kend = g.K;
  if (ks > 1) {
    const int kc = ((g.K + ks - 1) / ks + kBK - 1) / kBK * kBK;
    kbeg = max(kbeg, rank * kc);
    kend = min(g.K, (rank + 1) * kc);
  }
  const int per = kend > kbeg ? (kend - kbeg + kBK - 1) / kBK : 0;   // steps per batch entry
  const int steps = per * nb;

  const bool unit = !g.reduce && fabs(g.alpha[zo]) == 1.0;
  double ra[NA], rb[NB];
  auto fetch = [&](int step) {
    const int b = bbeg + step / per;
    const int k0 = kbeg + (step % per) * kBK;
    const double* A = g.A + (int64_t)b * g.strideA + zi * g.innerA;
    const double* B = g.B + (int64_t)b * g.strideB + zi * g.innerB;
#pragma unroll
    for (int u = 0; u < NA; ++u) {
      const int e = tid + u * NT;
      const int i = g.transA ? e / kBK : e % BM, kk = g.transA ? e % kBK : e / BM;
      const int gi = m0 + i, gk = k0 + kk;
      double v = 0.0;
      if (gi < g.M && gk < g.K)
        v = g.transA ? A[gk + (int64_t)gi * g.lda] : A[gi + (int64_t)gk * g.lda];
      ra[u] = v;
    }
#pragma unroll
    for (int u = 0; u < NB; ++u) {
      const int e = tid + u * NT;
      const int j = g.transB ? e % BN : e / kBK, kk = g.transB ? e / BN : e % kBK;
      const int gk = k0 + kk, gj = n0 + j;
      double v = 0.0;
      if (gk < g.K && gj < g.N)
        v = g.transB ? B[gj + (int64_t)gk * g.ldb] : B[gk + (int64_t)gj * g.ldb];
      rb[u] = v;
    }
  };
  auto stage = [&](int step, int buf) {
    double* As = sm + buf * kStage;
    double* Bs = As + kBK * (BM + 1);
    const double al = unit ? 1.0 : g.alpha[bbeg + step / per];
#pragma unroll
    for (int u = 0; u < NA; ++u) {
      const int e = tid + u * NT;
      const int i = g.transA ? e / kBK : e % BM, kk = g.transA ? e % kBK : e / BM;
      As[kk * (BM + 1) + i] = unit ? ra[u] : al * ra[u];
    }
#pragma unroll
    for (int u = 0; u < NB; ++u) {
      const int e = tid + u * NT;
      const int j = g.transB ? e % BN : e / kBK, kk = g.transB ? e / BN : e % kBK;
      Bs[kk * (BN + 1) + j] = rb[u];
    }
  };
  if (steps > 0) {
    fetch(0);
    stage(0, 0);
  }
  __syncthreads();
  for (int step = 0; step < steps; ++step) {
    if (step + 1 < steps) fetch(step + 1);
    const double* As = sm + (step & 1) * kStage;
    const double* Bs = As + kBK * (BM + 1);
#pragma unroll
    for (int kk = 0; kk < kBK; ++kk) {
      double a[TM], bv[TN];
#pragma unroll
      for (int i = 0; i < TM; ++i) a[i] = As[kk * (BM + 1) + tr + i * RT];
#pragma unroll
      for (int j = 0; j < TN; ++j) bv[j] = Bs[kk * (BN + 1) + tc + j * CT];
#pragma unroll
      for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) acc[i][j] = fma(a[i], bv[j], acc[i][j]);
    }
    if (step + 1 < steps) stage(step + 1, (step + 1) & 1);
    __syncthreads();
  }

  double* C = g.Cout + (int64_t)zo * g.strideCout + zi * g.innerC;
  const double* Cin = g.Cin ? g.Cin + (int64_t)zo * g.strideCin + zi * g.innerC : nullptr;
  const bool use_in = Cin != nullptr && g.beta != 0.0;
  const bool minus = unit && g.alpha[zo] < 0.0;
  auto put = [&](int i, int j, double v) {
    const int gi = m0 + i, gj = n0 + j;
    if (gi >= g.M || gj >= g.N) return;
    if (minus) v = -v;
    if (use_in) v = fma(g.beta, Cin[gi + (int64_t)gj * g.ldcin], v);
    C[gi + (int64_t)gj * g.ldcout] = v;
  };
  if (ks == 1) {
#pragma unroll
    for (int j = 0; j < TN; ++j)
#pragma unroll
      for (int i = 0; i < TM; ++i) put(tr + i * RT, tc + j * CT, acc[i][j]);
    return;
  }
  // every rank of this tile has read its operands before any rank writes C (the barrier)
  namespace cgrp = cooperative_groups;
  cgrp::cluster_group cluster = cgrp::this_cluster();
#pragma unroll
  for (int j = 0; j < TN; ++j)
#pragma unroll
    for (int i = 0; i < TM; ++i) sm[(tr + i * RT) + (tc + j * CT) * BM] = acc[i][j];
  cluster.sync();
  const int share = BM * BN / ks;
  for (int e = rank * share + tid; e < (rank + 1) * share; e += NT) {
    double v = 0.0;
    for (int q = 0; q < ks; ++q) v += cluster.map_shared_rank(sm, q)[e];
    put(e % BM, e / BM, v);
  }
  cluster.sync();   // no rank leaves while another reads its partial tile
}

__global__ void gemm_beta_only(const GemmArgs g) {
  const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (e >= (int64_t)g.M * g.N) return;
  const int64_t i = e % g.M, j = e / g.M;
  const int z = blockIdx.z;
  double* C = g.Cout + (int64_t)z * g.strideCout;
  const double* Cin = g.Cin ? g.Cin + (int64_t)z * g.strideCin : nullptr;
  C[i + j * g.ldcout] = (Cin && g.beta != 0.0) ? g.beta * Cin[i + j * g.ldcin] : 0.0;
}

template <int BM, int BN, int TM, int TN>
cudaError_t launch(const GemmArgs& g, int ks, cudaStream_t st) {
  const int nz = g.reduce ? 1 : g.batch * g.inner;
  constexpr int NT = (BM / TM) * (BN / TN);
  dim3 grid((g.N + BN - 1) / BN * ks, (g.M + BM - 1) / BM, nz);
  const double bytes = 8.0 * g.batch * ((double)g.M * g.K + (double)g.K * g.N) +
                       8.0 * nz * (double)g.M * g.N * (g.beta != 0.0 ? 2 : 1);
  ProfScope ps(kProfGemm, st, gemm_flops(g), bytes);
  ps.blocks((const void*)gemm_f64_kernel<BM, BN, TM, TN>, dim3(NT), 0, grid);
  if (ks == 1) {
    gemm_f64_kernel<BM, BN, TM, TN><<<grid, NT, 0, st>>>(g, 1);
    return cudaGetLastError();
  }
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(NT);
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = ks;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, gemm_f64_kernel<BM, BN, TM, TN>, g, ks);
}

}  // namespace

// Algorithmic flops of one call: the products the structure leaves non-zero.
double gemm_flops(const GemmArgs& g) {
  double per = 2.0 * g.M * (double)g.N * g.K;
  if (g.c_upper) per = (double)g.K * g.N * (g.N + 1.0);
  else if (g.b_lower) per = 2.0 * g.M * ((double)g.N * g.K - 0.5 * (double)g.N * (g.N - 1.0));
  return per * g.batch * g.inner;
}

namespace {
thread_local bool t_gemm_crowded = false;
}
CrowdedScope::CrowdedScope(bool on) : prev(t_gemm_crowded) { t_gemm_crowded = on; }
CrowdedScope::~CrowdedScope() { t_gemm_crowded = prev; }

int gemm_f64_default_variant(const GemmArgs&) { return kGemmVRule; }

// The tile and K split the rule takes: the least estimated time, in clocks, of
//   c (BM BN K / ks) / 2 / eff(c) + a cluster's fixed cost,   c = ceil(CTAs / SMs)
// (2 DFMA per clock per SM; the c CTAs that share an SM share its FP64 units, so a
// wave that is not full costs as much as a full one, and a single small CTA leaves
// them waiting at its barriers).  Measured at 2.0 GHz: 1024^3 takes 2.09 / 1.88 /
// 1.88 ms with one 64 / 32 / 16 tile per CTA (c = 2 / 7 / 27); 256^3 takes 271 / 88
// / 44 us unsplit and 39 us as 16 x 16 tiles cut in four; 32 x 96 x 8224 in a batch
// of six takes 980 / 494 / 338 / 297 us as 16 x 16 tiles cut in 1 / 2 / 4 / 8 (c = 1
// / 1 / 2 / 4); 144 CTAs in clusters of eight found two to an SM.
F64Tile gemm_f64_rule(const GemmArgs& g) {
  struct Cand { int id, bm, bn; double eff[4]; };   // eff at c = 1, 2, 3, >= 4
  static const Cand all[] = {{0, 64, 64, {0.95, 0.99, 1.0, 1.0}},
                             {1, 32, 32, {0.73, 0.92, 0.96, 0.98}},
                             {2, 16, 16, {0.54, 0.78, 0.86, 0.93}}};
  static const Cand inplace[] = {{3, 64, 16, {0.73, 0.92, 0.96, 0.97}},
                                 {0, 64, 64, {0.95, 0.99, 1.0, 1.0}}};
  // C in the address range of A or B: tiles that are right in place where elements are
  // shared (if none is, gemm_f64_variant forms the product beside C), and tall ones where
  // none are (the Cholesky updates)
  const bool alias = gemm_output_aliases_input(g);
  const Cand* c = alias ? inplace : all;
  const int nc = alias ? 2 : 3;
  F64Tile best{0, 1};
  // with many lanes in flight (the split forms' batch) large clusters wait for
  // room: 48 matrices take 201.5 / 199.2 / 197.2 / 198.1 ms with up to 8 / 4 / 2 / 1
  const bool crowded = get_split_engine() && get_split_engine()->throughput;
  // an FP64 batch's larger matrices fill the FP64 units between them: their products take
  // the tile that costs the units least, whole (24 matrices of 800^2 .. 1024^2: 955 ms, 975
  // unsplit by the estimate of a call's own time, 993 by that estimate with K splits, 979
  // with 64 x 64 tiles throughout)
  const bool shared = t_gemm_crowded;
  const int ks_max = shared ? 1 : g.b_lower || crowded ? 2 : 8;
  double best_t = 1e300;
  for (int q = 0; q < nc; ++q) {
    const double tm = (g.M + c[q].bm - 1) / c[q].bm, tn = (g.N + c[q].bn - 1) / c[q].bn;
    if (tm > 65535.0) continue;   // grid.y
    if (alias && !gemm_tile_in_place(g, c[q].bm, c[q].bn)) continue;
    double tiles = tm * tn * (g.reduce ? 1 : g.batch * g.inner);
    if (g.c_upper) tiles *= 0.5 * (1.0 + 1.0 / tn);
    const double kfrac = g.b_lower ? 0.5 * (1.0 + (double)c[q].bn / std::max(g.K, c[q].bn)) : 1.0;
    for (int ks = 1; ks <= ks_max; ks *= 2) {
      if (ks > 1 && g.K < 2 * kBK * ks) break;
      const double kc = ((g.K + ks - 1) / ks + kBK - 1) / kBK * kBK;
      const double cta = 0.5 * c[q].bm * c[q].bn * kc * (g.reduce ? g.batch : 1);
      double per_sm = std::ceil(tiles * ks / 152.0);
      if (ks == 8 && tiles * ks > 128.0) per_sm = std::max(per_sm, 2.0);
      const double eff = c[q].eff[per_sm > 4.0 ? 3 : (int)per_sm - 1];
      // triangular op(B): the CTAs' lengths differ, so an SM that holds few of them
      // ends with the longest one alone, and K slices are uneven (1024^3, r = 6
      // reduced: 8.98 / 7.11 / 5.70 ms with 64 / 32 / 16 tiles, 8.45 as 16 cut in two)
      const double uneven = g.b_lower ? (1.0 + 2.0 / per_sm) * (ks > 1 ? 1.5 : 1.0) : 1.0;
      double t = std::max(per_sm * kfrac, 1.0) * cta * uneven / eff + (ks > 1 ? 3000.0 + 300.0 * ks : 0.0);
      if (shared) t = tiles * kfrac * cta / c[q].eff[3] / 152.0;
      if (t < best_t) {
        best_t = t;
        best = {c[q].id, ks};
      }
    }
  }
  return best;
}

cudaError_t gemm_f64_tile(const GemmArgs& g, F64Tile t, cudaStream_t st) {
  switch (t.tile) {
    case 1: return launch<32, 32, 4, 2>(g, t.ks, st);
    case 2: return launch<16, 16, 1, 2>(g, t.ks, st);
    case 3: return launch<64, 16, 4, 2>(g, t.ks, st);
    default: return launch<64, 64, 4, 4>(g, t.ks, st);
  }
}

namespace {

// The product into a scratch, then copied over C: for an output that shares elements
// with an input and a tile that would write what another tile has yet to read.
cudaError_t gemm_f64_beside(const GemmArgs& g, int variant, cudaStream_t st) {
  const int nz = g.reduce ? 1 : g.batch * g.inner;
  double* tmp = nullptr;
  cudaError_t e = cudaMallocAsync((void**)&tmp, sizeof(double) * (size_t)nz * g.M * (size_t)g.N, st);
  if (e != cudaSuccess) {
    cudaGetLastError();
    return e;
  }
  GemmArgs h = g;
  h.Cout = tmp;
  h.ldcout = g.M;
  h.innerC = (int64_t)g.M * g.N;
  h.strideCout = h.innerC * g.inner;
  e = gemm_f64_variant(h, variant, st);
  for (int z = 0; z < nz && e == cudaSuccess; ++z)
    e = copy_matrix(tmp + z * h.innerC, g.M,
                    g.Cout + (z / g.inner) * g.strideCout + (z % g.inner) * g.innerC, g.ldcout, g.M, g.N, st);
  const cudaError_t f = cudaFreeAsync(tmp, st);
  return e != cudaSuccess ? e : f;
}

}  // namespace

cudaError_t gemm_f64_variant(const GemmArgs& g, int variant, cudaStream_t st) {
  if (g.M <= 0 || g.N <= 0 || g.batch <= 0) return cudaSuccess;
  if (g.batch > kGemmMaxBatch) return cudaErrorInvalidValue;
  if (g.K <= 0) {
    // empty contraction: C_out = beta * C_in (or 0)
    const int nz = g.reduce ? 1 : g.batch;
    dim3 grid((unsigned)((g.M * (int64_t)g.N + 255) / 256), 1, nz);
    ProfScope ps(kProfOther, st);
    ps.blocks((const void*)gemm_beta_only, dim3(256), 0, dim3(grid));
    gemm_beta_only<<<grid, 256, 0, st>>>(g);
    return cudaGetLastError();
  }
  static const int kTile[4][2] = {{64, 64}, {32, 32}, {16, 16}, {64, 16}};   // by F64Tile::tile
  const bool wide = variant == kGemmV32x128 || variant == kGemmV32x64;
  const bool split_k = variant == kGemmVSplitK2 || variant == kGemmVSplitK4 || variant == kGemmVSplitK8;
  const F64Tile t = wide || split_k ? F64Tile{0, 1} : gemm_f64_rule(g);
  const int bm = wide ? 32 : kTile[t.tile][0];
  const int bn = variant == kGemmV32x128 ? 128 : wide ? 64 : kTile[t.tile][1];
  if (!gemm_tile_in_place(g, bm, bn)) return gemm_f64_beside(g, variant, st);
  switch (variant) {
    case kGemmV32x128: return launch<32, 128, 4, 4>(g, 1, st);
    case kGemmV32x64: return launch<32, 64, 4, 4>(g, 1, st);
    case kGemmVSplitK2: return launch<64, 64, 4, 4>(g, 2, st);
    case kGemmVSplitK4: return launch<64, 64, 4, 4>(g, 4, st);
    case kGemmVSplitK8: return launch<64, 64, 4, 4>(g, 8, st);
    default: return gemm_f64_tile(g, t, st);
  }
}

}  // namespace zolo
