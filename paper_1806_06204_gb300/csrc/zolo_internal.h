// Internal declarations shared by the libzolo translation units.
#pragma once

#include <array>
#include <cstddef>
#include <cstdint>
#include <map>

#ifdef __CUDACC__
#include <cuda_runtime.h>
#else
typedef struct CUstream_st* cudaStream_t;
#endif

namespace zolo {

constexpr int kMaxR = 8;
constexpr int kMaxIters = 8;
constexpr double kTable1Tol = 1e-15;

// ---------------------------------------------------------------- coefficients
struct Coefficients {
  double ell = 0.0;
  int r = 0;
  double c[2 * kMaxR] = {};   // c_1 .. c_{2r}
  double a[kMaxR] = {};       // a_1 .. a_r
  double mhat = 0.0;          // M_hat
  double gap = 0.0;           // 1 - Zhat(l; l)
};

struct Schedule {
  int r = 0;
  int iters = 0;
  bool converged = false;
  double ell[kMaxIters + 1] = {};
  bool use_qr[kMaxIters] = {};
  Coefficients co[kMaxIters];
};

int compute_coefficients(double ell, int r, Coefficients* out);
bool qr_form_needed(const Coefficients& co);
int build_schedule(double ell0, int r, int max_iter, Schedule* out);

#ifdef __CUDACC__

// ------------------------------------------------------------- launch scopes
enum ProfClass { kProfGemm = 0, kProfPanel, kProfCholDiag, kProfJacobi, kProfCombine, kProfOther,
                 kProfSplitGemm, kProfSlice, kProfJacobi32, kProfClasses };
// Counts the launch made inside its scope and, while profiling is on, brackets
// it with CUDA events on `st`.  flops/bytes: the launch's algorithmic work.
class ProfScope {
 public:
  ProfScope(int cls, cudaStream_t st, double flops = 0.0, double bytes = 0.0);
  ~ProfScope();
  ProfScope(const ProfScope&) = delete;
  ProfScope& operator=(const ProfScope&) = delete;
  // The launch's blocks, for its SM-time: blocks / (SMs x blocks per SM of
  // `kernel` at this block size and dynamic shared memory), at most 1.  Only
  // queried while profiling is on.
  void blocks(const void* kernel, dim3 block, size_t smem, dim3 grid);

 private:
  int cls_;
  cudaStream_t st_;
  double flops_, bytes_;
  double share_ = 1.0;
  void* a_ = nullptr;
};

// cudaFuncSetAttribute(MaxDynamicSharedMemorySize) applies to the current device
// only: set it once per (kernel, device), thread-safely.
cudaError_t smem_attr_once(const void* func, int bytes);

// Launch bookkeeping for graphs: kernels recorded at capture time are counted
// when the graph is launched.
void add_launches(int64_t n);
bool profiling_enabled();

// ----------------------------------------------------------------- device flags
// A small device array of int counters written by kernels and read once at the
// end of a call.
enum StatusSlot {
  kStatNonFinite = 0,   // a NaN/Inf was produced
  kStatCholFail = 1,    // non-positive pivot in a Cholesky diagonal block
  kStatJacobiRot = 2,   // rotations applied in the current Jacobi sweep
  kStatJacobiMaxCos = 3,  // largest |cos| between two columns seen in the sweep (float bits)
  kStatSlots = 4
};

// ------------------------------------------------------------------- FP64 GEMM
// C_out[b] = beta * C_in[b] + alpha[b] * op(A[b]) op(B[b])          (reduce = 0)
// C_out    = beta * C_in    + sum_b alpha[b] * op(A[b]) op(B[b])    (reduce = 1)
// Column-major, op = N or T.  Structural flags let the kernel skip known zeros:
//   b_lower  : op(B)[k][j] == 0 for k < j (e.g. op(B) = Q2^T with Q2 upper)
//   c_upper  : only tiles touching the upper triangle (i <= j) are computed
constexpr int kGemmMaxBatch = 16;
struct GemmArgs {
  int M = 0, N = 0, K = 0;
  int transA = 0, transB = 0;
  const double* A = nullptr; int64_t lda = 0; int64_t strideA = 0;
  const double* B = nullptr; int64_t ldb = 0; int64_t strideB = 0;
  const double* Cin = nullptr; int64_t ldcin = 0; int64_t strideCin = 0;
  double* Cout = nullptr; int64_t ldcout = 0; int64_t strideCout = 0;
  double beta = 0.0;
  double alpha[kGemmMaxBatch] = {};
  int batch = 1;
  // FP64 path only (not with reduce): each batch entry is `inner` products, the
  // inner ones at these strides (batch x inner output planes, alpha per entry)
  int inner = 1;
  int64_t innerA = 0, innerB = 0, innerC = 0;
  int reduce = 0;
  int b_lower = 0;
  int c_upper = 0;
  // split path only: rescale the inner index by exact powers of two so that every
  // row of op(B) has its largest magnitude in [1/4, 1/2), moving the factors into
  // op(A)'s columns (the product is unchanged).  For products whose op(B) rows
  // differ by orders of magnitude, where one scale per output column would cost
  // the small rows their precision.
  int k_equilibrate = 0;
};
// Kernel variants of the FP64 contraction: the built-in rule (gemm_f64_rule picks
// the tile and the K split per shape), or one tile shape, or 64 x 64 tiles with
// K cut into 2 / 4 / 8 slices of whole steps over a thread-block cluster.
// kGemmVSplit names the split tensor-core path.
enum GemmVariant {
  kGemmVRule = 0, kGemmV32x128 = 1, kGemmV32x64 = 2,
  kGemmVSplitK2 = 3, kGemmVSplitK4 = 4, kGemmVSplitK8 = 5,
  kGemmVSplit = 8
};
// one FP64 launch of the given variant
cudaError_t gemm_f64_variant(const GemmArgs& g, int variant, cudaStream_t st);
int gemm_f64_default_variant(const GemmArgs& g);
// the rule's choice: tile 0 = 64 x 64, 1 = 32 x 32, 2 = 16 x 16, 3 = 64 x 16; ks CTAs
// of one cluster share the tile's K
struct F64Tile {
  int tile, ks;
};
F64Tile gemm_f64_rule(const GemmArgs& g);
cudaError_t gemm_f64_tile(const GemmArgs& g, F64Tile t, cudaStream_t st);
// FP64 contraction: the variant the current thread's tuner chose for this
// shape, else the default one.
cudaError_t gemm_f64(const GemmArgs& g, cudaStream_t st);

// Measured kernel choice per contraction shape (sizes, batch, transposes,
// structure flags, slice count, products within an entry): the cache of a handle, made current for the
// calls of one API entry point by TunerScope.  With `tuning` set, a shape met
// for the first time is run with every candidate variant into a scratch output
// (the real output untouched) and timed with CUDA events; the fastest is kept.
// No tuning while the stream is being captured.
struct GemmTuner {
  std::map<std::array<int, 7>, int> choice;
  uint64_t gen = 0;      // bumped whenever `choice` changes (graph replay keys)
  bool tuning = false;
  bool busy = false;
  double* scratch = nullptr;
  size_t scratch_elems = 0;
  cudaEvent_t t0 = nullptr, t1 = nullptr;
  ~GemmTuner();
};
std::array<int, 7> gemm_key(const GemmArgs& g, int split_slices);
// C lies in the address range of A or B (flag 128 of the key)
bool gemm_output_aliases_input(const GemmArgs& g);
// whether tiles of bm x bn leave C right when it shares elements with A or B
bool gemm_tile_in_place(const GemmArgs& g, int bm, int bn);
// whether kernel v may serve a key (tile variants other than the built-in one
// are barred for in-place products: their CTAs would overwrite rows of B that
// other CTAs still read)
bool gemm_variant_allowed(const std::array<int, 7>& key, int v);
void set_gemm_tuner(GemmTuner* t);
GemmTuner* get_gemm_tuner();
struct TunerScope {
  GemmTuner* prev;
  explicit TunerScope(GemmTuner* t) : prev(get_gemm_tuner()) { set_gemm_tuner(t); }
  ~TunerScope() { set_gemm_tuner(prev); }
};
// FP64 products of this thread run among many others: gemm_f64_rule then counts the time
// of the FP64 units, not a call's own.
struct CrowdedScope {
  bool prev;
  explicit CrowdedScope(bool on);
  ~CrowdedScope();
};
// algorithmic flops of one call (structural zeros excluded)
double gemm_flops(const GemmArgs& g);

// --------------------------------------------------- split-precision GEMM
// Same contract as gemm_f64, on the tensor cores with the operands cut into
// slices of one of three forms.
enum : int {
  kFormBF16 = 0,   // 7 (slices = 9) or 6 (slices = 8) base-256 digits in BF16
  kFormFP16 = 1,   // 7 base-256 digits in FP16
  kFormFP8 = 2     // 11 base-32 digits in E4M3
};
struct SplitWork {
  void* slices;          // slice planes
  size_t slice_elems;    // their size in 16-bit units
  int* exps;             // per-row / per-column power-of-two exponents
  size_t exp_elems;
  int* err;              // device error flag (bounded waits)
  int slices_s;          // the caller's slice count (9, 8 or 11; see split_planes)
  int form = kFormBF16;
  // test hook of the failure path: with stall = 1 the MMA issuer first waits,
  // for stall_ns, on an mbarrier that nothing arrives at, then takes the
  // bounded-wait error exit
  int stall = 0;
  long long stall_ns = 0;
  // the router's cost model: false = one call alone on the GPU (its launch and
  // pipeline latency counts); true = many calls in flight at once (zolo_pd_batched's
  // lanes), where latency is hidden and each path costs the share of the GPU's
  // FP64 pipe, tensor pipe and memory bandwidth it takes
  bool throughput = false;
};
cudaError_t gemm_split(const GemmArgs& g, SplitWork& w, cudaStream_t st);
// slice planes the caller's slice count stands for
int split_planes(int slices, int form);
// slice planes (16-bit units) one call of the given shape needs in a form
size_t split_slice_elems(int64_t M, int64_t N, int64_t K, int batch, int S, int form = kFormBF16);
// exponent entries (ints) one call of the given shape needs
size_t split_exp_elems(int64_t M, int64_t N, int64_t K, int batch, int k_equilibrate,
                       int form = kFormBF16);
// The engine every contraction of the current call goes through: FP64 (DFMA)
// when no split workspace is installed, the split tensor-core path otherwise.
void set_split_engine(SplitWork* w);
SplitWork* get_split_engine();
// the built-in router: true when the split path's estimated time (slicing and
// output traffic, slice-pair products, launch latency) beats the FP64 pipe's
bool split_preferred(const GemmArgs& g, const SplitWork& w);
// the same estimate as a ratio: split-path time / FP64 time
double split_time_ratio(const GemmArgs& g, const SplitWork& w);
// Sets the kernels' launch attributes ahead of a stream capture.
void split_prepare();
cudaError_t gemm_any(const GemmArgs& g, cudaStream_t st);

// --------------------------------------------------------------- elementwise
cudaError_t scale_copy(const double* A, int64_t lda, double* X, int64_t ldx, int64_t m, int64_t n,
                       double s, cudaStream_t st);
cudaError_t copy_matrix(const double* A, int64_t lda, double* B, int64_t ldb, int64_t m, int64_t n,
                        cudaStream_t st);
// W_j = [X; sqrt(c_j) I] for j < r, W_j at W + j*strideW with ld = m + n
cudaError_t init_stacked(const double* X, int64_t ldx, double* W, int64_t strideW, int64_t m,
                         int64_t n, const double* sqrt_c, int r, cudaStream_t st);
// Q_j = [I_n; 0] ((m+n) x n, ld m+n) for j < r
cudaError_t init_q_identity(double* Q, int64_t strideQ, int64_t m, int64_t n, int r,
                            cudaStream_t st);
// Z_j = G + shift_j I for j < r (full copy of G, n x n, ld n)
cudaError_t init_shifted(const double* G, double* Z, int64_t strideZ, int64_t n, const double* shift,
                         int r, cudaStream_t st);
// Xn = mhat * (X + sum_j coef_j * T_j) (T_j at T + j*strideT, ld ldt; nt may be 0),
// partial sums of ||Xn - X||^2 and ||Xn||^2 to norms[0..1] (after norms_finish).
cudaError_t combine(const double* X, int64_t ldx, double* Xn, int64_t ldxn, int64_t m, int64_t n,
                    double mhat, const double* T, int64_t ldt, int64_t strideT, const double* coef,
                    int nt, double* partials, double* norms, int* status, cudaStream_t st);
// S = sum_t coef_t T_t, T_t at T + t * strideT (ld ldt), t < nt <= 8
cudaError_t weighted_sum(const double* T, int64_t ldt, int64_t strideT, const double* coef, int nt,
                         double* S, int64_t lds, int64_t m, int64_t n, cudaStream_t st);
// guard zones: fill with 0xFF bytes; set *flag if any byte differs
cudaError_t guard_fill(void* p, size_t bytes, cudaStream_t st);
cudaError_t guard_check(const void* p, size_t bytes, int* flag, cudaStream_t st);
// *out = (*flag != 0) as a double
cudaError_t flag_to_double(const int* flag, double* out, cudaStream_t st);
// H = (M + M^T) / 2
// W(i, j) = W(j, i) for i > j (n x n, ld ldw): a symmetric W from its upper triangle
cudaError_t mirror_upper(double* W, int64_t ldw, int64_t n, cudaStream_t st);
cudaError_t symmetrize(const double* M, int64_t ldm, double* H, int64_t ldh, int64_t n,
                       cudaStream_t st);
cudaError_t check_finite(const double* A, int64_t lda, int64_t m, int64_t n, int* status,
                         cudaStream_t st);
// ||G - I||_F^2 into out[0] from the upper triangle of a symmetric n x n G
// (out[1] = 0)
cudaError_t gram_identity_dev2(const double* G, int64_t ldg, int64_t n, double* partials,
                               double* out, cudaStream_t st);
// ||A||_F^2 into out[0] (via partials)
cudaError_t frob_norm2(const double* A, int64_t lda, int64_t m, int64_t n, double* partials,
                       double* out, cudaStream_t st);
// alpha >= sigma_max(A) when the caller gives none: sums[0] = ||A||_F^2, sums[1] =
// ||A||_1, sums[2] = ||A||_inf (sums: 3 device doubles, written by
// alpha_bound_sums; part: alpha_bound_part_elems(m, n) doubles, colsum: n,
// partials: 2 * 1024), then alpha_from_sums = min(||A||_F, sqrt(||A||_1 ||A||_inf))
// on the host.
int64_t alpha_bound_part_elems(int64_t m, int64_t n);
cudaError_t alpha_bound_sums(const double* A, int64_t lda, int64_t m, int64_t n, double* part,
                             double* colsum, double* partials, double* sums, cudaStream_t st);
double alpha_from_sums(const double* sums);

// ------------------------------------------------------------ structured QR
constexpr int kQrNB = 32;      // panel width (columns factored by one panel kernel)
constexpr int kQrBlock = 128;  // block width (columns a panel's reflectors are applied to at once)
// Widest super-block of an n-column problem on the 16-bit split forms: the columns whose
// reflectors are applied together to everything to their right.
int qr_super_width(int64_t n);
struct QrBuffers {
  int sb;                         // qr_super_width(n) or kQrBlock: the strides below hold super-blocks this wide
  double* W;   int64_t strideW;   // stacked (m+n) x n per shift, ld m+n
  double* V;   int64_t strideV;   // explicit reflectors (m+sb) x n per shift, ld m+sb, rows
                                  // relative to the start of each column's super-block
  double* T;   int64_t strideT;   // nb x nb triangular factor per panel
  double* Tb;  int64_t strideTb;  // sb x sb triangular factor per super-block
  double* G;   int64_t strideG;   // sb x sb Gram V^T V scratch
  double* W1;  int64_t strideW1;  // sb x n scratch
  double* W2;  int64_t strideW2;  // sb x n scratch
};
// Factor [X; sqrt(c_j) I] for j < r and overwrite W_j with the thin Q_j
// (explicit_q = false: leave R on and above the diagonal of W_j's top block).
// narrow_panels: many problems are in flight on other streams; the panel kernel
// then takes the fewest CTAs per shift whose registers hold the rows.
cudaError_t structured_qr_q(const QrBuffers& b, int64_t m, int64_t n, int r, int* status,
                            cudaStream_t st, bool explicit_q = true, bool narrow_panels = false);
// Asks the current device for its cluster sizes (before a stream capture).
void qr_prepare();
// This thread's panels take clusters of `limit` CTAs at most (8, 12 or 16; 0: as they are).
struct PanelClusterScope {
  int prev;
  explicit PanelClusterScope(int limit);
  ~PanelClusterScope();
};
// Inverses of the NB x NB diagonal blocks of an upper-triangular R (ld n) in the
// layout cholesky_upper_batched leaves in Rinv; a zero pivot sets status.
cudaError_t tri_inv_diag_blocks(const double* R, int64_t n, double* Rinv, int* status,
                                cudaStream_t st);

// ----------------------------------------------------------------- Cholesky
constexpr int kCholNB = 64;
struct CholBuffers {
  double* Z;    int64_t strideZ;     // n x n, ld n: in = Z_j (upper), out = R_j (upper)
  double* Rinv; int64_t strideRinv;  // inverses of the nb x nb diagonal blocks, nb x nb each
};
cudaError_t cholesky_upper_batched(const CholBuffers& b, int64_t n, int r, int* status,
                                   cudaStream_t st);
// Y_j = X R_j^{-1} then Y_j <- Y_j R_j^{-T} (in place), j < r.
cudaError_t trsm_pair_batched(const double* X, int64_t ldx, const CholBuffers& b, double* Y,
                              int64_t strideY, double* tmp, int64_t strideTmp, int64_t m,
                              int64_t n, int r, cudaStream_t st);

// ------------------------------------------------------------ eigensolver
struct EigWork {
  double* R;        // n x n
  double* X;        // n x n, one-sided Jacobi iterate
  double* HV;       // n x n
  double* Rinv;     // (n/nb+1) * nb * nb
  double* lam;      // n
  int* perm;        // n (device)
  int* status;
  float* X32;       // n x n, FP32 sweeps
  float* Z32;       // n x n, accumulated FP32 rotations
  double* Z;        // n x n, Z orthonormalised in FP64
  double* tmp;      // n x 64 scratch of the triangular solve
  int* ver;         // n + 1 round counters, per column (FP64 sweeps) or block (FP32 ones)
  int* err;         // bounded-wait error flag
  // test hook of the failure path: with stall = 1, block 0 of the first FP32
  // sweep waits, for stall_ns, on a flag nothing sets, then takes the
  // bounded-wait error exit (its cluster and the blocks that wait leave on the flag)
  int stall = 0;
  // the same for the first FP64 sweep: block 0 waits on a flag nothing sets, the
  // blocks whose work items need its columns leave on the error flag
  int stall64 = 0;
  long long stall_ns = 0;
};
// Y <- X R^{-1} for upper R with inverted diagonal blocks (cholesky_upper_batched output)
cudaError_t trsm_right_upper_batched(const double* X, int64_t ldx, const CholBuffers& b, double* Y,
                                     int64_t strideY, double* tmp, int64_t strideTmp, int64_t m,
                                     int64_t n, int r, cudaStream_t st);
int eig_sym_jacobi(const double* H, int64_t ldh, int64_t n, double* V, int64_t ldv, double* lam_out,
                   const EigWork& w, int* sweeps, cudaStream_t st);
cudaError_t column_norms(const double* X, int64_t ldx, int64_t m, int64_t n, double* out,
                         cudaStream_t st);
cudaError_t scale_columns(double* X, int64_t ldx, int64_t m, int64_t n, const double* s, int invert,
                          cudaStream_t st);
cudaError_t column_dots(const double* A, int64_t lda, const double* B, int64_t ldb, int64_t m,
                        int64_t n, double* out, cudaStream_t st);
cudaError_t gather_columns(const double* X, int64_t ldx, double* Y, int64_t ldy, int64_t m,
                           int64_t n, const int* perm, const double* sign, cudaStream_t st);
// X = *scale R^T (lower triangular, zero above)
cudaError_t transpose_lower(const double* R, int64_t ldr, double* X, int64_t ldx, int64_t n,
                            const double* scale, cudaStream_t st);
// One FP64 sweep of the one-sided Jacobi rounds (a cooperative launch; ver holds
// n_even round counters, err the bounded waits' flag).
cudaError_t jacobi_sweep(double* X, int64_t ldx, int64_t m, int64_t n_even, int64_t n_real,
                         double tol, int* status, double* nrm2, double* dsc, int* ver, int* err,
                         int stall, long long stall_ns, cudaStream_t st);

#endif  // __CUDACC__

}  // namespace zolo
