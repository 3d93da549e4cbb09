// Per-call device context and the internal launch interface of libchase.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <vector>

#include "common.cuh"

namespace chase {

// A block of workspace for the buffers of one product after the other on one
// stream: taken in turn, and all of it free again once each has been released.
struct Arena {
  unsigned char* base = nullptr;
  size_t size = 0, at = 0;
  int live = 0;
};

// Device context of one ABI call: the stream, a device error flag and the
// stream-ordered workspace allocations, released when the context ends.
struct Dev {
  cudaStream_t st = nullptr;
  int* err = nullptr;  // device int, bit field of KERR_* codes
  struct Block {
    void* p;
    size_t bytes;
  };
  std::vector<Block> bufs;
  size_t held = 0;   // bytes of bufs
  size_t limit;      // chase_workspace_limit of the thread that made the context
  Arena* arena = nullptr;  // where allocations come from while they fit; borrowed
  // A view on another context's stream with a flag slot of its own (the
  // per-problem flags of a batch): err is borrowed, and leaving the view
  // does not synchronise (its workspace is released stream-ordered).
  bool own_err = true, sync_on_exit = true;

  explicit Dev(void* stream);
  Dev(const Dev&) = delete;
  Dev& operator=(const Dev&) = delete;
  ~Dev();

  int init();
  int alloc_bytes(void** p, size_t bytes);
  template <class T>
  int alloc(T** p, size_t count) {
    return alloc_bytes(reinterpret_cast<void**>(p), count * sizeof(T));
  }
  // Give an allocation of this context back before the context ends.
  void release(void* p);
  // Bytes that this context can still allocate.
  int free_bytes(size_t* bytes);
  // Synchronise the stream and turn the device error flag into a status.
  int sync_check(const char* where);
};

bool is_device_ptr(const void* p);

// Records a CUDA event pair on stream `s` around product launches while
// chase_kernel_timing is on (a no-op otherwise).  end() gives the launches
// the range covered and their algorithmic (FP64-equivalent) and executed
// tensor FLOPs; a timer destroyed without end() records nothing.
class KernelTimer {
 public:
  KernelTimer(cudaStream_t s, int kind);
  ~KernelTimer();
  KernelTimer(const KernelTimer&) = delete;
  KernelTimer& operator=(const KernelTimer&) = delete;
  void end(long long launches, double flops, double tensor_flops);

 private:
  cudaStream_t st_;
  int kind_;
  cudaEvent_t a_ = nullptr, b_ = nullptr;
  bool active_ = false;
};

// 2-D copies of column-major complex128 blocks (rows x cols).
int copy_block(Dev& d, chase_c64* dst, int64_t ldd, const chase_c64* src, int64_t lds, int64_t rows,
               int64_t cols, cudaMemcpyKind kind);
int copy_block(Dev& d, double* dst, int64_t ldd, const double* src, int64_t lds, int64_t rows,
               int64_t cols, cudaMemcpyKind kind);
int copy_block(Dev& d, chase_c32* dst, int64_t ldd, const chase_c32* src, int64_t lds, int64_t rows,
               int64_t cols, cudaMemcpyKind kind);
int copy_block(Dev& d, float* dst, int64_t ldd, const float* src, int64_t lds, int64_t rows,
               int64_t cols, cudaMemcpyKind kind);

// ---- kernels.cu ------------------------------------------------------------
// Element launchers are templates over the scalar T: chase_c64 (Hermitian
// problems) or double (real symmetric ones); both are instantiated.
// Stable counting sort of the degrees (warp-level match/popc scans):
// perm[pos] = original column at sorted position pos; start[i] = number of
// columns with degree < i (i = 0 .. max_deg + 1); info[0] = max degree.
int launch_filter_plan(Dev& d, const int* deg, int b, int max_allowed, int* perm, int* start,
                       int* info);
// Y[:, j] = X[:, perm[j]]  (gather) or Y[:, perm[j]] = X[:, j] (scatter)
template <class T>
int launch_permute_cols(Dev& d, const T* X, int64_t ldx, T* Y, int64_t ldy, int64_t N, int b,
                        const int* perm, bool scatter);
// out[j] = ||X[:, j]||_2
template <class T>
int launch_col_norms(Dev& d, const T* X, int64_t ldx, int64_t N, int b, double* out);
// out[0] = the largest magnitude of X as bits: the high word of a double's, an
// FP32 value's own; infinities and NaN above every finite one.
template <class T>
int launch_max_magnitude(Dev& d, const T* X, int64_t ldx, int64_t rows, int64_t cols, unsigned* out);
// X[:, j] *= 1 / s[j]   (s[j] == 0 leaves the column)
template <class T>
int launch_col_inv_scale(Dev& d, T* X, int64_t ldx, int64_t N, int b, const double* s);
// res[j] = ||HV[:, j] - lam[j] V[:, j]||_2
template <class T>
int launch_resid_norms(Dev& d, const T* HV, int64_t ldhv, const T* V, int64_t ldv, int64_t N, int b,
                       const double* lam, double* res);
// Upper triangle of the p x p matrix G <- conjugate of its lower triangle,
// diagonal made real: the Hermitian matrix that G's lower triangle defines.
template <class T>
int launch_fill_upper_hermitian(Dev& d, T* G, int64_t ldg, int p);
// G (p x p, its lower triangle) = L L^H becomes L^-H: upper triangular, zeros
// below the diagonal.  Sets KERR_CHOL_BREAKDOWN when a pivot is not above
// rel_tol * G_jj.  `shift` is added to the diagonal first; diag_ref: p doubles
// of workspace.
template <class T>
int cholesky_inverse(Dev& d, T* G, int64_t ldg, int p, double rel_tol, double shift,
                     double* diag_ref);
// R (p x p) = L^-H up to ||E||^2 for G = I + E (its lower triangle) = L L^H;
// e2[j]: the squared norm of column j of E's lower triangle.
template <class T>
int launch_near_identity(Dev& d, const T* G, int64_t ldg, int p, T* R, int64_t ldr, double* e2);
// One Lanczos three-term step on r independent runs (one CTA per run, run c
// in column c of each N x r block, leading dimension ld):
// alpha = Re(v^H w); w -= alpha v + beta_prev v_prev; beta = ||w||;
// v_next = w / beta (zero when beta <= tiny * the run's largest coefficient,
// i.e. rounding noise).  alpha/beta arrays are indexed [step * r + run].
template <class T>
int launch_lanczos_step(Dev& d, int64_t N, int64_t ld, int r, int step, const T* Vj,
                        const T* Vprev, T* W, T* Vnext, double* alpha, double* beta, double tiny);
// Normalise r columns in place (Lanczos start vectors).
template <class T>
int launch_normalize_cols(Dev& d, T* X, int64_t ldx, int64_t N, int r);
// F (n x n, ldf) = the Hermitian (real: symmetric) matrix whose lower
// triangle, diagonal included, is that of L; L's strict upper part is not read.
template <class T>
int launch_hermitian_from_lower(Dev& d, const T* L, int64_t ldl, T* F, int64_t ldf, int64_t n);
// dst (rows x cols, ldd) = src rounded to / widened from single precision.
int launch_convert(Dev& d, const chase_c32* src, int64_t lds, chase_c64* dst, int64_t ldd,
                   int64_t rows, int64_t cols);
int launch_convert(Dev& d, const chase_c64* src, int64_t lds, chase_c32* dst, int64_t ldd,
                   int64_t rows, int64_t cols);
int launch_convert(Dev& d, const float* src, int64_t lds, double* dst, int64_t ldd, int64_t rows,
                   int64_t cols);
int launch_convert(Dev& d, const double* src, int64_t lds, float* dst, int64_t ldd, int64_t rows,
                   int64_t cols);
// Fill the strict lower (lower=true) or upper part of a p x p matrix with zero.
template <class T>
int launch_zero_triangle(Dev& d, T* A, int64_t lda, int p, bool lower);
// Real Gram product C = X^T Y (X N x p, Y N x q) on the FP64 tensor pipe.
int dgram(Dev& d, int64_t N, const double* X, int64_t ldx, int p, const double* Y, int64_t ldy,
          int q, double* C, int64_t ldc, bool lower = false);
inline int gram(Dev& d, int64_t N, const chase_c64* X, int64_t ldx, int p, const chase_c64* Y,
                int64_t ldy, int q, chase_c64* C, int64_t ldc, bool lower = false) {
  return zgram(d, N, X, ldx, p, Y, ldy, q, C, ldc, lower);
}
inline int gram(Dev& d, int64_t N, const double* X, int64_t ldx, int p, const double* Y,
                int64_t ldy, int q, double* C, int64_t ldc, bool lower = false) {
  return dgram(d, N, X, ldx, p, Y, ldy, q, C, ldc, lower);
}
int cgram(Dev& d, int64_t N, const chase_c32* X, int64_t ldx, int p, const chase_c32* Y,
          int64_t ldy, int q, chase_c32* C, int64_t ldc, bool lower = false);
int sgram(Dev& d, int64_t N, const float* X, int64_t ldx, int p, const float* Y, int64_t ldy,
          int q, float* C, int64_t ldc, bool lower = false);
inline int gram(Dev& d, int64_t N, const chase_c32* X, int64_t ldx, int p, const chase_c32* Y,
                int64_t ldy, int q, chase_c32* C, int64_t ldc, bool lower = false) {
  return cgram(d, N, X, ldx, p, Y, ldy, q, C, ldc, lower);
}
inline int gram(Dev& d, int64_t N, const float* X, int64_t ldx, int p, const float* Y,
                int64_t ldy, int q, float* C, int64_t ldc, bool lower = false) {
  return sgram(d, N, X, ldx, p, Y, ldy, q, C, ldc, lower);
}

// ---- rns.cu: products with H in residue arithmetic on the tensor cores -----
// Moduli per accuracy: kRnsFp64 stands in for FP64 GEMMs (operands rounded to
// 2^-60 of a row's or column's 2-norm), rns_split_moduli for the split filter
// (2^-48, or 2^-52), kRnsSplitRR for a single product that replaces one at FP64
// accuracy (H Q of CHASE_SPLIT_BF16_RR; 2^-52), rns_low_moduli(N) for the
// filter's reduced precisions and for single precision (2^-30).
constexpr int kRnsMaxModuli = 14;
constexpr int kRnsFp64 = 14;
constexpr int kRnsSplitRR = 12;
int rns_split_moduli(int64_t N, bool cplx, int least_degree = 8);
int rns_low_moduli(int64_t N);
// Residue planes of H (per modulus two planes of N x Kp bf16 for complex H,
// one for real), row exponents and the real diagonal, which the epilogue
// applies in FP64.  sym: all rows share one scale, 2^exponent; complex H has one
// plane per modulus too, the other being its transpose, and real H's planes
// hold the lower triangle and the 256 x 256 blocks on the diagonal.  resident < nmod: memory holds only that many moduli at a
// time, and every product slices H anew (src, lds) for each group of them.
struct RnsH {
  void* A = nullptr;
  int* E = nullptr;
  double* Dg = nullptr;
  int64_t N = 0, Kp = 0;
  int cplx = 1, nmod = 0, resident = 0;
  const void* src = nullptr;
  int64_t lds = 0;
  int src_kind = 0;  // 0 complex128, 1 float64, 2 complex64, 3 float32
  int sym = 0, exponent = 0;
};
// Workspace for up to cap_cols columns at a time: residue planes of the block
// (B), of the product (G), column exponents.
struct RnsX {
  void* B = nullptr;
  int16_t* G = nullptr;
  int* F = nullptr;
  int cap_cols = 0, planes = 0;
  int64_t Kp = 0, ldg = 0;
  int flip = 0;  // which half of F (2 cap_cols) the residues in B belong to
};
// most: moduli resident at most.  reserve: bytes to leave free.  many: the planes
// serve many products, which pays for looking whether one scale fits all rows
// (a pass over H and a synchronisation).  CHASE_OUT_OF_MEMORY leaves nothing
// behind, of the workspace (rns_alloc_x) either.
bool rns_sym_pays(int planes, double entries);  // of H's, or of a whole batch's
template <class T>
int rns_prepare_h(Dev& d, const T* H, int64_t N, int64_t ldh, int nmod, int most, size_t reserve,
                  bool many, RnsH& out);
int rns_alloc_x(Dev& d, int64_t N, int max_cols, int max_moduli, bool cplx, RnsX& out);
void rns_release(Dev& d, RnsH& h);
void rns_release(Dev& d, RnsX& x);
// C[:, j0:j1] = alpha (H X[:, j0:j1] - shift X[:, j0:j1]) + beta C[:, j0:j1].
// Chained products (where rns_chains allows it for the widest): next0 >= 0
// leaves the residues of C[:, next0:j1] in x, and a product with sliced takes
// those as X[:, j0:j1] for its j0 = next0.
bool rns_chains(const RnsH& h, int b, const RnsX& x);
template <class T>
int rns_product(Dev& d, const RnsH& h, RnsX& x, const T* X, int64_t ldx, int j0, int j1, T* C,
                int64_t ldc, double alpha, double beta, double shift, bool sliced = false,
                int next0 = -1);

// Products of tall blocks (orthogonalisation, Rayleigh-Ritz) at FP64 accuracy.
// n vectors of K entries in residue planes: the columns of a block, or its rows.
// Memory comes with the vectors and goes with rns_release; CHASE_OUT_OF_MEMORY
// leaves nothing behind and nothing changed.
struct RnsBlock {
  void* P = nullptr;
  int* E = nullptr;
  int64_t n = 0, K = 0, Kp = 0;
};
template <class T>
int rns_columns(Dev& d, const T* X, int64_t ldx, int64_t K, int n, RnsBlock& out);
template <class T>
int rns_rows(Dev& d, const T* X, int64_t ldx, int64_t M, int K, RnsBlock& out);
void rns_release(Dev& d, RnsBlock& b);
// C[r, c] = alpha sum_k (a_r or conj(a_r))[k] b_c[k] + beta C[r, c]
template <class T>
int rns_dense(Dev& d, const RnsBlock& a, bool conj_a, const RnsBlock& b, T* C, int64_t ldc,
              double alpha, double beta);

// alpha P, beta and shift of one residue product, prepared on the host.
struct RnsScale {
  double alpha, beta, shift;
  double ap, ap_lo;  // 2^-64 alpha P as the sum of two doubles
  int plain;         // |alpha| within [2^-100, 2^100]: alpha P 2^e may be formed first
  int has_beta;
  float apf, apf_lo, bf, bf_lo;  // ap and beta as sums of two floats
  int single;                    // those are in FP32's range
};

// ---- grouped filter: many independent problems per launch ----------------
// One problem of a grouped filter, in device memory.  buf0 holds the block
// sorted by degree (the filter's input and final output), buf1 is the second
// buffer of the three-term recurrence.  Tensor maps live in device memory too:
// of H and both buffers for FP64 tiles, of the residue planes of H and of the
// active block for residue products.
struct GroupedProblem {
  const CUtensorMap* mapA;   // H, or the residue planes of H
  const CUtensorMap* mapB0;  // FP64: buf0; residues: the block's planes, a map per tile width
  const CUtensorMap* mapB1;  // FP64: buf1
  double2* buf0;
  double2* buf1;
  long long ld0, ld1;
  const int* E;       // residues: row exponents of H
  int* F;             // residues: column exponents of the active block
  const double* Dg;   // residues: real diagonal of H
  void* Bsl;          // residue planes of the block [plane][bcap][Kp] (bf16)
  void* G;            // residues of the product, the same shape (int16)
  long long Kp;       // residues: n rounded up to 64
  int n, b, bcap;     // rows, columns of the block, column capacity of Bsl and G
  int sym;            // residues: as RnsH
};
// One active problem of one degree step: columns [s, b) of problem `prob`
// are filtered; its output tiles are [tile0, next.tile0), its columns
// [col0, next.col0) of the step's column range and its reconstruction blocks
// [blk0, next.blk0).  A step's list ends with a sentinel entry holding the
// totals.
struct GroupedStep {
  int prob, s, tile0, col0, blk0;
  double alpha, beta, shift;
  RnsScale sc;
};
// FP64 tile shapes of the grouped product (rows x complex columns per CTA).
constexpr int kGroupedFp64Cfgs = 4;
void grouped_fp64_tile(int cfg, int* bm, int* bn);
// One degree step of the FP64 grouped filter: X = parity ? buf1 : buf0,
// Y = the other buffer.
int zgemm_grouped_fp64(Dev& d, int cfg, const GroupedProblem* probs, const GroupedStep* steps,
                       int nact, int ntiles, int parity);
// Kernel attributes (shared memory size) set outside any stream capture.
int zgemm_grouped_fp64_prepare(int cfg);
// Residue planes of every problem's H: one CTA per row over all problems;
// row0 is the first global row of each problem.
struct GroupedSliceH {
  const double2* H;
  long long ldh;
  void* A;
  int* E;
  double* Dg;
  long long Kp;
  int n, row0, tile0;  // first global row, first global 64 x 64 tile
  int s;               // the rows' common exponent (sym)
};
int64_t rns_k_padded(int64_t N);
// Row exponents of every H, and their least and largest in minmax (per problem);
// rns_same_scale says whether these allow one scale for all rows.
int rns_grouped_row_exponents(Dev& d, int nmod, const GroupedSliceH* probs, int P, int total_rows,
                              int* minmax);
bool rns_same_scale(int lo, int hi);
int rns_sym_tiles(int64_t n);
// Planes of the problems with a scale per row, and of those with one scale.
int rns_grouped_prepare_h(Dev& d, int nmod, const GroupedSliceH* probs, int P, int total_rows);
int rns_grouped_prepare_sym(Dev& d, int nmod, const GroupedSliceH* probs, int P, int total_tiles);
int rns_grouped_maps(CUtensorMap* mapA, CUtensorMap* mapB, int nmod, int bn, bool sym, const void* A,
                     const void* B, int64_t n, int64_t b, int64_t bcap);
RnsScale rns_scale(int nmod, double alpha, double beta, double shift);  // complex problems
// Tiles (of width bn) and reconstruction blocks of one problem's step, and the
// relative time of a 64-wide K step of a tile.
int rns_grouped_tiles(int nmod, int bn, int n, int cols);
int rns_grouped_crt_blocks(int n, int cols);
double rns_stage_cost(int bn);
// One degree step on residue products: slice the active columns of every
// active problem, multiply, put the products together.
int rns_grouped_ready();  // kernel attributes, set outside any stream capture
int rns_grouped_slice_x(Dev& d, int nmod, const GroupedProblem* probs, const GroupedStep* steps,
                        int nact, int ncols, int parity);
// in_row: each pair takes tiles that follow one another, else they take turns
int rns_grouped_gemm(Dev& d, int nmod, int bn, const GroupedProblem* probs,
                     const GroupedStep* steps, int nact, int ntiles, bool in_row);
int rns_grouped_crt(Dev& d, int nmod, const GroupedProblem* probs, const GroupedStep* steps,
                    int nact, int nblocks, int parity);
// One problem of a grouped filter: the block X (b columns, sorted by
// ascending degree) is filtered in place with W as the second buffer;
// start[i] (host, i = 0 .. maxdeg + 1) counts the columns of degree < i.
// Residue products: the planes of H (A, E, Dg) and the workspace of bcap >= b
// columns (Bsl, G, F), as made by grouped_rns_prepare.
struct GroupedFilterInput {
  const chase_c64* H = nullptr;
  int64_t ldh = 0;
  int n = 0;
  chase_c64* X = nullptr;
  int64_t ldx = 0;
  chase_c64* W = nullptr;
  int64_t ldw = 0;
  int b = 0;
  const int* start = nullptr;
  int maxdeg = 0;
  double b_sup = 0, mu1 = 0, mu_nn = 0;
  void* A = nullptr;
  int* E = nullptr;
  double* Dg = nullptr;
  void* Bsl = nullptr;
  void* G = nullptr;
  int* F = nullptr;
  int bcap = 0, sym = 0;
};
struct GroupedFilterTimes {
  int tile_config = -1, steps = 0, launches = 0;
  long long matvecs = 0;
  double flops = 0, t_autotune = 0, t_graph_build = 0, t_steps = 0, t_product = 0;
};
// Moduli of a batch's residue products: of the split filter's accuracy, or
// FP64's; 0 where the FP64 tiles take less time.
// rr: the planes serve H Q of CHASE_SPLIT_BF16_RR too.
int grouped_moduli(const std::vector<GroupedFilterInput>& in, bool split, int tile, bool rr = false);
// Residue planes of every problem's H and the workspace for bcap[q] columns
// (one grouped slicing launch), which leave `reserve` bytes free; fills the
// residue fields of `in`.  A status other than CHASE_OK leaves nothing behind.
struct GroupedWork {  // of all problems: their planes of H, and the rest
  void *block = nullptr, *planes = nullptr;
};
int grouped_rns_prepare(Dev& d, std::vector<GroupedFilterInput>& in, const std::vector<int>& bcap,
                        int nmod, size_t reserve, GroupedWork& w);
void grouped_rns_release(Dev& d, std::vector<GroupedFilterInput>& in, GroupedWork& w);
// Alg. 4 on every problem of `in` (problems with b == 0 are skipped), one
// grouped launch per degree step and part, all steps in one CUDA graph.
// nmod: residue products with that many moduli (prepared inputs are used as
// they are; others are prepared here, a part of the batch at a time where the
// memory does not hold all), 0: FP64 tiles of shape `tile` or, with
// CHASE_TILE_AUTO, the fastest.  Synchronises the stream.  With prepared inputs
// CHASE_OUT_OF_MEMORY leaves every block as it was.
int grouped_filter_sorted(Dev& d, const std::vector<GroupedFilterInput>& in, int nmod, int tile,
                          GroupedFilterTimes* times);

// Column gather / scatter for many problems: one CTA per column.
struct GroupedPermute {
  const double2* src;
  double2* dst;
  long long lds, ldd;
  const int* perm;
  int n, col0;
};
int launch_grouped_permute(Dev& d, const GroupedPermute* probs, int P, int total_cols, bool scatter);

// ---- eigh_refine.cu: the projected eigensolve of Alg. 2 line 3 ------------
// G (p x p, Hermitian, both triangles) becomes its eigenvectors, w_dev its
// eigenvalues ascending: FP64 problems by refining an FP32 solve, or where
// that does not serve with eigh_device; single precision with eigh_device.
int eigh(Dev& d, chase_c64* G, int64_t ldg, int p, double* w_dev);
int eigh(Dev& d, double* G, int64_t ldg, int p, double* w_dev);
int eigh(Dev& d, chase_c32* G, int64_t ldg, int p, double* w_dev);
int eigh(Dev& d, float* G, int64_t ldg, int p, double* w_dev);
// ---- the same by cuSOLVER alone -------------------------------------------
int eigh_device(Dev& d, chase_c64* G, int64_t ldg, int p, double* w_dev);
int eigh_device(Dev& d, double* G, int64_t ldg, int p, double* w_dev);
// Single precision (cheevd / ssyevd); eigenvalues returned in double.
int eigh_device(Dev& d, chase_c32* G, int64_t ldg, int p, double* w_dev);
int eigh_device(Dev& d, float* G, int64_t ldg, int p, double* w_dev);
// Many small projected eigenproblems at once (cuSOLVER's batched Hermitian
// eigensolver on buckets of sizes rounded up to 16, each matrix padded as
// diag(G, pad I)): item q's G (p x p, ldg, Hermitian, both triangles) is
// overwritten by its eigenvectors and w (p doubles, device) receives its
// eigenvalues ascending.  *info_dev (device, one int per item in bucket
// order) is nonzero where the eigensolver failed; the caller reads it after
// its next synchronisation.
struct EighItem {
  chase_c64* G;
  long long ldg;
  int p;
  double* w;
};
int eigh_batched(Dev& d, const std::vector<EighItem>& items, int** info_dev);
// Destroy the calling thread's cuSOLVER handle (worker threads, before they end).
void release_thread_solver();

// ---- host_alg.cpp ----------------------------------------------------------
// Symmetric tridiagonal eigenproblem (implicit QL with Wilkinson shifts):
// diag[k], off[k-1] -> eigenvalues ascending in w, eigenvectors (k x k,
// column-major) in z.  Returns false if it fails to converge.
bool tridiag_eigh(int k, const double* diag, const double* off, double* w, double* z);
// Alg. 6 line 11 (Eq. 10 quantile with its width safeguard); see
// chase_dos_estimate in chase.h.  halvings / fallback may be NULL.
double dos_estimate(int nruns, const int* steps, const double* theta, const double* w,
                    double target, double mu1, double b_sup, double dos_sigma, int* halvings,
                    bool* fallback);

}  // namespace chase
