// Internal declarations shared by the solver's translation units.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>
#include <stdio.h>

#include "device_once.cuh"
#include "gep.h"

#define GEP_IX(i, j, ld) ((size_t)(i) + (size_t)(j) * (size_t)(ld))

struct gep_handle_s {
  cudaStream_t stream = nullptr;
  int* d_status = nullptr;   // [0] numerical info, [1] error code (timeouts etc.)
  char* ws = nullptr;        // caller workspace
  size_t ws_bytes = 0;
  char* eng_ws = nullptr;    // scratch of the split-BF16 product engine
  size_t eng_bytes = 0;
  double* d_splitk = nullptr;     // handle-owned partial tiles of FP64 products with a split depth
  int* d_splitk_count = nullptr;  // arrivals per output tile, zero between products
  long long launches = 0;
  int sm_count = 152;
  // bounded device-side waits: their limit, and a test hook that drops the progress
  // releases of one bulge-chasing sweep so that the waits behind it run out
  unsigned long long wait_limit_ns = 4000000000ull;
  int fault_drop_sweep = -1;
  // test hook: rows per CTA of the single-launch panel QR (64, 128 or 256), -1 for the
  // one-launch-per-column kernel, 0 for the automatic choice
  int pqr_rows = 0;
  int band_group_min = -1;  // trailing order from which S1b takes panels in groups of four (-1: default)
  // test hooks: the cluster kernels decline, and every pencil that may takes the one-CTA solver
  int no_clusters = 0, force_one_cta = 0;
  int magic = 0x6e70;
  cudaEvent_t ev[8] = {};
  cudaEvent_t ev_band = nullptr;  // between full->band and bulge chasing (two-stage, timers on)
  // second stream of the solve: the dense Q2 tiles are built there while the tridiagonal
  // eigensolver runs on the handle's stream (fork/join by events)
  cudaStream_t side = nullptr;
  cudaEvent_t ev_fork = nullptr, ev_join = nullptr;
  bool band_recorded = false;
  bool timers_recorded = false;
  // optional per-launch timing of the tensor-core product kernel
  int prof_on = 0;
  int prof_cap = 0, prof_used = 0;
  long long prof_skipped = 0;
  cudaEvent_t* prof_ev = nullptr;   // 2 * prof_cap events
  double* prof_flops = nullptr;     // tensor flops of each recorded launch
  double* prof_f64eq = nullptr;     // FP64-equivalent flops of each recorded launch
  int* prof_mnk = nullptr;          // m, n, k of each recorded launch
  // batched solves: child handles, one per concurrent stream (created on first use)
  int nchild = 0;
  gep_handle_s* child[64] = {};
  cudaStream_t child_stream[64] = {};
  cudaEvent_t child_done[64] = {};
  cudaEvent_t fork_ev = nullptr;
  int* d_batch_info = nullptr;  // 2 ints per pencil of the last batched call
  int* d_small_next = nullptr;  // work-queue counter of the one-CTA small-pencil launch
  int batch_count = 0;
  int refine_steps = 0;  // FP64 refinement steps taken by the last mixed-precision solve
};

namespace gep {

constexpr int STATUS_EXPONENTS = 16;  // ints of the status block: exponents of A, B and C of a solve
constexpr int STATUS_SCRATCH = 20;    // and four ints of scratch for them

// Bump allocator over the caller's workspace.
struct Arena {
  char* base;
  size_t cap, off = 0;
  bool ok = true;
  Arena(void* b, size_t c) : base((char*)b), cap(c) {}
  template <class T>
  T* take(size_t n) {
    size_t a = (off + 255) & ~(size_t)255;
    size_t need = a + n * sizeof(T);
    if (need > cap || base == nullptr) { ok = false; off = need; return nullptr; }
    off = need;
    return (T*)(base + a);
  }
};

// Counting-only arena: used by workspace queries to size the same carving.
inline size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

inline int check_launch(gep_handle_t h) {
  h->launches++;
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) {
    fprintf(stderr, "gep: kernel launch failed: %s\n", cudaGetErrorString(e));
    return GEP_ERR_CUDA;
  }
  return GEP_OK;
}

#define GEP_CHECK(x)                        \
  do {                                      \
    int _r = (x);                           \
    if (_r != GEP_OK) return _r;            \
  } while (0)

#define GEP_CUDA(x)                                                                  \
  do {                                                                               \
    cudaError_t _e = (x);                                                            \
    if (_e != cudaSuccess) {                                                         \
      fprintf(stderr, "gep: %s failed: %s (%s:%d)\n", #x, cudaGetErrorString(_e), __FILE__, \
              __LINE__);                                                             \
      return GEP_ERR_CUDA;                                                           \
    }                                                                                \
  } while (0)

// Kernel attributes (the dynamic shared-memory limit) and what can be resident belong to a device context: one
// static of these per call site.
inline int current_device() {
  int d = -1;
  return cudaGetDevice(&d) == cudaSuccess ? d : -1;
}
template <class F>
int once_per_device(DeviceOnce& once, F&& f) {
  return once.run(current_device(), f);
}

// Whether a cluster of this size of the kernel can be resident at all.
inline bool cluster_fits(DeviceValue& known, const void* kernel, int cluster, int threads, size_t smem) {
  int fits = 0;
  known.get(current_device(), &fits, [&](int* v) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(cluster);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = cluster;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) != cudaSuccess) {
      cudaGetLastError();
      n = 0;
    }
    *v = n > 0;
    return 0;
  });
  return fits != 0;
}

constexpr int SPLITK_TILES = 2048;          // output tiles of a product with a split depth
constexpr int SPLITK_DOUBLES = 1 << 18;     // doubles of their partial tiles

// ---- dense contraction engines (gemm_f64.cu, gemm_oz.cu) ----
// Structure of op(A) a product may exploit: rows [128 r, 128 r + 128) of op(A) are exactly
// zero outside the columns [lo[r], hi[r]) for r < n (the other row blocks are dense).  The
// split-BF16 engine skips the zero part (same result bits); the FP64 engine ignores it.
constexpr int OZ_KR_MAX = 32;
struct OzKRange {
  int n = 0;
  int lo[OZ_KR_MAX], hi[OZ_KR_MAX];
};
// C = alpha op(A) op(B) + beta C; uplo 'L' restricts computation/storage to i >= j.
int dgemm(gep_handle_t h, char ta, char tb, char uplo, int m, int n, int k, double alpha,
          const double* A, int lda, const double* B, int ldb, double beta, double* C, int ldc,
          int engine, const OzKRange* kr = nullptr);
// Whether dgemm takes the split-BF16 engine for this product (gemm_f64.cu).
bool product_on_tensor_cores(gep_handle_t h, char uplo, int m, int n, int k, int engine);
int dgemm_f64(gep_handle_t h, char ta, char tb, char uplo, int m, int n, int k, double alpha,
              const double* A, int lda, const double* B, int ldb, double beta, double* C, int ldc);
// C_z += A_z B_z for a batch of equal products (split-BF16, FP64 setting).
int dgemm_oz_batched(gep_handle_t h, int m, int n, int k, const double* A, int lda, long long sa, const double* B,
                     int ldb, long long sb, double* C, int ldc, long long sc, int count);
// The same product through residues (gemm_res.cu): where it is the faster form, and the product itself
// (GEP_ERR_ALLOC / GEP_ERR_UNSUPPORTED before any work if the scratch is too small or C overlaps an operand).
bool res_product_wins(gep_handle_t h, char uplo, int m, int n, int k);
size_t res_workspace_bytes(int m, int n, int k);
int dgemm_res(gep_handle_t h, char ta, char tb, char uplo, int m, int n, int k, double alpha, const double* A,
              int lda, const double* B, int ldb, double beta, double* C, int ldc);
int dgemm_oz(gep_handle_t h, char ta, char tb, char uplo, int m, int n, int k, double alpha,
             const double* A, int lda, const double* B, int ldb, double beta, double* C, int ldc,
             int levels, const OzKRange* kr = nullptr);
size_t oz_workspace_bytes(int m, int n, int k);
// Digit planes of a symmetric operand (the lower triangle of an m x m matrix), split once
// so that several products can share them (the C22 products of a panel group in the full ->
// band reduction): plane s, row r at planes + (s m + r) ldk; the row exponent fields of K panel
// p (OZ_SYM_KP columns) at ea + p m.
constexpr int OZ_SYM_KP = 4096;
struct OzSymPlanes {
  unsigned short* planes = nullptr;
  int* ea = nullptr;
  int m = 0, ldk = 0, levels = 0;
};
size_t oz_sym_planes_bytes(int m, int levels);
int oz_split_sym(gep_handle_t h, int m, const double* A, int lda, int levels, void* buf, size_t bytes,
                 OzSymPlanes* P);
// C (m - row0 x n) = alpha A(row0:m, 0:m) B + beta C with A given by its planes P (B is
// m x n, column-major, ld ldb): rows row0.. of the symmetric operand against all of K.  parts:
// oz_sym_part_elems(P.m, n) doubles for the partial products of a split depth.
size_t oz_sym_part_elems(int m, int n);
int dgemm_oz_sym_planes(gep_handle_t h, const OzSymPlanes& P, int row0, int n, double alpha, const double* B,
                        int ldb, double beta, double* C, int ldc, double* parts, size_t part_elems);

// ---- small dense helpers (blas_util.cu) ----
int copy_matrix(gep_handle_t h, int m, int n, const double* src, int lds, double* dst, int ldd);
int copy_lower(gep_handle_t h, int M, const double* src, int lds, double* dst, int ldd);
int set_matrix(gep_handle_t h, int m, int n, double offdiag, double diag, double* A, int lda);
// *ex (zero on entry) := largest exponent field of the lower triangle of A
int max_exponent(gep_handle_t h, int M, const double* A, int lda, int* ex);
// *ex := exponent field of the power of two nearest to ||A||_F / (2 sqrt(M)) (0 for a zero matrix), A symmetric, lower
int norm_exponent(gep_handle_t h, int M, const double* A, int lda, int* ex);
// lower triangle (cols = m) or vector (cols = 1): dst = src 2^(*up - *down), device exponent fields, null: that of 1
int scale_pow2(gep_handle_t h, int m, int cols, const double* src, int lds, double* dst, int ldd, const int* up,
               const int* down);
int symmetrize_lower(gep_handle_t h, int M, double* A, int lda);  // upper := lower^T
int transpose(gep_handle_t h, int m, int n, const double* src, int lds, double* dst, int ldd);
int zero_upper(gep_handle_t h, int M, double* A, int lda);          // strict upper := 0
int symmetric_part(gep_handle_t h, int M, const double* W, int ldw, double* X, int ldx);  // X = (W + W^T) / 2
// X(:, j) *= d_j^-1/2 (m x n); first records the number of d_j <= 0 as numerical status k > 0
int scale_cols_rsqrt_checked(gep_handle_t h, int m, int n, const double* d, double* X, int ldx);
int scan_nonfinite(gep_handle_t h, int M, const double* A, int lda);  // lower triangle

// ---- triangular building blocks (tri.cu) ----
constexpr int TRI_NB = 256;  // order of the inverted diagonal blocks
// Inverts every nb x nb diagonal block of the lower triangular L into invD
// (block b at invD + b*nb*nb, column-major nb x nb, lower; ragged last block padded
// with identity).
int tri_inv_diag_blocks(gep_handle_t h, int M, const double* L, int ldl, double* invD, int nb);
// X (M x n) := L^-1 X  (left, lower, no transpose)
int trsm_lln(gep_handle_t h, int M, int n, const double* L, int ldl, const double* invD, int nb,
             double* X, int ldx, double* tmp, int engine);
// X (M x n) := L^-T X  (left, lower, transpose)
int trsm_llt(gep_handle_t h, int M, int n, const double* L, int ldl, const double* invD, int nb,
             double* X, int ldx, double* tmp, int engine);
size_t trsm_tmp_elems(int M, int n, int nb);

// ---- stages ----
int cholesky(gep_handle_t h, int M, double* B, int ldb, double* ws_invdiag, int engine);
int reduce_twosided(gep_handle_t h, int M, double* A, int lda, const double* L, int ldl,
                    const double* invD, double* X, double* tmp, int engine);
int reduce_explicit_inv(gep_handle_t h, int M, double* A, int lda, double* L, int ldl,
                        const double* invD, double* X, double* tmp, int engine);
// QR of a panel of at most 32 columns with its T factor in one cluster (panel_cluster.cu).
bool panel_qr_cluster_takes(int n, int nb);
int panel_qr_cluster(gep_handle_t h, int n, int nb, double* P, int ldp, double* tau, double* Va, double* Vb, int r0,
                     int ldv, double* T, const int* wide);
// Small trailing matrices of it in one cluster (tridiag_cluster.cu).
bool tridiag_cluster_takes(int n);
int tridiag_cluster(gep_handle_t h, int n, double* C, int ldc, double* d, double* e, double* tau);
int tridiag_1stage(gep_handle_t h, int M, double* C, int ldc, double* d, double* e, double* tau,
                   double* ws, size_t ws_elems, int engine);
size_t tridiag_ws_elems(int M);
int backtransform_q(gep_handle_t h, int M, int ncol, const double* C, int ldc, const double* tau,
                    double* Z, int ldz, double* ws, size_t ws_elems, int engine, int off = 1);
// T (nb x nb, upper) of the block reflector whose Gram matrix is G = V^T V (backtrans.cu).
int larft_rec(gep_handle_t h, int nb, const double* G, int ldg, const double* tau, double* T, int ldt,
              double* tmp, int engine);
// two-stage SEP path (band.cu)
size_t q2_elems(int M, int b);
size_t band_ws_elems(int M, int b);
int band_reduce(gep_handle_t h, int M, double* C, int ldc, int b, double* tau1, double* ws, size_t ws_elems,
                int eng);
int band_to_tridiag(gep_handle_t h, int M, const double* C, int ldc, int b, double* d, double* e, double* q2,
                    double* ws, size_t ws_elems);
size_t q2_tile_ws_elems(int M, int b);
int apply_q2(gep_handle_t h, int M, int b, const double* q2, double* Z, int ldz, int ncol, int engine, double* ws,
             size_t ws_elems, const double* U_all = nullptr);
// every dense Q2 tile at once (tensor-core engines), e.g. on a second stream
size_t q2_all_tiles_elems(int M, int b);
int build_q2_tiles(gep_handle_t h, cudaStream_t stream, int M, int b, const double* q2, double* U);
size_t backtransform_ws_elems(int M, int ncol);
int tridiag_eig_dc(gep_handle_t h, int M, const double* d, const double* e, double* w, double* Z,
                   int ldz, double* ws, size_t ws_elems, int engine);
size_t dc_ws_bytes(int M);
int tridiag_eig_bisect(gep_handle_t h, int M, const double* d, const double* e, double* w, int n = -1);
int sign_convention(gep_handle_t h, int M, int ncol, double* Y, int ldy);
size_t refine_ws_elems(int M);
int refine_eigenpairs(gep_handle_t h, int M, const double* Af, const double* Bf, double* X, int ldx, double* w,
                      double* ws, int iters, int engine);
size_t adjoint_ws_elems(int M, int no);
int adjoint(gep_handle_t h, int M, int no, const double* w, const double* Y, int ldy, const double* lbar,
            const double* W, int ldw, double* Abar, double* Bbar, int ldab, double* ws, int engine);

// block-Jacobi SEP solver (jacobi.cu)
size_t jacobi_ws_elems(int M);
int jacobi_sep(gep_handle_t h, int M, double* C, int ldc, double* w, double* Z, int ldz, double* ws);

// small pencils of a batched solve, one CTA each in one persistent launch (batched.cu)
constexpr int SMALL_MAX = 128;         // largest order solved by one CTA
constexpr int SMALL_PER_LAUNCH = 256;  // pencils whose table one launch carries in its parameters
size_t small_gep_scratch_bytes(int ctas);
int small_gep_batched(gep_handle_t h, cudaStream_t s, int count, const int* M, double* const* A, double* const* B,
                      double* const* w, double* const* Y, const int* order, double* scratch, int ctas, int* next,
                      int* info);

// A column whose sum of squares (alpha's included) lies below 2^-1010 is taken as zero beside its first entry (H = I):
// squares that underflow would give a reflector that is not orthogonal.  Its entries are below 2^-505.  (Compared
// as integers: an FP64 instruction holds a scheduler for 64 clocks.)
__device__ __forceinline__ bool tiny_squares(double n2) { return __double2hiint(n2) < (13 << 20); }

// Kernel-side helper: returns true when an earlier stage recorded an error.
__device__ __forceinline__ bool status_bad(const int* st) { return st != nullptr && (st[0] != 0 || st[1] != 0); }

}  // namespace gep
