// Reducer stages (section 3.1 (b)):
//   Eq. 4  B = L L^T              blocked right-looking Cholesky
//   Eq. 5  C = L^-1 A L^-T         "ScaLAPACK style" (triangular solves, L^-1 never formed)
//                                  "ELPA style" (R = L^-1 formed, then C = R A R^T)
//   Eq. 6  Y = L^-T Z              blocked back-substitution
// plus the triangular building blocks they share.  Every nb x nb diagonal block
// of L is factored and inverted by one cluster of CTAs; everything else is
// a dense product on the GEMM engine, so the O(M^3) work runs as matrix products.
#include <cooperative_groups.h>
#include <math.h>

#include "cluster.cuh"
#include "gep_internal.cuh"

namespace cg = cooperative_groups;

namespace gep {
namespace {

constexpr int NB = 128;  // diagonal block order

// In-place inverse of the r x r lower triangular S (shared, leading dim NB),
// from the bottom-right: column j of L^-1 is -(1/l_jj) * L22^-1 * l(j+1:, j).
__device__ void tri_inv_smem(double* S, double* tmp, int r) {
  // X = L^-1 column by column from the last: X(i, j) = -X(j, j) sum_{q=j+1..i} X(i, q) L(q, j),
  // columns q > j already inverted in place.  Two threads per row i (lanes 2i, 2i + 1 take
  // alternate q) halve the dependent FMA chain of each dot product.
  __shared__ double ajj_s;
  const int i = threadIdx.x >> 1, part = threadIdx.x & 1;
  for (int j = r - 1; j >= 0; --j) {
    __syncthreads();
    if (threadIdx.x == 0) ajj_s = 1.0 / S[j + j * NB];  // one division per column
    double s = 0.0, s2 = 0.0;  // two independent FMA chains per thread
    if (i > j && i < r) {
      int q = j + 1 + part;
      for (; q + 2 <= i; q += 4) {
        s = fma(S[i + q * NB], S[q + j * NB], s);
        s2 = fma(S[i + (q + 2) * NB], S[q + 2 + j * NB], s2);
      }
      if (q <= i) s = fma(S[i + q * NB], S[q + j * NB], s);
    }
    s += s2;
    s += __shfl_xor_sync(0xffffffffu, s, 1);
    if (part == 0 && i > j && i < r) tmp[i] = s;
    __syncthreads();
    const double ajj = ajj_s;
    if (part == 0 && i > j && i < r) S[i + j * NB] = -ajj * tmp[i];
    if (threadIdx.x == 0) S[j + j * NB] = ajj;
  }
  __syncthreads();
}

// Writes the r x r lower inverse from shared memory into an NB x NB block (identity
// padding for r < NB, zero strict upper triangle).
__device__ void store_inv(const double* S, int r, double* out, int ldo) {
  for (int idx = threadIdx.x; idx < NB * NB; idx += blockDim.x) {
    int i = idx % NB, j = idx / NB;
    double v;
    if (i < r && j < r) v = (i >= j) ? S[i + j * NB] : 0.0;
    else v = (i == j) ? 1.0 : 0.0;
    out[i + j * ldo] = v;
  }
}

// Cholesky factor of the diagonal block B(kb:kb+r, kb:kb+r) (already updated by earlier
// trailing products) in place, and its inverse L_kk^-1 into invD, by one cluster of 8 CTAs.
//
// Symmetric elimination on the augmented matrix [A | I], kept in place: row i holds A's
// columns c >= j and the growing inverse's columns c < j at step j.  Warp w of rank q owns row
// q + 8 w (cyclic, so every CTA keeps work to the end), lane l its columns l, l + 32, ... in
// registers.  Step j: every row i > j takes row_i -= f_i row_j with f_i = M(i, j) / p_j, and
// column j becomes -f_i; L(i, j) = f_i sqrt(p_j), and row j of the inverse is row_j / sqrt(p_j).
// The owner of a finished row pushes it, its pivot and 1 / pivot into the shared memory of all
// 8 CTAs (st.async, one mbarrier per row; every row has its own slot, so nothing is reused and
// no cluster barrier is needed inside the loop) and is done.
//
// Bound: the FP64 pipe (64 clocks a warp instruction) and the chain of 128 pivots.  On one SM
// the 0.7 M FMAs alone take 200 us; over 8 SMs they hide behind the chain, a step of which is
// the next row's 4 FMAs, the reciprocal of its pivot and the push.  The other warps of the CTA
// that owns the next row therefore wait for that row before they spend FP64 issue slots on this
// one.  A 128 x 128 block takes 123 us
// (0.95 us a pivot; one CTA working in shared memory took 636 us), a 64 x 64 one 68 us.
constexpr int PC = 8;            // CTAs of the cluster
constexpr int PW = NB / PC;      // rows per CTA = warps
constexpr int PROW = NB + 2;     // a published row: 128 values, 1 / pivot, pivot

struct PotrfShared {
  double rows[NB][PROW];           // row j at [lane * 4 + u] for column lane + 32 u
  double f[PW][NB];                // f_i of this CTA's rows
  double sq[NB], rs[NB];
  unsigned long long bar[NB];
  unsigned pushed;                 // bit w: the row of warp w has been pushed
};

__global__ void __cluster_dims__(PC, 1, 1) __launch_bounds__(32 * PW) k_potrf_diag(int r, double* B, int ldb,
                                                                                   double* invD, int ldi, int kb,
                                                                                   int* st) {
  extern __shared__ __align__(16) unsigned char smraw[];
  PotrfShared& sh = *reinterpret_cast<PotrfShared*>(smraw);
  constexpr int U = NB / 32;
  cg::cluster_group cl = cg::this_cluster();
  const int rank = cl.block_rank(), w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int i = rank + PC * w;
  const bool bad = status_bad(st);  // an earlier stage failed: every warp passes through
  if (threadIdx.x < NB) {
    const uint32_t bar = cta_shared(&sh.bar[threadIdx.x]);
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("{ .reg .b64 t; mbarrier.arrive.expect_tx.shared::cta.b64 t, [%0], %1; }" ::"r"(bar),
                 "r"(PROW * 8) : "memory");
  }
  if (threadIdx.x == 0) sh.pushed = 0;
  double x[U];
#pragma unroll
  for (int u = 0; u < U; ++u) {
    const int c = lane + 32 * u, a = max(i, c), b = min(i, c);
    x[u] = a < r ? B[GEP_IX(a, b, ldb)] : (i == c ? 1.0 : 0.0);
  }
  cl.sync();
  auto publish = [&](int j, double pivot) {
    const double ri = 1.0 / pivot;
    if (lane == 0) atomicOr(&sh.pushed, 1u << w);
    const uint32_t dst = cta_shared(&sh.rows[j][lane * U]), sc = cta_shared(&sh.rows[j][NB]), bar = cta_shared(&sh.bar[j]);
#pragma unroll
    for (int q = 0; q < PC; ++q) {
      uint32_t rd, rb, rsc;
      asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(rd) : "r"(dst), "r"(q));
      asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(rb) : "r"(bar), "r"(q));
#pragma unroll
      for (int u = 0; u < U; u += 2)
        asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v2.b64 [%0], {%1, %2}, [%3];" ::"r"(
                         rd + 8 * u), "l"(__double_as_longlong(x[u])), "l"(__double_as_longlong(x[u + 1])), "r"(rb)
                     : "memory");
      if (lane == q) {
        asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(rsc) : "r"(sc), "r"(q));
        asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v2.b64 [%0], {%1, %2}, [%3];" ::"r"(
                         rsc), "l"(__double_as_longlong(ri)), "l"(__double_as_longlong(pivot)), "r"(rb)
                     : "memory");
      }
    }
  };
  int fail = bad ? -1 : 0;
  if (i == 0 && !fail) publish(0, __shfl_sync(0xffffffffu, x[0], 0));
  const int last = i < r ? i : 0;  // rows past the block are identity rows: nothing to do
#pragma unroll
  for (int ju = 0; ju < U; ++ju) {
    for (int jl = 0; jl < 32; ++jl) {
      const int j = 32 * ju + jl;
      if (j >= last || fail) break;
      bool ok = true;
      if (rank == (j + 1) % PC && i != j + 1) ok = cluster_wait<false>(cta_shared(&sh.bar[j + 1]), 0, st);
      if (ok) ok = cluster_wait<false>(cta_shared(&sh.bar[j]), 0, st);
      if (!ok) { fail = -1; break; }
      const double ri = sh.rows[j][NB];  // a bad pivot is found at the end: the rows keep coming
      const double f = __shfl_sync(0xffffffffu, x[ju], jl) * ri;
#pragma unroll
      for (int u = 0; u < U; ++u) x[u] = fma(-f, sh.rows[j][lane * U + u], x[u]);
      if (lane == jl) x[ju] = -f;
      if (lane == 0) sh.f[w][j] = f;
      if (i == j + 1) {
        double piv = 0.0;
#pragma unroll
        for (int u = 0; u < U; ++u)
          if (u == (i >> 5)) piv = __shfl_sync(0xffffffffu, x[u], i & 31);
        publish(i, piv);
      }
    }
  }
  cl.sync();  // every row that is to come has been pushed
  // no CTA leaves before every push into its shared memory has landed (after a timeout some rows never come)
  if (threadIdx.x < NB) {
    const unsigned pushed = *cl.map_shared_rank(&sh.pushed, threadIdx.x % PC);
    if (!(pushed >> (threadIdx.x / PC) & 1) || !cluster_wait<true>(cta_shared(&sh.bar[threadIdx.x]), 0, st))
      sh.rows[threadIdx.x][NB + 1] = 0.0;  // not here: no pivot
  }
  cl.sync();
  if (bad) return;
  // the pivots; the first that is not positive is the leading minor reported
  __shared__ int first_bad;
  if (threadIdx.x == 0) first_bad = NB;
  __syncthreads();
  if (threadIdx.x < NB) {
    sh.rs[threadIdx.x] = sh.sq[threadIdx.x] = 1.0;
    if (threadIdx.x < r) {
      const double p = sh.rows[threadIdx.x][NB + 1];
      if (!(p > 0.0) || !isfinite(p)) {
        atomicMin(&first_bad, (int)threadIdx.x);
      } else {
        const double l = sqrt(p);
        sh.sq[threadIdx.x] = l;
        sh.rs[threadIdx.x] = 1.0 / l;
      }
    }
  }
  __syncthreads();
  if (first_bad < NB) {
    if (rank == 0 && threadIdx.x == 0) atomicCAS(st, 0, kb + first_bad + 1);
    return;
  }
  const double ri = sh.rs[i];
#pragma unroll
  for (int u = 0; u < U; ++u) {
    const int c = lane + 32 * u;
    if (i < r && c <= i) B[GEP_IX(i, c, ldb)] = c == i ? sh.sq[i] : sh.f[w][c] * sh.sq[c];
    invD[i + c * ldi] = c < i ? x[u] * ri : (c == i ? ri : 0.0);
  }
}

// One CTA per diagonal block of an existing lower triangular L: invert it.
__global__ void __launch_bounds__(256) k_inv_diag(int M, const double* L, int ldl, double* invD,
                                                  const int* st) {
  extern __shared__ double sm[];
  if (status_bad(st)) return;
  double* S = sm;
  double* tmp = sm + NB * NB;
  int b = blockIdx.x, kb = b * NB;
  int r = min(NB, M - kb);
  for (int idx = threadIdx.x; idx < r * r; idx += blockDim.x) {
    int i = idx % r, j = idx / r;
    S[i + j * NB] = (i >= j) ? L[GEP_IX(kb + i, kb + j, ldl)] : 0.0;
  }
  tri_inv_smem(S, tmp, r);
  // block b is the upper or lower diagonal half of an inverse block of TRI_NB
  constexpr int Q = TRI_NB / NB;
  store_inv(S, r, invD + (size_t)(b / Q) * TRI_NB * TRI_NB + GEP_IX(b % Q * NB, b % Q * NB, TRI_NB), TRI_NB);
}

constexpr size_t kSmemDiag = (size_t)NB * NB * sizeof(double) + NB * sizeof(double);

int set_smem_attr() {
  static DeviceOnce attributes;
  return once_per_device(attributes, []() -> int {
    GEP_CUDA(cudaFuncSetAttribute(k_potrf_diag, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(PotrfShared)));
    GEP_CUDA(cudaFuncSetAttribute(k_inv_diag, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemDiag));
    return GEP_OK;
  });
}

}  // namespace

size_t trsm_tmp_elems(int M, int n, int nb) { (void)M; return (size_t)nb * (size_t)(n > 0 ? n : 1); }

namespace {

// X21 = -X22 L21 X11 of a block of order n > NB whose diagonal halves are inverted in X (ld
// TRI_NB), and the zero above it; tmp holds NB x NB.
int inv_merge(gep_handle_t h, int n, const double* L21, int ldl, double* X, double* tmp, int engine) {
  const int n1 = NB, n2 = n - NB;
  GEP_CHECK(set_matrix(h, n1, n2, 0.0, 0.0, X + GEP_IX(0, n1, TRI_NB), TRI_NB));
  GEP_CHECK(dgemm(h, 'N', 'N', 'F', n2, n1, n1, 1.0, L21, ldl, X, TRI_NB, 0.0, tmp, n2, engine));
  return dgemm(h, 'N', 'N', 'F', n2, n1, n2, -1.0, X + GEP_IX(n1, n1, TRI_NB), TRI_NB, tmp, n2, 0.0, X + n1, TRI_NB,
               engine);
}

}  // namespace

int tri_inv_diag_blocks(gep_handle_t h, int M, const double* L, int ldl, double* invD, int nb) {
  if (nb != TRI_NB) return GEP_ERR_UNSUPPORTED;
  if (M <= 0) return GEP_OK;
  GEP_CHECK(set_smem_attr());
  int nblk = (M + NB - 1) / NB;
  k_inv_diag<<<nblk, 256, kSmemDiag, h->stream>>>(M, L, ldl, invD, h->d_status);
  GEP_CHECK(check_launch(h));
  double* tmp = invD + (size_t)((M + TRI_NB - 1) / TRI_NB) * TRI_NB * TRI_NB;
  for (int o = 0; o + NB < M; o += TRI_NB)
    GEP_CHECK(inv_merge(h, M - o < TRI_NB ? M - o : TRI_NB, L + GEP_IX(o + NB, o, ldl), ldl,
                        invD + (size_t)(o / TRI_NB) * TRI_NB * TRI_NB, tmp, GEP_PREC_FP64));
  return GEP_OK;
}

// All triangular solves and the Cholesky factorisation below recurse on halves whose
// split points are multiples of TRI_NB, down to the diagonal blocks of TRI_NB = 256 (leaf o covers
// rows o .. o+TRI_NB-1 and uses invD block o/TRI_NB; a block's factor and inverse come from two
// halves of NB).  With leaves of NB = 128 the solves took twice as many products, most of them
// 25 to 60 us of launches and splits (order 2047: reduction 7.0 -> 4.3 ms, back-substitution 1.25 ->
// 0.76 ms; order 8192: 47 -> 34 and 16.7 -> 15 ms).  The off-diagonal work is then a few
// products with a long inner dimension (n/2, n/4, ...), which the tensor-core engine
// runs near its best rate, instead of many rank-NB updates.
namespace {

int split_nb(int n) { return ((n / TRI_NB + 1) / 2) * TRI_NB; }

// rows [o, o+n) of X (X points at row o) := L(o:o+n, o:o+n)^-1 X
int lln_rec(gep_handle_t h, int o, int n, int ncol, const double* L, int ldl, const double* invD, double* X, int ldx,
            double* tmp, int engine) {
  if (n <= TRI_NB) {
    const double* Dk = invD + (size_t)(o / TRI_NB) * TRI_NB * TRI_NB;
    GEP_CHECK(dgemm(h, 'N', 'N', 'F', n, ncol, n, 1.0, Dk, TRI_NB, X, ldx, 0.0, tmp, n, engine));
    return copy_matrix(h, n, ncol, tmp, n, X, ldx);
  }
  int n1 = split_nb(n), n2 = n - n1;
  GEP_CHECK(lln_rec(h, o, n1, ncol, L, ldl, invD, X, ldx, tmp, engine));
  GEP_CHECK(dgemm(h, 'N', 'N', 'F', n2, ncol, n1, -1.0, L + GEP_IX(o + n1, o, ldl), ldl, X, ldx, 1.0, X + n1, ldx,
                  engine));
  return lln_rec(h, o + n1, n2, ncol, L, ldl, invD, X + n1, ldx, tmp, engine);
}

// rows [o, o+n) of X := L(o:o+n, o:o+n)^-T X
int llt_rec(gep_handle_t h, int o, int n, int ncol, const double* L, int ldl, const double* invD, double* X, int ldx,
            double* tmp, int engine) {
  if (n <= TRI_NB) {
    const double* Dk = invD + (size_t)(o / TRI_NB) * TRI_NB * TRI_NB;
    GEP_CHECK(dgemm(h, 'T', 'N', 'F', n, ncol, n, 1.0, Dk, TRI_NB, X, ldx, 0.0, tmp, n, engine));
    return copy_matrix(h, n, ncol, tmp, n, X, ldx);
  }
  int n1 = split_nb(n), n2 = n - n1;
  GEP_CHECK(llt_rec(h, o + n1, n2, ncol, L, ldl, invD, X + n1, ldx, tmp, engine));
  GEP_CHECK(dgemm(h, 'T', 'N', 'F', n1, ncol, n2, -1.0, L + GEP_IX(o + n1, o, ldl), ldl, X + n1, ldx, 1.0, X, ldx,
                  engine));
  return llt_rec(h, o, n1, ncol, L, ldl, invD, X, ldx, tmp, engine);
}

// X (m x n, columns o .. o+n of the factor) := X L(o:o+n, o:o+n)^-T
int rlt_rec(gep_handle_t h, int o, int n, int m, const double* L, int ldl, const double* invD, double* X, int ldx,
            double* tmp, int engine) {
  if (n <= TRI_NB) {
    const double* Dk = invD + (size_t)(o / TRI_NB) * TRI_NB * TRI_NB;
    GEP_CHECK(dgemm(h, 'N', 'T', 'F', m, n, n, 1.0, X, ldx, Dk, TRI_NB, 0.0, tmp, m, engine));
    return copy_matrix(h, m, n, tmp, m, X, ldx);
  }
  int n1 = split_nb(n), n2 = n - n1;
  GEP_CHECK(rlt_rec(h, o, n1, m, L, ldl, invD, X, ldx, tmp, engine));
  GEP_CHECK(dgemm(h, 'N', 'T', 'F', m, n2, n1, -1.0, X, ldx, L + GEP_IX(o + n1, o, ldl), ldl, 1.0,
                  X + (size_t)n1 * ldx, ldx, engine));
  return rlt_rec(h, o + n1, n2, m, L, ldl, invD, X + (size_t)n1 * ldx, ldx, tmp, engine);
}

// Eq. 4 on the diagonal block (o, o) of order n; B points at the full matrix.
int potrf_rec(gep_handle_t h, int o, int n, double* B, int ldb, double* invD, double* tmp, int engine) {
  if (n <= TRI_NB) {
    double* X = invD + (size_t)(o / TRI_NB) * TRI_NB * TRI_NB;
    const int n1 = n < NB ? n : NB, n2 = n - n1;
    auto leaf = [&](int at, int r) {
      k_potrf_diag<<<PC, 32 * PW, sizeof(PotrfShared), h->stream>>>(r, B + GEP_IX(o + at, o + at, ldb), ldb,
                                                                    X + GEP_IX(at, at, TRI_NB), TRI_NB, o + at, h->d_status);
      return check_launch(h);
    };
    GEP_CHECK(leaf(0, n1));
    if (n2 == 0) return GEP_OK;
    double* L21 = B + GEP_IX(o + n1, o, ldb);
    GEP_CHECK(dgemm(h, 'N', 'T', 'F', n2, n1, n1, 1.0, L21, ldb, X, TRI_NB, 0.0, tmp, n2, engine));  // A21 L11^-T
    GEP_CHECK(copy_matrix(h, n2, n1, tmp, n2, L21, ldb));
    GEP_CHECK(dgemm(h, 'N', 'T', 'L', n2, n2, n1, -1.0, L21, ldb, L21, ldb, 1.0, B + GEP_IX(o + n1, o + n1, ldb), ldb,
                    engine));
    GEP_CHECK(leaf(n1, n2));
    return inv_merge(h, n, L21, ldb, X, tmp, engine);
  }
  int n1 = split_nb(n), n2 = n - n1;
  GEP_CHECK(potrf_rec(h, o, n1, B, ldb, invD, tmp, engine));
  double* L21 = B + GEP_IX(o + n1, o, ldb);
  GEP_CHECK(rlt_rec(h, o, n1, n2, B, ldb, invD, L21, ldb, tmp, engine));   // L21 = A21 L11^-T
  GEP_CHECK(dgemm(h, 'N', 'T', 'L', n2, n2, n1, -1.0, L21, ldb, L21, ldb, 1.0, B + GEP_IX(o + n1, o + n1, ldb), ldb,
                  engine));                                                 // A22 -= L21 L21^T
  return potrf_rec(h, o + n1, n2, B, ldb, invD, tmp, engine);
}

}  // namespace

// X := L^-1 X (forward substitution); tmp holds TRI_NB x n doubles.
int trsm_lln(gep_handle_t h, int M, int n, const double* L, int ldl, const double* invD, int nb,
             double* X, int ldx, double* tmp, int engine) {
  if (nb != TRI_NB) return GEP_ERR_UNSUPPORTED;
  if (M <= 0 || n <= 0) return GEP_OK;
  return lln_rec(h, 0, M, n, L, ldl, invD, X, ldx, tmp, engine);
}

// X := L^-T X (backward substitution with the upper triangular L^T).
int trsm_llt(gep_handle_t h, int M, int n, const double* L, int ldl, const double* invD, int nb,
             double* X, int ldx, double* tmp, int engine) {
  if (nb != TRI_NB) return GEP_ERR_UNSUPPORTED;
  if (M <= 0 || n <= 0) return GEP_OK;
  return llt_rec(h, 0, M, n, L, ldl, invD, X, ldx, tmp, engine);
}

// Eq. 4: recursive Cholesky.  invD receives the inverses of the TRI_NB x TRI_NB diagonal
// blocks (reused by the reduction and the back-substitution).  tmp (M x TRI_NB doubles)
// follows invD in the caller's workspace.
int cholesky(gep_handle_t h, int M, double* B, int ldb, double* invD, int engine) {
  if (M <= 0) return GEP_OK;
  GEP_CHECK(set_smem_attr());
  int nblk = (M + TRI_NB - 1) / TRI_NB;
  double* tmp = invD + (size_t)nblk * TRI_NB * TRI_NB;
  return potrf_rec(h, 0, M, B, ldb, invD, tmp, engine);
}

// Eq. 5, "ScaLAPACK style": C = L^-1 A L^-T without forming L^-1, blocked over panels of
// nb columns and exploiting the symmetry of A and C (the blocking of ScaLAPACK's pdsygst):
// with the leading panel A11 (nb x nb), A21 below it and the trailing A22,
//     C11 = L11^-1 A11 L11^-T                       (two triangular solves of order nb)
//     A21 <- A21 L11^-T - 1/2 L21 C11
//     A22 <- A22 - A21 L21^T - L21 A21^T            (lower triangle, one product of depth 2 nb)
//     C21 = L22^-1 (A21 - 1/2 L21 C11)              (triangular solve with the trailing factor)
// and the trailing matrix is reduced the same way.  About M^3 flops in products (two
// thirds in the symmetric rank-2nb updates, one third in the solves), against 2 M^3 for two
// full triangular solves.  A (lower) is overwritten by the full symmetric C; X is an M x M
// scratch matrix, tmp a TRI_NB x M one.
int reduce_twosided(gep_handle_t h, int M, double* A, int lda, const double* L, int ldl,
                    const double* invD, double* X, double* tmp, int engine) {
  if (M <= 0) return GEP_OK;
  // Panel width: a multiple of TRI_NB (the triangular recursions split there), half the
  // matrix up to 2048.  Every panel is a chain of some twenty launches that depend on one another,
  // and its rank-2 nb update splits its operands anew; wide panels have fewer chains and give the
  // tensor engine deep products.  R2 at 1501 / 2047 / 3000 / 4000 / 6000 / 8192: with M / 8 up to
  // 1024 2.4 / 4.2 / 8.6 / 15.1 / 23.1 / 33.5 ms, with M / 3 up to 2048 2.4 / 3.0 / 5.3 / 7.9 /
  // 15.9 / 29.3 ms, so 1.8 / 2.8 / 4.7 / 7.6 / 14.8 / 29.2 ms; up to 4096 order 6000 takes 15.7 ms.
  // [A21 L21] and its twin need 4 (M - nb) nb <= M^2 numbers of X for every nb.
  int nbp = (M / 2) / TRI_NB * TRI_NB;
  if (nbp < TRI_NB) nbp = TRI_NB;
  if (nbp > 2048) nbp = 2048;
  for (int k = 0; k < M; k += nbp) {
    const int nb = (M - k) < nbp ? (M - k) : nbp, n2 = M - k - nb;
    double* A11 = A + GEP_IX(k, k, lda);
    double* A21 = A + GEP_IX(k + nb, k, lda);
    double* A22 = A + GEP_IX(k + nb, k + nb, lda);
    const double* L21 = L + GEP_IX(k + nb, k, ldl);
    // C11 = L11^-1 (L11^-1 A11)^T, full symmetric in A11
    double* T1 = X;
    GEP_CHECK(symmetrize_lower(h, nb, A11, lda));
    GEP_CHECK(lln_rec(h, k, nb, nb, L, ldl, invD, A11, lda, tmp, engine));
    GEP_CHECK(transpose(h, nb, nb, A11, lda, T1, nb));
    GEP_CHECK(lln_rec(h, k, nb, nb, L, ldl, invD, T1, nb, tmp, engine));
    GEP_CHECK(copy_lower(h, nb, T1, nb, A11, lda));
    GEP_CHECK(symmetrize_lower(h, nb, A11, lda));
    if (n2 == 0) break;
    // A21 <- A21 L11^-T - 1/2 L21 C11
    GEP_CHECK(rlt_rec(h, k, nb, n2, L, ldl, invD, A21, lda, tmp, engine));
    GEP_CHECK(dgemm(h, 'N', 'N', 'F', n2, nb, nb, -0.5, L21, ldl, A11, lda, 1.0, A21, lda, engine));
    // A22 <- A22 - [A21 L21] [L21 A21]^T (lower triangle)
    double* AA = X;
    double* BB = X + (size_t)n2 * 2 * nb;
    GEP_CHECK(copy_matrix(h, n2, nb, A21, lda, AA, n2));
    GEP_CHECK(copy_matrix(h, n2, nb, L21, ldl, AA + (size_t)n2 * nb, n2));
    GEP_CHECK(copy_matrix(h, n2, nb, L21, ldl, BB, n2));
    GEP_CHECK(copy_matrix(h, n2, nb, A21, lda, BB + (size_t)n2 * nb, n2));
    GEP_CHECK(dgemm(h, 'N', 'T', 'L', n2, n2, 2 * nb, -1.0, AA, n2, BB, n2, 1.0, A22, lda, engine));
    // C21 = L22^-1 (A21 - 1/2 L21 C11)
    GEP_CHECK(dgemm(h, 'N', 'N', 'F', n2, nb, nb, -0.5, L21, ldl, A11, lda, 1.0, A21, lda, engine));
    GEP_CHECK(lln_rec(h, k + nb, n2, nb, L, ldl, invD, A21, lda, tmp, engine));
  }
  return symmetrize_lower(h, M, A, lda);
}

// Eq. 5, "ELPA style": R = L^-1 formed explicitly (R2), then C = (R A) R^T (R3, R4).
// L (lower of B) is overwritten by R.  X and T are M x M scratch matrices (T = tmp2).
int reduce_explicit_inv(gep_handle_t h, int M, double* A, int lda, double* L, int ldl,
                        const double* invD, double* X, double* tmp, int engine) {
  if (M <= 0) return GEP_OK;
  double* T = tmp;                    // M x M
  double* tmp_small = tmp + (size_t)M * M;  // TRI_NB x M
  GEP_CHECK(set_matrix(h, M, M, 0.0, 1.0, X, M));
  GEP_CHECK(trsm_lln(h, M, M, L, ldl, invD, TRI_NB, X, M, tmp_small, engine));  // X = R = L^-1
  GEP_CHECK(symmetrize_lower(h, M, A, lda));
  GEP_CHECK(dgemm(h, 'N', 'N', 'F', M, M, M, 1.0, X, M, A, lda, 0.0, T, M, engine));   // T = R A
  GEP_CHECK(dgemm(h, 'N', 'T', 'L', M, M, M, 1.0, T, M, X, M, 0.0, A, lda, engine));   // C = T R^T
  GEP_CHECK(symmetrize_lower(h, M, A, lda));
  return copy_lower(h, M, X, M, L, ldl);  // lower(B) <- R
}

}  // namespace gep
