// SEP solver, stage "BACK" (Table 3): Z <- Q Z with Q = H_0 H_1 ... H_{M-off-1} left
// in C by the tridiagonalisation (off = 1: reflector j on rows j+1..M-1) or by the
// full-to-band reduction (off = b: reflector j on rows j+b..M-1).  Reflectors are
// grouped in panels of NBB and applied from the last panel to the first in compact-WY
// form,
//     H_j ... H_{j+nb-1} = I - V T V^T    (T upper triangular, forward/columnwise),
//     Z(j+1:, :) -= V (T (V^T Z(j+1:, :))),
// so all O(M^3) work is three matrix products per panel.  Panels are NBB = 1024
// reflectors wide (the update product then has depth 1024); their T factor is built
// recursively, T = [T1, -T1 (V1^T V2) T2; 0, T2], from 64-wide leaves.
#include "gep_internal.cuh"

namespace gep {
namespace {

constexpr int NBB = 1024;
constexpr int LB = 64;  // leaf order of the T-factor recursion

// Explicit V (rows j0+off .. M-1, nb columns): unit entry at local row q, reflector below.
__global__ void k_build_v(int rows, int nb, int j0, int off, const double* __restrict__ C, int ldc,
                          double* __restrict__ V, const int* st) {
  if (status_bad(st)) return;
  int t = blockIdx.x * blockDim.x + threadIdx.x;
  int q = blockIdx.y;
  if (t >= rows || q >= nb) return;
  double val;
  if (t < q) val = 0.0;
  else if (t == q) val = 1.0;
  else val = C[GEP_IX(j0 + off + t, j0 + q, ldc)];
  V[GEP_IX(t, q, rows)] = val;
}

// T factors of every leaf of 64 reflectors of a panel, one CTA each, from G = V^T V:
// T(i,i) = tau_i,  T(0:i, i) = -tau_i T(0:i, 0:i) G(0:i, i).
// Leaves of 16 column by column (a warp each), then T12 = -T1 (G12 T2) on 32 and 64; a product's
// loop takes only the nonzero part of its triangular factor.  Bound: FP64 issue (64 clocks a warp
// instruction).  One warp column by column took 147 us a leaf, and the leaves of a panel
// followed each other; now 33 us for
// all of them (back-transformation of order 500: 2.14 -> 1.07 ms, 2047: 9.2 -> 4.0 ms).
__global__ void __launch_bounds__(256) k_larft(int nbt, const double* __restrict__ G, int ldg,
                                               const double* __restrict__ tau, double* __restrict__ T, int ldt,
                                               const int* st) {
  __shared__ double Gs[LB][LB + 1], Ts[LB][LB + 1];
  double(*Xs)[LB + 1] = reinterpret_cast<double(*)[LB + 1]>(&Gs[32][0]);  // rows 32.. of G are free at the last merge
  if (status_bad(st)) return;
  const int o = blockIdx.x * LB, nb = min(LB, nbt - o), t = threadIdx.x, lane = t & 31, w = t >> 5;
  for (int idx = t; idx < LB * LB; idx += 256) {
    const int r = idx % LB, c = idx / LB;
    Gs[r][c] = r < c && c < nb ? G[GEP_IX(o + r, o + c, ldg)] : 0.0;
    Ts[r][c] = 0.0;
  }
  __syncthreads();
  if (w < 4) {
    const int c0 = 16 * w;
    for (int i = 0; i < 16; ++i) {
      const double ti = c0 + i < nb ? tau[o + c0 + i] : 0.0;
      double s = 0.0;
      for (int u = 0; u < i; ++u)  // (zeros below the diagonal of T)
        if (lane < 16) s = fma(Ts[c0 + lane][c0 + u], Gs[c0 + u][c0 + i], s);
      __syncwarp();
      if (lane < i) Ts[c0 + lane][c0 + i] = -ti * s;
      if (lane == i) Ts[c0 + i][c0 + i] = ti;
      __syncwarp();
    }
  }
  __syncthreads();
  {  // 16 + 16: merge w / 4, lanes 16 rows (columns) x 2, four warps share the other index
    const int b0 = 32 * (w >> 2), l = lane & 15, h = (lane >> 4) + 2 * (w & 3);  // h in 0..7
    double x[2];
#pragma unroll
    for (int u = 0; u < 2; ++u) {  // X(l, j) = sum_{q <= j} G12(l, q) T2(q, j)
      const int j = h + 8 * u;
      x[u] = 0.0;
      for (int q = 0; q < 16; ++q) x[u] = fma(Gs[b0 + l][b0 + 16 + q], Ts[b0 + 16 + q][b0 + 16 + j], x[u]);
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < 2; ++u) Gs[b0 + l][b0 + 16 + h + 8 * u] = x[u];
    __syncthreads();
#pragma unroll
    for (int u = 0; u < 2; ++u) {  // T12(i, l) = -sum_{q >= i} T1(i, q) X(q, l)
      const int i = h + 8 * u;
      double s = 0.0;
      for (int q = 0; q < 16; ++q) s = fma(Ts[b0 + i][b0 + q], Gs[b0 + q][b0 + 16 + l], s);
      Ts[b0 + i][b0 + 16 + l] = -s;
    }
  }
  __syncthreads();
  {  // 32 + 32
    double x[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int j = w + 8 * u;
      x[u] = 0.0;
      for (int q = 0; q <= j; ++q) x[u] = fma(Gs[lane][32 + q], Ts[32 + q][32 + j], x[u]);
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < 4; ++u) Xs[lane][w + 8 * u] = x[u];
    __syncthreads();
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int i = w + 8 * u;
      double s = 0.0;
      for (int q = i; q < 32; ++q) s = fma(Ts[i][q], Xs[q][lane], s);
      Ts[i][32 + lane] = -s;
    }
  }
  __syncthreads();
  for (int idx = t; idx < nb * nb; idx += 256) T[GEP_IX(o + idx % nb, o + idx / nb, ldt)] = Ts[idx % nb][idx / nb];
}

// One level of the T recursion for all its merges (halves of n1 reflectors, blockIdx.z the merge):
// side 0: X = G12 T2 (to the place of T12), side 1: T12 <- -T1 X, through X in `tmp`.
template <int SIDE>
__global__ void __launch_bounds__(256) k_larft_merge(int nbt, int n1, const double* __restrict__ G, int ldg,
                                                     double* __restrict__ T, int ldt, double* __restrict__ tmp,
                                                     const int* st) {
  __shared__ double As[64][17], Bs[64][17];
  if (status_bad(st)) return;
  const int o = blockIdx.z * 2 * n1, n2 = min(n1, nbt - o - n1);
  const int r0 = blockIdx.x * 16, c0 = blockIdx.y * 16;
  if (c0 >= n2) return;
  const double* A = SIDE == 0 ? G + GEP_IX(o, o + n1, ldg) : T + GEP_IX(o, o, ldt);
  const int lda = SIDE == 0 ? ldg : ldt;
  double* X = tmp + (size_t)blockIdx.z * n1 * n1;
  const double* B = SIDE == 0 ? T + GEP_IX(o + n1, o + n1, ldt) : X;
  const int ldb = SIDE == 0 ? ldt : n1;
  const int k0 = SIDE == 0 ? 0 : r0 / 64 * 64, k1 = SIDE == 0 ? min(n2, c0 + 16) : n1;
  const int t = threadIdx.x, i = t & 15, j = t >> 4;
  double acc = 0.0;
  for (int kb = k0; kb < k1; kb += 64) {
    const int kn = min(64, k1 - kb);
    __syncthreads();
    for (int idx = t; idx < 16 * 64; idx += 256) {
      const int r = idx & 15, kk = idx >> 4;
      As[kk][r] = kk < kn ? A[GEP_IX(r0 + r, kb + kk, lda)] : 0.0;
      const int kk2 = idx & 63, c = idx >> 6;
      Bs[kk2][c] = kk2 < kn && c0 + c < n2 ? B[GEP_IX(kb + kk2, c0 + c, ldb)] : 0.0;
    }
    __syncthreads();
#pragma unroll 8
    for (int kk = 0; kk < kn; ++kk) acc = fma(As[kk][i], Bs[kk][j], acc);
  }
  if (c0 + j >= n2) return;
  if (SIDE == 0) X[GEP_IX(r0 + i, c0 + j, n1)] = acc;
  else T[GEP_IX(o + r0 + i, o + n1 + c0 + j, ldt)] = -acc;
}

}  // namespace

// T (nb x nb, upper) of the block reflector whose Gram matrix is G = V^T V: leaves of 64, then
// T12 = -T1 (G12 T2) level by level, narrow levels with all their merges in one FP64 launch per
// product, wide ones (512^3 and up: 250 us on the FP64 units) as FP64-accurate products on the tensor cores unless
// the engine is FP64 (also of the FP32-grade engine: T keeps the accuracy of G).  tmp: nb x nb.
int larft_rec(gep_handle_t h, int nb, const double* G, int ldg, const double* tau, double* T, int ldt,
              double* tmp, int engine) {
  if (nb <= 0) return GEP_OK;
  if (engine == GEP_PREC_MIXED_REFINED) engine = GEP_PREC_FP64_EMULATED;
  if (nb > LB) GEP_CHECK(set_matrix(h, nb, nb, 0.0, 0.0, T, ldt));
  k_larft<<<(nb + LB - 1) / LB, 256, 0, h->stream>>>(nb, G, ldg, tau, T, ldt, h->d_status);
  GEP_CHECK(check_launch(h));
  for (int n1 = LB; n1 < nb; n1 *= 2) {
    const int merges = (nb - n1 + 2 * n1 - 1) / (2 * n1);
    if (n1 < 256 || engine == GEP_PREC_FP64) {
      const dim3 g(n1 / 16, n1 / 16, merges);
      k_larft_merge<0><<<g, 256, 0, h->stream>>>(nb, n1, G, ldg, T, ldt, tmp, h->d_status);
      GEP_CHECK(check_launch(h));
      k_larft_merge<1><<<g, 256, 0, h->stream>>>(nb, n1, G, ldg, T, ldt, tmp, h->d_status);
      GEP_CHECK(check_launch(h));
      continue;
    }
    for (int o = 0; o + n1 < nb; o += 2 * n1) {
      const int n2 = n1 < nb - o - n1 ? n1 : nb - o - n1;
      GEP_CHECK(dgemm(h, 'N', 'N', 'F', n1, n2, n2, 1.0, G + GEP_IX(o, o + n1, ldg), ldg,
                      T + GEP_IX(o + n1, o + n1, ldt), ldt, 0.0, tmp, n1, engine));
      GEP_CHECK(dgemm(h, 'N', 'N', 'F', n1, n2, n1, -1.0, T + GEP_IX(o, o, ldt), ldt, tmp, n1, 0.0,
                      T + GEP_IX(o, o + n1, ldt), ldt, engine));
    }
  }
  return GEP_OK;
}

size_t backtransform_ws_elems(int M, int ncol) {
  auto r = [](size_t n) { return (n + 31) & ~(size_t)31; };
  return r((size_t)M * NBB) + r((size_t)NBB * NBB) * 3 + r((size_t)NBB * (ncol > 0 ? ncol : 1)) * 2;
}

int backtransform_q(gep_handle_t h, int M, int ncol, const double* C, int ldc, const double* tau,
                    double* Z, int ldz, double* ws, size_t ws_elems, int engine, int off) {
  if (M <= off || ncol <= 0) return GEP_OK;
  if (ws_elems < backtransform_ws_elems(M, ncol)) return GEP_ERR_ALLOC;
  auto r = [](size_t n) { return (n + 31) & ~(size_t)31; };
  double* V = ws;
  double* G = V + r((size_t)M * NBB);
  double* T = G + r((size_t)NBB * NBB);
  double* Tt = T + r((size_t)NBB * NBB);  // recursion scratch
  double* W1 = Tt + r((size_t)NBB * NBB);
  double* W2 = W1 + r((size_t)NBB * ncol);
  int nref = M - off;  // reflectors exist for columns 0 .. M-off-1 (reflector j on rows j+off ..)
  int last = ((nref - 1) / NBB) * NBB;
  for (int j0 = last; j0 >= 0; j0 -= NBB) {
    int nb = min(NBB, nref - j0);
    int rows = M - j0 - off;
    dim3 g((rows + 255) / 256, nb);
    k_build_v<<<g, 256, 0, h->stream>>>(rows, nb, j0, off, C, ldc, V, h->d_status);
    GEP_CHECK(check_launch(h));
    GEP_CHECK(dgemm(h, 'T', 'N', 'F', nb, nb, rows, 1.0, V, rows, V, rows, 0.0, G, nb, engine));
    GEP_CHECK(larft_rec(h, nb, G, nb, tau + j0, T, nb, Tt, engine));
    double* Zs = Z + (j0 + off);
    // transposed products keep the long dimension (ncol) as the row dimension of
    // each product, so all three fill full tensor-core tiles:
    //   W1^T = Z^T V,  W2^T = W1^T T^T,  Z -= V W2 = V (W2^T)^T
    GEP_CHECK(dgemm(h, 'T', 'N', 'F', ncol, nb, rows, 1.0, Zs, ldz, V, rows, 0.0, W1, ncol, engine));
    GEP_CHECK(dgemm(h, 'N', 'T', 'F', ncol, nb, nb, 1.0, W1, ncol, T, nb, 0.0, W2, ncol, engine));
    GEP_CHECK(dgemm(h, 'N', 'T', 'F', rows, ncol, nb, -1.0, V, rows, W2, ncol, 1.0, Zs, ldz, engine));
  }
  return GEP_OK;
}

}  // namespace gep
