// FP64 FMA matrix product C = alpha op(A) op(B) + beta C (column-major); op(A) may also
// be a symmetric matrix given by its lower triangle (transa 'S', m = k).
//
// The dense contraction under every blocked stage (trailing updates of the
// Cholesky factorisation, triangular solves, the SYR2K update of the
// tridiagonalisation, the compact-WY back-transformation and the divide-and-
// conquer merge).  64 x 64 output tile per 256-thread CTA, 16-deep k slices
// staged through shared memory, 4 x 4 register micro-tile per thread; the row
// index is the fast thread index so C is read and written coalesced.
// uplo 'L' skips tiles strictly above the diagonal and stores only i >= j
// (SYRK / SYR2K shaped updates of a symmetric lower triangle).
#include <algorithm>

#include "gep_internal.cuh"

namespace gep {
namespace {

constexpr int BM = 64, BN = 64, BK = 16;

template <bool TA, bool TB, bool SA = false>
__global__ void __launch_bounds__(256) k_dgemm(int m, int n, int k, double alpha,
                                               const double* __restrict__ A, int lda,
                                               const double* __restrict__ B, int ldb, double beta,
                                               double* __restrict__ C, int ldc, int lower,
                                               const int* __restrict__ st) {
  const int bi = blockIdx.x, bj = blockIdx.y;
  if (lower && bi < bj) return;
  if (status_bad(st)) return;
  __shared__ double As[BK][BM + 1];
  __shared__ double Bs[BK][BN + 1];
  const int tid = threadIdx.x;
  const int tx = tid & 15, ty = tid >> 4;
  const int row0 = bi * BM, col0 = bj * BN;
  double acc[4][4];
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int c = 0; c < 4; ++c) acc[r][c] = 0.0;

  for (int k0 = 0; k0 < k; k0 += BK) {
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      int idx = tid + r * 256;
      int i, kk;
      if (!TA) { i = idx & 63; kk = idx >> 6; }
      else { kk = idx & 15; i = idx >> 4; }
      int gi = row0 + i, gk = k0 + kk;
      double v = 0.0;
      if (gi < m && gk < k) {
        if (SA) v = gi >= gk ? A[GEP_IX(gi, gk, lda)] : A[GEP_IX(gk, gi, lda)];  // symmetric, lower stored
        else v = TA ? A[GEP_IX(gk, gi, lda)] : A[GEP_IX(gi, gk, lda)];
      }
      As[kk][i] = v;
    }
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      int idx = tid + r * 256;
      int j, kk;
      if (!TB) { kk = idx & 15; j = idx >> 4; }
      else { j = idx & 63; kk = idx >> 6; }
      int gj = col0 + j, gk = k0 + kk;
      double v = 0.0;
      if (gj < n && gk < k) v = TB ? B[GEP_IX(gj, gk, ldb)] : B[GEP_IX(gk, gj, ldb)];
      Bs[kk][j] = v;
    }
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < BK; ++kk) {
      double a[4], b[4];
#pragma unroll
      for (int r = 0; r < 4; ++r) a[r] = As[kk][tx + 16 * r];
#pragma unroll
      for (int c = 0; c < 4; ++c) b[c] = Bs[kk][ty + 16 * c];
#pragma unroll
      for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int c = 0; c < 4; ++c) acc[r][c] = fma(a[r], b[c], acc[r][c]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    int j = col0 + ty + 16 * c;
    if (j >= n) continue;
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      int i = row0 + tx + 16 * r;
      if (i >= m || (lower && i < j)) continue;
      double v = alpha * acc[r][c];
      if (beta != 0.0) v = fma(beta, C[GEP_IX(i, j, ldc)], v);
      C[GEP_IX(i, j, ldc)] = v;
    }
  }
}

// Products whose 64 x 64 tiles are too few to occupy the GPU: a T x T output tile per CTA
// (T = 16 or 32), the depth split over z CTAs per tile where even the 16 x 16 tiles are few.
// The last CTA of a tile to arrive adds the partial tiles in slice order (deterministic, one
// launch; its counter is zero again afterwards).
//
// Bound: an FP64 FMA warp instruction holds its scheduler for 64 clocks (76 with all four busy;
// measured), so a product takes m n k / (SMs in use * 1.68) clocks however its operands are
// staged: one or four outputs per thread straight from shared memory lose nothing against
// register tiles, and the time falls with the number of SMs.  Measured before (64 x 64 tiles,
// split-K with a second launch from k = 1024) and now, launches included: 64 x 64 x 64
// 70 -> 8.5 us, 64 x 64 x 512 530 -> 10.7 us, 64 x 64 x 4096 82 -> 39 us, 128 x 128 x 128
// 137 -> 10.5 us, 500 x 500 x 500 531 -> 228 us (0.55 of the FP64 pipe's rate before, 1 now).
constexpr int SK = 64;  // k slice staged per step

template <int T, bool TA, bool TB, bool SA>
__global__ void __launch_bounds__(256) k_dgemm_small(int m, int n, int k, int kc, double alpha,
                                                     const double* __restrict__ A, int lda,
                                                     const double* __restrict__ B, int ldb, double beta,
                                                     double* __restrict__ C, int ldc, int lower,
                                                     double* __restrict__ part, int* __restrict__ count,
                                                     const int* __restrict__ st) {
  constexpr int R = T * T / 256;  // outputs per thread
  __shared__ double As[SK][T + 1];
  __shared__ double Bs[SK][T + 1];
  __shared__ int last;
  const int bi = blockIdx.x, bj = blockIdx.y, z = blockIdx.z, nz = gridDim.z;
  if (lower && bi < bj) return;
  // with a split depth every CTA counts in, also after an earlier stage's error (which then only
  // suppresses the stores), so that the counters are zero again when the kernel ends
  const bool bad = status_bad(st);
  if (nz == 1 && bad) return;
  const int tid = threadIdx.x, tx = tid % T, ty = tid / T;
  const int row0 = bi * T, col0 = bj * T;
  const int kb = z * kc, ke = min(k, kb + kc);
  double acc[R];
#pragma unroll
  for (int r = 0; r < R; ++r) acc[r] = 0.0;
  // the next k slice is fetched into registers while this one is multiplied (the addresses are
  // clamped into the matrices, so the loads are unconditional and stay in flight together)
  constexpr int U = SK * T / 256;
  double pa[U], pb[U];
  auto fetch = [&](int k0) {
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int idx = tid + u * 256;
      const int i = TA ? idx / SK : idx % T, ka = k0 + (TA ? idx % SK : idx / T);
      const int gi = min(row0 + i, m - 1), ga = min(ka, k - 1);
      const double va = SA ? (gi >= ga ? A[GEP_IX(gi, ga, lda)] : A[GEP_IX(ga, gi, lda)])
                           : (TA ? A[GEP_IX(ga, gi, lda)] : A[GEP_IX(gi, ga, lda)]);
      pa[u] = ka < ke && row0 + i < m ? va : 0.0;
      const int j = TB ? idx % T : idx / SK, kq = k0 + (TB ? idx / T : idx % SK);
      const int gj = min(col0 + j, n - 1), gb = min(kq, k - 1);
      const double vb = TB ? B[GEP_IX(gj, gb, ldb)] : B[GEP_IX(gb, gj, ldb)];
      pb[u] = kq < ke && col0 + j < n ? vb : 0.0;
    }
  };
  if (kb < ke) fetch(kb);
  for (int k0 = kb; k0 < ke; k0 += SK) {
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int idx = tid + u * 256;
      As[TA ? idx % SK : idx / T][TA ? idx / SK : idx % T] = pa[u];
      Bs[TB ? idx / T : idx % SK][TB ? idx % T : idx / SK] = pb[u];
    }
    __syncthreads();
    if (k0 + SK < ke) fetch(k0 + SK);
    const int kn = min(SK, ke - k0);
#pragma unroll 8
    for (int kk = 0; kk < kn; ++kk) {
      const double a = As[kk][tx];
#pragma unroll
      for (int r = 0; r < R; ++r) acc[r] = fma(a, Bs[kk][ty + r * (256 / T)], acc[r]);
    }
    __syncthreads();
  }
  if (nz > 1) {
    const size_t tile = (size_t)bj * gridDim.x + bi;
    double* P = part + tile * nz * (T * T);
#pragma unroll
    for (int r = 0; r < R; ++r) __stcg(P + (size_t)z * (T * T) + tid + r * 256, acc[r]);
    __threadfence();
    __syncthreads();
    if (tid == 0) {
      last = atomicAdd(count + tile, 1) == nz - 1;
      if (last) count[tile] = 0;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
#pragma unroll
    for (int r = 0; r < R; ++r) {
      double s0 = 0.0, s1 = 0.0;
      int q = 0;
      for (; q + 8 <= nz; q += 8) {
        double x[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) x[u] = __ldcg(P + (size_t)(q + u) * (T * T) + tid + r * 256);
#pragma unroll
        for (int u = 0; u < 8; u += 2) {
          s0 += x[u];
          s1 += x[u + 1];
        }
      }
      for (; q < nz; ++q) s0 += __ldcg(P + (size_t)q * (T * T) + tid + r * 256);
      acc[r] = s0 + s1;
    }
  }
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int i = row0 + tx, j = col0 + ty + r * (256 / T);
    if (bad || i >= m || j >= n || (lower && i < j)) continue;
    double v = alpha * acc[r];
    if (beta != 0.0) v = fma(beta, C[GEP_IX(i, j, ldc)], v);
    C[GEP_IX(i, j, ldc)] = v;
  }
}

template <int T>
int launch_small(gep_handle_t h, bool TA, bool TB, bool SA, int z, int m, int n, int k, double alpha, const double* A,
                 int lda, const double* B, int ldb, double beta, double* C, int ldc, int lower) {
  const dim3 g((m + T - 1) / T, (n + T - 1) / T, z);
  const int kc = (k + z - 1) / z;
  const int* st = h->d_status;
  double* P = h->d_splitk;
  int* cnt = h->d_splitk_count;
#define GEP_SMALL(ta, tb, sa) \
  k_dgemm_small<T, ta, tb, sa><<<g, 256, 0, h->stream>>>(m, n, k, kc, alpha, A, lda, B, ldb, beta, C, ldc, lower, P, cnt, st)
  if (SA) GEP_SMALL(false, false, true);
  else if (!TA && !TB) GEP_SMALL(false, false, false);
  else if (!TA && TB) GEP_SMALL(false, true, false);
  else if (TA && !TB) GEP_SMALL(true, false, false);
  else GEP_SMALL(true, true, false);
#undef GEP_SMALL
  return check_launch(h);
}

__global__ void k_scale(int m, int n, double beta, double* C, int ldc, int lower,
                        const int* __restrict__ st) {
  if (status_bad(st)) return;
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  int j = blockIdx.y;
  if (i >= m || j >= n || (lower && i < j)) return;
  C[GEP_IX(i, j, ldc)] = beta == 0.0 ? 0.0 : beta * C[GEP_IX(i, j, ldc)];
}

}  // namespace

int dgemm_f64(gep_handle_t h, char ta, char tb, char uplo, int m, int n, int k, double alpha,
              const double* A, int lda, const double* B, int ldb, double beta, double* C, int ldc) {
  if (m <= 0 || n <= 0) return GEP_OK;
  int lower = (uplo == 'L' || uplo == 'l');
  if (k <= 0 || alpha == 0.0) {
    if (beta == 1.0) return GEP_OK;
    dim3 g((m + 255) / 256, n);
    k_scale<<<g, 256, 0, h->stream>>>(m, n, beta, C, ldc, lower, h->d_status);
    return check_launch(h);
  }
  bool TA = (ta == 'T' || ta == 't'), TB = (tb == 'T' || tb == 't');
  const bool SA = (ta == 'S' || ta == 's');  // A symmetric (m x m, k = m), lower triangle stored
  if (SA && (TB || k != m)) return GEP_ERR_UNSUPPORTED;
  dim3 grid((m + BM - 1) / BM, (n + BN - 1) / BN);
  // Tile choice: the largest tile that still gives every SM about four CTAs, else 16 x 16 tiles
  // with the depth split over CTAs until there are two CTAs per SM (slices of at least 32)
  auto tiles_of = [&](int t) {
    long long gx = (m + t - 1) / t, gy = (n + t - 1) / t;
    return lower ? gx * gy - (gy < gx ? gy : gx) * ((gy < gx ? gy : gx) - 1) / 2 : gx * gy;
  };
  const long long full = 4LL * h->sm_count;
  if (tiles_of(BM) < full && (n + 15) / 16 <= 65535) {
    if (tiles_of(32) >= full)
      return launch_small<32>(h, TA, TB, SA, 1, m, n, k, alpha, A, lda, B, ldb, beta, C, ldc, lower);
    const long long grid16 = (long long)((m + 15) / 16) * ((n + 15) / 16);
    int z = 1;
    if (h->d_splitk && grid16 <= SPLITK_TILES) {
      // the depth split with the least work on the busiest SM, plus the cost of the final sums
      const long long t16 = tiles_of(16), zmax = std::min<long long>({64, k / 32, SPLITK_DOUBLES / (grid16 * 256)});
      double best = 1e30;
      for (int q = 1; q <= zmax && t16 * (q - 1) < 8LL * h->sm_count; ++q) {
        const double busiest = (double)((t16 * q + h->sm_count - 1) / h->sm_count) / q;
        const double cost = busiest * (1.0 + (q > 1 ? 0.64 * q / (k / q + 32.0) : 0.0));
        if (cost < best * 0.97) {
          best = cost;
          z = q;
        }
      }
    }
    return launch_small<16>(h, TA, TB, SA, z, m, n, k, alpha, A, lda, B, ldb, beta, C, ldc, lower);
  }
  if (SA)
    k_dgemm<false, false, true><<<grid, 256, 0, h->stream>>>(m, n, k, alpha, A, lda, B, ldb, beta, C, ldc, lower,
                                                              h->d_status);
  else if (!TA && !TB)
    k_dgemm<false, false><<<grid, 256, 0, h->stream>>>(m, n, k, alpha, A, lda, B, ldb, beta, C, ldc, lower, h->d_status);
  else if (!TA && TB)
    k_dgemm<false, true><<<grid, 256, 0, h->stream>>>(m, n, k, alpha, A, lda, B, ldb, beta, C, ldc, lower, h->d_status);
  else if (TA && !TB)
    k_dgemm<true, false><<<grid, 256, 0, h->stream>>>(m, n, k, alpha, A, lda, B, ldb, beta, C, ldc, lower, h->d_status);
  else
    k_dgemm<true, true><<<grid, 256, 0, h->stream>>>(m, n, k, alpha, A, lda, B, ldb, beta, C, ldc, lower, h->d_status);
  return check_launch(h);
}

// The faster engine for a product on the tensor-core precisions, by the measured costs of both
// (us, launches included; checked against 14 shapes from 128^3 to 4096^3, within a fifth):
//   FP64 units:    8 + mnk / 0.525e6
//   split-BF16:    20 for the digit splits and launches, per wave of 128 x 64 tiles 4 (epilogue)
//                  + 0.047 k (36 plane products; 0.01 k with 3 planes), and the operands' digits
//                  (24 bytes an element at 5 TB/s).
// So 128^3 (10.5 / 28 us) and 128 x 128 x 2048 stay on the FP64 units, 256^3 (35 / 35 us) and
// 127 x 1024 x 1024 (234 / 60 us) go to the tensor cores (deep ones in the form of gemm_res.cu).
bool product_on_tensor_cores(gep_handle_t h, char uplo, int m, int n, int k, int engine) {
  if (engine == GEP_PREC_FP64 || m < 32 || n < 16 || k < 16) return false;
  const double half = (uplo == 'L' || uplo == 'l') ? 0.5 : 1.0;
  const double tiles = half * ((m + 127) / 128) * ((n + 63) / 64);
  const double waves = tiles <= h->sm_count ? 1.0 : tiles / h->sm_count;
  const double oz = 20.0 + waves * (4.0 + (engine == GEP_PREC_FP64_EMULATED ? 0.047 : 0.01) * k) +
                    5e-6 * ((double)m + n) * k;
  const double f64 = 8.0 + half * (double)m * n * k * (1e-6 / 0.525);
  return oz < f64;
}

int dgemm(gep_handle_t h, char ta, char tb, char uplo, int m, int n, int k, double alpha,
          const double* A, int lda, const double* B, int ldb, double beta, double* C, int ldc,
          int engine, const OzKRange* kr) {
  const bool big = product_on_tensor_cores(h, uplo, m, n, k, engine);
  if (engine == GEP_PREC_FP64_EMULATED && big)
    return dgemm_oz(h, ta, tb, uplo, m, n, k, alpha, A, lda, B, ldb, beta, C, ldc, 9, kr);
  if (engine == GEP_PREC_MIXED_REFINED && big)
    return dgemm_oz(h, ta, tb, uplo, m, n, k, alpha, A, lda, B, ldb, beta, C, ldc, 4, kr);
  return dgemm_f64(h, ta, tb, uplo, m, n, k, alpha, A, lda, B, ldb, beta, C, ldc);
}

}  // namespace gep
