// SEP solver, two-stage path: the narrow-band reduction SEP solvers of section 3
// (ELPA2 / Eigen_sx), stages "TRD/BAND" and "BACK" of Table 3.
//
// S1b full -> band.  C = Q1 C_b Q1^T with C_b of bandwidth b.  For each panel of b
// columns the n x b block below the band is QR-factorised with Householder
// reflectors (Q_p = I - V T V^T), R stays in the band and the trailing matrix takes
// the two-sided update
//     X = C22 V T,  W = X - V (T^T V^T X) / 2,  C22 <- C22 - W V^T - V W^T,
// i.e. all O(M^3) work is matrix products (split-BF16 tensor-core engine).  Only the
// lower triangle of C22 is stored and updated; C22 V reads it as a symmetric operand.
//
// S1c band -> tridiagonal (bulge chasing).  Sweep s annihilates column s below the
// subdiagonal with a reflector H(s,0) on rows s+1..s+b, then chases the bulge that
// the right-application creates one b x b block further down per step:
//     step k: B = C(st_k:, st_{k-1}:) <- B H(s,k-1);  H(s,k) annihilates B(1:, 0);
//             B <- H(s,k) B;  D = C(st_k:, st_k:) <- H(s,k) D H(s,k),
// st_k = s + 1 + k b.  Step k of sweep s+1 only needs step k+1 of sweep s to be done,
// so sweeps run concurrently on different CTAs, each one step-pipelined behind the
// previous sweep (progress counters with acquire/release, bounded waits).
//
// Back-transformation.  Z = Q1 (Q2 Z_T), Q2 = prod_s prod_k H(s,k).  The reflectors
// H(s,k) of the b sweeps s0..s0+b-1 of group j (s0 = j b) at the same step k occupy a
// (2b-1)-row "diamond" G(j,k) = H(s0,k) ... H(s0+b-1,k), and
//     Q2 = prod_{j ascending} prod_{k descending} G(j,k),
// because H(s,k) commutes with every H(s',k') (s' < s, k' < k) it has to pass.  The
// diamonds are applied in wavefronts t = (J - j) + k: diamonds of one wavefront touch
// disjoint rows and every diamond that must precede one of them lies in an earlier
// wavefront.  Q1 is applied with the compact-WY back-transformation of the 1-stage
// path, its reflectors starting b rows (instead of one) below their column.
#include <math.h>

#include <algorithm>
#include <vector>

#include "fixed.cuh"
#include "gep_internal.cuh"

namespace gep {
namespace {

constexpr int BMAX = 64;      // largest bandwidth
constexpr int BULGE_CTAS_PER_SM = 1;  // resident bulge-chasing CTAs per SM
constexpr int BAND_GROUP = 4;  // panels per group of the full -> band reduction (trailing update depth 2 G b)
constexpr int BAND_GROUP_MIN_N = 8192;  // trailing order from which groups of BAND_GROUP are used (b = 64; half of
                                        // it at b <= 32: order 8192 S1b 130 -> 123 ms, order 4000 no gain)
constexpr int PQ_ROWS = 256;  // panel rows per CTA in the panel QR (one per thread)
constexpr int PQ_CH = 16;     // columns per reduction chunk in the panel QR

size_t rr(size_t n) { return (n + 31) & ~(size_t)31; }

// ------------------------------------------------------------------ S1b panel QR

// One Householder step (column c) of the QR factorisation of the n x nb panel P (ld ldp),
// fused with the partial dot products the next step needs.  part_in[j][g] (g over the
// CTAs) = sum over rows r > c of P(r,c) P(r,j), prow_in[j] = P(c,j): the pivot row is
// kept out of the sums so that the norm of the tail is never formed by cancellation.
// c = -1 only produces part/prow for column 0.  The reflector follows LAPACK's dlarfg:
// beta = -sign(alpha) ||x||, tau = (beta - alpha) / beta, v = [1; x(1:) / (alpha - beta)].
__global__ void __launch_bounds__(PQ_ROWS) k_pqr_step(int n, int nb, int c, double* __restrict__ P, int ldp,
                                                      const double* __restrict__ part_in,
                                                      const double* __restrict__ prow_in,
                                                      double* __restrict__ part_out, double* __restrict__ prow_out,
                                                      double* __restrict__ tau, const int* st) {
  __shared__ double sd[BMAX], sw[BMAX], sc[3];
  __shared__ double prod[PQ_ROWS][PQ_CH + 1];
  __shared__ double seg[PQ_ROWS / PQ_CH][PQ_CH];
  if (status_bad(st)) return;
  const int t = threadIdx.x, G = gridDim.x;
  const int r = blockIdx.x * PQ_ROWS + t;
  double tk = 0.0, scale = 0.0, beta = 0.0;
  if (c >= 0) {
    {  // column j's partials part_in[j * G + g]: one warp per column, fixed-order tree
      const int w = t >> 5, lane = t & 31;
      for (int j = c + w; j < nb; j += PQ_ROWS / 32) {
        double s = 0.0;
        for (int g = lane; g < G; g += 32) s += part_in[(size_t)j * G + g];
        for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (lane == 0) sd[j] = s;
      }
    }
    __syncthreads();
    if (t == 0) {
      double alpha = prow_in[c], xn2 = sd[c];
      double tt = 0.0, sl = 0.0, be = alpha;
      if (xn2 > 0.0 && !tiny_squares(alpha * alpha + xn2)) {
        be = -copysign(sqrt(alpha * alpha + xn2), alpha);
        tt = (be - alpha) / be;
        sl = 1.0 / (alpha - be);
      }
      sc[0] = tt;
      sc[1] = sl;
      sc[2] = be;
      if (blockIdx.x == 0) tau[c] = tt;
    }
    __syncthreads();
    tk = sc[0];
    scale = sc[1];
    beta = sc[2];
    if (t < nb && t > c) sw[t] = prow_in[t] + scale * sd[t];  // v^T P(:, t)
    __syncthreads();
  }
  const int nc = c + 1;  // pivot column of the next step
  // this row: reflector entry and the new value of P(r, nc)
  double vr = 0.0, pn = 0.0;
  bool live = r < n && r >= (c < 0 ? 0 : c);
  if (live && c >= 0) {
    if (r == c) {
      P[r + (size_t)c * ldp] = beta;
    } else {
      vr = P[r + (size_t)c * ldp] * scale;
      P[r + (size_t)c * ldp] = vr;
    }
  }
  if (live && nc < nb) {
    double x = (c >= 0 && r == c) ? prow_in[nc] : P[r + (size_t)nc * ldp];
    if (c >= 0) x -= tk * (r == c ? 1.0 : vr) * sw[nc];
    pn = x;
  }
  for (int cb = (nc < 0 ? 0 : nc); cb < nb; cb += PQ_CH) {
    for (int q = 0; q < PQ_CH; ++q) {
      int j = cb + q;
      double pr = 0.0;
      if (live && j < nb) {
        double x = (c >= 0 && r == c) ? prow_in[j] : P[r + (size_t)j * ldp];
        if (c >= 0) {
          x -= tk * (r == c ? 1.0 : vr) * sw[j];
          P[r + (size_t)j * ldp] = x;
        }
        if (r == nc) prow_out[j] = x;
        if (r > nc) pr = pn * x;
      }
      prod[t][q] = pr;
    }
    __syncthreads();
    {
      int q = t % PQ_CH, sg = t / PQ_CH;
      double s = 0.0;
      for (int i = 0; i < PQ_CH; ++i) s += prod[sg * PQ_CH + i][q];
      seg[sg][q] = s;
    }
    __syncthreads();
    if (t < PQ_CH && cb + t < nb) {
      double s = 0.0;
      for (int sg = 0; sg < PQ_ROWS / PQ_CH; ++sg) s += seg[sg][t];
      part_out[(size_t)(cb + t) * G + blockIdx.x] = s;
    }
    __syncthreads();
  }
}

__device__ __forceinline__ unsigned long long gclock() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
__device__ __forceinline__ int ld_acquire(const int* p) {
  int v;
  asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_release(int* p, int v) {
  asm volatile("st.release.gpu.global.s32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// Absolute row sums (zero on entry) of the symmetric matrix in the lower triangle of C, as integers: in units of
// 2^-40 of the power of two of the largest entry (*ex its exponent field), an entry that is not zero at least
// one.  A 64 x 64 tile a CTA; integer sums, so that the rule below gives the same answer every time.  One pass over the
// triangle: order 8192 about 60 us.
__global__ void __launch_bounds__(256) k_row_sums(int M, const double* __restrict__ C, int ldc, const int* __restrict__ ex,
                                                  unsigned long long* __restrict__ sum, const int* st) {
  __shared__ unsigned long long row[64], col[64];
  if (blockIdx.x < blockIdx.y || status_bad(st)) return;
  const int t = threadIdx.x, r0 = blockIdx.x * 64, c0 = blockIdx.y * 64, r = r0 + (t & 63), sh = 1023 - *ex + 40;
  if (t < 64) row[t] = col[t] = 0;
  __syncthreads();
  ll m = 0;
#pragma unroll
  for (int u = 0; u < 16; ++u) {
    const int q = (t >> 6) + 4 * u, c = c0 + q;
    const ll x = r < M && c <= r ? __double_as_longlong(C[r + (size_t)c * ldc]) & ~(1ll << 63) : 0;
    const ll v = max(qfix(x, sh), (ll)(x != 0));
    m += v;
    const ll w = qwarp_sum(r != c ? v : 0);
    if ((t & 31) == 0) atomicAdd(&col[q], (unsigned long long)w);
  }
  atomicAdd(&row[t & 63], (unsigned long long)m);
  __syncthreads();
  if (t < 64 && r0 + t < M) atomicAdd(sum + r0 + t, row[t]);
  else if (t >= 64 && t < 128 && c0 + t - 64 < M) atomicAdd(sum + c0 + t - 64, col[t - 64]);
}

// *wide: whether the sums of the rows that are not zero lie further apart than 2^4.
__global__ void __launch_bounds__(1024) k_row_spread(int M, const unsigned long long* __restrict__ sum,
                                                     const int* __restrict__ ex, int* __restrict__ wide, const int* st) {
  __shared__ unsigned long long hi, lo;
  if (status_bad(st)) return;
  if (threadIdx.x == 0) {
    hi = 0;
    lo = ~0ull;
  }
  __syncthreads();
  for (int i = threadIdx.x; i < M; i += 1024)
    if (sum[i]) {
      atomicMax(&hi, sum[i]);
      atomicMin(&lo, sum[i]);
    }
  __syncthreads();
  if (threadIdx.x == 0) *wide = *ex < 0x7FF && hi != 0 && lo < hi >> 4;
}

// The whole panel QR in one cooperative launch: CTA g keeps panel rows [rp g, rp g + rp)
// (rp = 64, 128 or 256: the per-SM FP64 rate bounds a step, so short panels take more
// CTAs of fewer rows) in shared memory for all column steps.  Each step is k_pqr_step's
// Householder step; the partial dot products of the next step are accumulated per column
// with FMAs down the CTA's rows (four row quarters, then three adds).  The partial sums and
// the next pivot row go through part/prow (ping-pong) across a grid barrier.  bar[0]
// counts barrier arrivals (zero on entry); a barrier that does not complete within 4 s
// records GEP_ERR_TIMEOUT and the CTA returns.
__global__ void __launch_bounds__(PQ_ROWS) k_pqr_coop(int n, int nb, int rp, double* __restrict__ P, int ldp,
                                                      double* __restrict__ part0, double* __restrict__ part1,
                                                      double* __restrict__ prow0, double* __restrict__ prow1,
                                                      double* __restrict__ tau, int* bar, int* st) {
  extern __shared__ double Ps[];  // [rp][nb + 1]
  __shared__ double sd[BMAX], sw[BMAX], sc[3];
  __shared__ double pnv[PQ_ROWS];      // P(r, nc) of the rows below the next pivot, else 0
  __shared__ double red4[4][BMAX];     // per-column partial dots of the four row quarters
  __shared__ int gok;
  if (status_bad(st)) return;
  const int t = threadIdx.x, G = gridDim.x, blk = blockIdx.x;
  const bool mine = t < rp;
  const int r = blk * rp + t;
  const int ld = nb + 1;
  if (mine)
    for (int j = 0; j < nb; ++j) Ps[t * ld + j] = (r < n) ? P[r + (size_t)j * ldp] : 0.0;
  const int nref = n < nb ? n : nb;
  double *pin = part0, *pout = part1, *rin = prow0, *rout = prow1;
  int epoch = 0;
  __syncthreads();
  for (int c = -1; c < nref; ++c) {
    double tk = 0.0, scale = 0.0, beta = 0.0;
    if (c >= 0) {
      {  // column j's partials pin[j * G + g], one warp per column, fixed-order tree
        const int w = t >> 5, lane = t & 31;
        for (int j = c + w; j < nb; j += PQ_ROWS / 32) {
          double s = 0.0;
          for (int g = lane; g < G; g += 32) s += __ldcg(pin + (size_t)j * G + g);
          for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
          if (lane == 0) sd[j] = s;
        }
      }
      __syncthreads();
      if (t == 0) {
        double alpha = __ldcg(rin + c), xn2 = sd[c];
        double tt = 0.0, sl = 0.0, be = alpha;
        if (xn2 > 0.0 && !tiny_squares(alpha * alpha + xn2)) {
          be = -copysign(sqrt(alpha * alpha + xn2), alpha);
          tt = (be - alpha) / be;
          sl = 1.0 / (alpha - be);
        }
        sc[0] = tt;
        sc[1] = sl;
        sc[2] = be;
        if (blk == 0) tau[c] = tt;
      }
      __syncthreads();
      tk = sc[0];
      scale = sc[1];
      beta = sc[2];
      if (t < nb && t > c) sw[t] = __ldcg(rin + t) + scale * sd[t];  // v^T P(:, t)
      __syncthreads();
    }
    const int nc = c + 1;
    const bool live = mine && r < n && r >= (c < 0 ? 0 : c);
    double* row = Ps + t * ld;
    if (live && c >= 0) {
      const double vr = (r == c) ? 1.0 : row[c] * scale;
      row[c] = (r == c) ? beta : vr;
      for (int j = c + 1; j < nb; ++j) row[j] -= tk * vr * sw[j];
    }
    if (nc < nb) {
      // partial dots of column nc with columns j >= nc over this CTA's rows below the pivot:
      // thread (j = t mod 64, quarter t / 64) accumulates with FMAs down its rows, then the
      // four quarters are added (the FP64 pipe, not the loads, bounds this phase)
      if (mine) {
        pnv[t] = (live && r > nc) ? row[nc] : 0.0;
        if (live && r == nc)
          for (int j = nc; j < nb; ++j) rout[j] = row[j];
      }
      __syncthreads();
      {
        const int j = t & (BMAX - 1), qtr = t >> 6;
        double sum = 0.0;
        if (j >= nc && j < nb)
          for (int i = qtr; i < rp; i += 4) sum = fma(pnv[i], Ps[i * ld + j], sum);
        red4[qtr][j] = sum;
      }
      __syncthreads();
      if (t >= nc && t < nb) pout[(size_t)t * G + blk] = (red4[0][t] + red4[1][t]) + (red4[2][t] + red4[3][t]);
    }
    if (c + 1 >= nref) break;  // the last step needs no exchange
    // grid barrier: this CTA's pout / rout are complete and visible before any CTA reads them
    __syncthreads();
    if (t == 0) {
      __threadfence();
      const int target = (epoch + 1) * G;
      int ok = 1;
      if (atomicAdd(bar, 1) + 1 < target) {
        unsigned long long t0 = gclock();
        for (;;) {
          if (ld_acquire(bar) >= target) break;
          if (*(volatile int*)(st + 1) != 0) { ok = 0; break; }
          if (gclock() - t0 > 4000000000ull) {
            atomicExch(st + 1, GEP_ERR_TIMEOUT);
            ok = 0;
            break;
          }
        }
      }
      gok = ok;
    }
    __syncthreads();
    if (!gok) return;
    ++epoch;
    double* tp = pin; pin = pout; pout = tp;
    tp = rin; rin = rout; rout = tp;
  }
  __syncthreads();
  if (mine && r < n)
    for (int j = 0; j < nb; ++j) P[r + (size_t)j * ldp] = Ps[t * ld + j];
}

size_t pqr_coop_smem_bytes(int rp, int nb) { return (size_t)rp * (nb + 1) * sizeof(double); }

// ---- panel QR of at most 32 columns, registers only, with its T factor (panels of more than 2048 rows;
// panel_cluster.cu takes the shorter ones)
//
// One cooperative launch: warp w of a CTA holds RPW consecutive rows of the panel, lane j column j,
// so that a column's update and the next column's dot products are one FMA each per row of a
// warp (an FP64 instruction holds a scheduler 64 clocks whatever its lanes do) and the entries
// of the pivot column reach the lanes by shuffle.  Per column one grid barrier carries the
// partial dots of the next pivot column with all columns: those to its right give w = v^T P, those
// to its left the Gram entries v_q^T v of the T factor, which a ninth warp of CTA 0 accumulates
// beside the others.  The results go where the two-sided update reads them: P (R and the
// reflectors), both group buffers of V at full height (zero rows above), T.
//
// Bound: the barrier (1.2 us), the partial sums (G / 8 adds a thread) and the scalars' chain.
// Rows per CTA balance row work against partial sums: 304 RPW + 2.4 n / RPW clocks, least at
// RPW = sqrt(n / 127).  Measured per panel of 32 columns with everything up to W (before: QR, V, Gram
// product, T, four copies and four products in 14 launches): order 2047 460 -> 305 us, S1b 29.8 ->
// 19.6 ms; order 8192 224 -> 184 ms.
constexpr int PQN = 32;        // columns, one per lane
constexpr int PQW = 8;         // row warps
struct PanelArgs {
  int n, nb, ldp, r0, ldv;  // r0: zero rows above the panel in Va, Vb
  double *P, *tau, *part, *prow, *Va, *Vb, *T;
  int *bar, *st;
};

template <int RPW>
__global__ void __launch_bounds__(32 * (PQW + 1)) k_panel_qr(PanelArgs a) {
  constexpr int ROWS = PQW * RPW;
  __shared__ double tile[PQN][ROWS + 1];
  __shared__ double red[PQW][PQN], hv[PQN], cv[PQN], gb[2][PQN], ts[2];
  __shared__ double Ts[PQN][PQN + 1];
  __shared__ int ok_s;
  if (status_bad(a.st)) return;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, blk = blockIdx.x, G = gridDim.x;
  const int n = a.n, nb = a.nb, rb = blk * ROWS;
  const int nref = n < nb ? n : nb;
  const bool worker = warp < PQW;
  auto work_sync = [&]() { asm volatile("bar.sync 1, %0;" ::"n"(32 * PQW) : "memory"); };
  for (int idx = tid; idx < ROWS * PQN; idx += blockDim.x) {
    const int r = idx % ROWS, j = idx / ROWS;
    tile[j][r] = rb + r < n && j < nb ? a.P[rb + r + (size_t)j * a.ldp] : 0.0;
  }
  for (int idx = tid; idx < PQN * (PQN + 1); idx += blockDim.x) (&Ts[0][0])[idx] = 0.0;
  for (int idx = blk * blockDim.x + tid; idx < a.r0 * nb; idx += G * blockDim.x) {
    const size_t o = (size_t)(idx / a.r0) * a.ldv + idx % a.r0;
    a.Va[o] = 0.0;
    a.Vb[o] = 0.0;
  }
  __syncthreads();
  double x[RPW];
  const int row0 = rb + warp * RPW;
#pragma unroll
  for (int u = 0; u < RPW; ++u) x[u] = worker ? tile[lane][warp * RPW + u] : 0.0;
  for (int c = -1; c < nref; ++c) {
    double *pin = a.part + (size_t)(c & 1) * G * PQN, *pout = a.part + (size_t)((c + 1) & 1) * G * PQN;
    double *rin = a.prow + (c & 1) * PQN, *rout = a.prow + ((c + 1) & 1) * PQN;
    if (c >= 0) {
      if (worker) {
        double s0 = 0.0, s1 = 0.0;
        int g = warp;
        for (; g + 3 * PQW < G; g += 4 * PQW) {
          const double p0 = __ldcg(pin + (size_t)g * PQN + lane), p1 = __ldcg(pin + (size_t)(g + PQW) * PQN + lane);
          const double p2 = __ldcg(pin + (size_t)(g + 2 * PQW) * PQN + lane), p3 = __ldcg(pin + (size_t)(g + 3 * PQW) * PQN + lane);
          s0 += p0; s1 += p1; s0 += p2; s1 += p3;
        }
        for (; g < G; g += PQW) s0 += __ldcg(pin + (size_t)g * PQN + lane);
        red[warp][lane] = s0 + s1;
        const double pr = warp == 0 ? __ldcg(rin + lane) : 0.0;
        work_sync();
        if (warp == 0) {
          double s = ((red[0][lane] + red[1][lane]) + (red[2][lane] + red[3][lane])) +
                     ((red[4][lane] + red[5][lane]) + (red[6][lane] + red[7][lane]));
          const double xn2 = __shfl_sync(0xffffffffu, s, c), alpha = __shfl_sync(0xffffffffu, pr, c);
          double tt = 0.0, sl = 0.0, be = alpha;
          const double n2 = fma(alpha, alpha, xn2);
          if (xn2 > 0.0 && !tiny_squares(n2)) {
            const double ri = rsqrt(n2);
            be = -copysign(n2 * ri, alpha);
            sl = 1.0 / (alpha - be);
            tt = fma(fabs(alpha), ri, 1.0);
          }
          const double wj = fma(sl, s, pr);  // v^T P(:, j); for j < c the Gram entry v_j^T v
          gb[c & 1][lane] = wj;
          cv[lane] = lane > c ? -(tt * wj) : 0.0;               // pivot row: P(c, j) -= tau w_j
          hv[lane] = lane > c ? -(sl * (tt * wj)) : (lane == c ? sl : 0.0);  // rows below: += P(r, c) h_j
          if (lane == 0) {
            ts[0] = tt;
            ts[1] = be;
            if (blk == 0) a.tau[c] = tt;
          }
        }
      }
      __syncthreads();
      if (worker) {
        const double h = hv[lane];
#pragma unroll
        for (int u = 0; u < RPW; ++u) {
          const int r = row0 + u;
          if (r > c) {
            const double xc = __shfl_sync(0xffffffffu, x[u], c);
            x[u] = fma(xc, h, lane == c ? 0.0 : x[u]);
          } else if (r == c) {
            x[u] = lane == c ? ts[1] : x[u] + cv[lane];
          }
        }
      } else if (blk == 0) {  // column c of T: T(0:c, c) = -tau T(0:c, 0:c) G(0:c, c)
        const double tt = ts[0];
        double s = 0.0;
        for (int q = 0; q < c; ++q) s = fma(Ts[lane][q], gb[c & 1][q], s);
        Ts[lane][c] = lane < c ? -tt * s : (lane == c ? tt : 0.0);
        __syncwarp();
      }
    }
    const int nc = c + 1;
    if (nc >= nref) break;
    if (worker) {
      double s = 0.0;
#pragma unroll
      for (int u = 0; u < RPW; ++u) {
        const int r = row0 + u;
        if (r > nc) s = fma(__shfl_sync(0xffffffffu, x[u], nc), x[u], s);
        else if (r == nc) __stcg(rout + lane, x[u]);
      }
      red[warp][lane] = s;
      work_sync();
      if (warp == 0) {
        s = ((red[0][lane] + red[1][lane]) + (red[2][lane] + red[3][lane])) +
            ((red[4][lane] + red[5][lane]) + (red[6][lane] + red[7][lane]));
        __stcg(pout + (size_t)blk * PQN + lane, s);
        __syncwarp();
        if (lane == 0) {
          int ok = 1;
          if (G > 1) {
            asm volatile("red.release.gpu.global.add.s32 [%0], 1;" ::"l"(a.bar) : "memory");
            const int target = (nc + 1) * G;
            unsigned long long t0 = 0;
            for (int it = 0; ld_acquire(a.bar) < target; ++it) {
              if ((it & 31) != 31) continue;
              if (*(volatile int*)(a.st + 1) != 0) { ok = 0; break; }
              const unsigned long long now = gclock();
              if (t0 == 0) t0 = now;
              if (now - t0 > 4000000000ull) {
                atomicExch(a.st + 1, GEP_ERR_TIMEOUT);
                ok = 0;
                break;
              }
            }
          }
          ok_s = ok;
        }
      }
    }
    __syncthreads();
    if (!ok_s) return;
  }
  __syncthreads();
  if (worker)
#pragma unroll
    for (int u = 0; u < RPW; ++u) tile[lane][warp * RPW + u] = x[u];
  __syncthreads();
  for (int idx = tid; idx < ROWS * nb; idx += blockDim.x) {
    const int lr = idx % ROWS, j = idx / ROWS, r = rb + lr;
    if (r >= n) continue;
    const double p = tile[j][lr], v = r > j ? p : (r == j ? 1.0 : 0.0);
    a.P[r + (size_t)j * a.ldp] = p;
    const size_t o = (size_t)j * a.ldv + a.r0 + r;
    a.Va[o] = v;
    a.Vb[o] = v;
  }
  if (blk == 0)
    for (int idx = tid; idx < nb * nb; idx += blockDim.x) a.T[idx] = Ts[idx % nb][idx / nb];
}

// W = (Y - V M) T with Y = C22 V (n x nb), M = T^T S / 2, S = V^T Y: the companion of V in the
// two-sided update, written to both group buffers at full height.  Lane j owns column j, a warp U
// rows; M is formed by every CTA for itself (a b^3 / 2 product: cheaper than a launch).
// Bound: FP64 issue, 2 U + 4 products of 32 FMAs a warp: U = 4 takes 29 us whatever n, so few rows go to
// more CTAs: U = 1 15 us, U = 2 20 us.
template <int U>
__global__ void __launch_bounds__(256) k_panel_w(int n, int nb, const double* __restrict__ V, int ldv,
                                                 const double* __restrict__ Y, const double* __restrict__ T,
                                                 const double* __restrict__ S, double* __restrict__ Wa,
                                                 double* __restrict__ Wb, int r0, const int* st) {
  __shared__ double Tm[PQN][PQN + 1], Sm[PQN][PQN + 1], Mm[PQN][PQN + 1];
  constexpr int ROWS = 8 * U;
  __shared__ double yt[PQN][ROWS + 1], vt[PQN][ROWS + 1];
  if (status_bad(st)) return;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (int idx = blockIdx.x * blockDim.x + tid; idx < r0 * nb; idx += gridDim.x * blockDim.x) {
    const size_t o = (size_t)(idx / r0) * ldv + idx % r0;
    Wa[o] = 0.0;
    Wb[o] = 0.0;
  }
  for (int idx = tid; idx < PQN * PQN; idx += 256) {
    const int i = idx & 31, j = idx >> 5;
    const bool in = i < nb && j < nb;
    Tm[i][j] = in && i <= j ? T[i + j * nb] : 0.0;
    Sm[i][j] = in ? S[i + j * nb] : 0.0;
  }
  __syncthreads();
#pragma unroll
  for (int i = warp; i < PQN; i += 8) {
    double s = 0.0;
    for (int q = 0; q <= i; ++q) s = fma(Tm[q][i], Sm[q][lane], s);
    Mm[i][lane] = 0.5 * s;
  }
  for (int b0 = blockIdx.x * ROWS; b0 < n; b0 += gridDim.x * ROWS) {
    __syncthreads();
    for (int idx = tid; idx < ROWS * nb; idx += 256) {
      const int r = b0 + idx % ROWS, j = idx / ROWS;
      yt[j][idx % ROWS] = r < n ? Y[r + (size_t)j * n] : 0.0;
      vt[j][idx % ROWS] = r < n ? V[r + (size_t)j * ldv] : 0.0;
    }
    __syncthreads();
    double y[U];
#pragma unroll
    for (int u = 0; u < U; ++u) y[u] = lane < nb ? yt[lane][warp * U + u] : 0.0;
#pragma unroll 4
    for (int q = 0; q < nb; ++q) {
      const double m = Mm[q][lane];
#pragma unroll
      for (int u = 0; u < U; ++u) y[u] = fma(-vt[q][warp * U + u], m, y[u]);
    }
    double w[U];
#pragma unroll
    for (int u = 0; u < U; ++u) w[u] = 0.0;
#pragma unroll 4
    for (int q = 0; q < nb; ++q) {
      const double t = Tm[q][lane];
#pragma unroll
      for (int u = 0; u < U; ++u) w[u] = fma(__shfl_sync(0xffffffffu, y[u], q), t, w[u]);
    }
    __syncthreads();
    if (lane < nb)
#pragma unroll
      for (int u = 0; u < U; ++u) yt[lane][warp * U + u] = w[u];
    __syncthreads();
    for (int idx = tid; idx < ROWS * nb; idx += 256) {
      const int r = b0 + idx % ROWS, j = idx / ROWS;
      if (r >= n) continue;
      const size_t o = (size_t)j * ldv + r0 + r;
      Wa[o] = yt[j][idx % ROWS];
      Wb[o] = yt[j][idx % ROWS];
    }
  }
}

// V (n x nb, ld n): unit lower trapezoidal factor of the panel QR stored in P.
__global__ void k_panel_v(int n, int nb, const double* __restrict__ P, int ldp, double* __restrict__ V,
                          const int* st) {
  if (status_bad(st)) return;
  int r = blockIdx.x * blockDim.x + threadIdx.x, q = blockIdx.y;
  if (r >= n || q >= nb) return;
  V[r + (size_t)q * n] = r < q ? 0.0 : (r == q ? 1.0 : P[r + (size_t)q * ldp]);
}

// ------------------------------------------------------------------ S1c bulge chasing

// Lower band storage with room for the bulge: AB[o + j*ldab] = C(j + o, j), 0 <= o < 2b.
__global__ void k_band_copy(int M, int b, const double* __restrict__ C, int ldc, double* __restrict__ AB, int ldab,
                            const int* st) {
  if (status_bad(st)) return;
  int o = threadIdx.x, j = blockIdx.x;
  if (o >= ldab || j >= M) return;
  AB[o + (size_t)j * ldab] = (o <= b && j + o < M) ? C[(j + o) + (size_t)j * ldc] : 0.0;
}

__device__ __forceinline__ int bulge_steps(int M, int b, int s) { return (M - 2 - s) / b + 1; }

struct BulgeArgs {
  int M, b, ldab, Q;  // Q = (M - 2) / b: groups 0..Q of b sweeps
  double* AB;
  int* prog;          // prog[s] = steps of sweep s completed (k_bulge_ws: see there)
  double* q2;         // diamond storage (or null)
  int* st;
  const unsigned long long* mx;  // norm bounds (k_band_rowsum) where both arithmetics are launched, else null
  unsigned long long wait_ns;  // limit of each progress wait
  int drop_sweep;              // test hook: this sweep publishes no progress (-1: none)
};

// Diamond (j, k) base in the reflector storage: [V: 2b x b][tau: b][T: b x b].
__host__ __device__ __forceinline__ size_t diamond_elems(int b) { return (size_t)3 * b * b + b; }
__host__ __device__ __forceinline__ size_t diamond_index(int Q, int j, int k) {
  return (size_t)j * (Q + 1) - (size_t)j * (j - 1) / 2 + k;
}

// dlarfg on x[0..len) (shared): v[0] = 1, v[i] = x[i] / (alpha - beta); returns tau, beta in out[0..1].  The
// squares are those of x scaled by the power of two out[3] into [1, 2): the bands that run in FP64 are those with
// rows of very different scale.
__device__ void house(const double* x, int len, double* v, double* out, int b) {
  const int t = threadIdx.x;
  if (t < 32) {
    int E = 0;
    for (int i = t; i < len; i += 32) E = max(E, (int)((__double_as_longlong(x[i]) >> 52) & 0x7FF));
    E = min(max(__reduce_max_sync(0xffffffffu, E), 23), 2023);
    const double f = __longlong_as_double((ll)(2046 - E) << 52), fi = __longlong_as_double((ll)E << 52);
    double s = 0.0;
    for (int i = 1 + t; i < len; i += 32) s += (x[i] * f) * (x[i] * f);
    for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (t < 2) {  // lane 0 forms tau, lane 1 the scale: one division sequence for both
      double alpha = x[0] * f, be = alpha, q = 0.0;
      if (s > 0.0) {
        be = -copysign(sqrt(alpha * alpha + s), alpha);
        const double num = (t == 0) ? be - alpha : 1.0, den = (t == 0) ? be : alpha - be;
        q = num / den;
      }
      out[t == 0 ? 0 : 2] = q;
      if (t == 0) {
        out[1] = be * fi;
        out[3] = f;
      }
    }
  }
  __syncthreads();
  const double sl = out[2], f = out[3];
  for (int i = t; i < b; i += blockDim.x) v[i] = (i == 0) ? 1.0 : (i < len ? (x[i] * f) * sl : 0.0);
  __syncthreads();
}

// D (len x len, full on entry, ld BMAX+1) <- H D H, H = I - tau v v^T; only the lower
// triangle of the result is formed.
__device__ void two_sided(double* D, int len, const double* v, double tau, double* p, double* red) {
  const int t = threadIdx.x, i = t & 63, part = t >> 6;
  double s = 0.0;
  if (i < len)
    for (int q = part; q < len; q += 4) s += D[i * (BMAX + 1) + q] * v[q];
  red[part * BMAX + i] = s;
  __syncthreads();
  if (t < len) p[t] = tau * (red[t] + red[BMAX + t] + red[2 * BMAX + t] + red[3 * BMAX + t]);
  __syncthreads();
  if (t < 32) {  // K = tau/2 p^T v
    double k = 0.0;
    for (int q = t; q < len; q += 32) k += p[q] * v[q];
    for (int o = 16; o; o >>= 1) k += __shfl_xor_sync(0xffffffffu, k, o);
    if (t == 0) red[4 * BMAX] = 0.5 * tau * k;
  }
  __syncthreads();
  double K = red[4 * BMAX];
  if (t < len) p[t] -= K * v[t];  // w
  __syncthreads();
  // lower triangle only: the block is stored back as its lower part and re-read (and
  // mirrored) from the band at every step
  for (int idx = t; idx < len * len; idx += blockDim.x) {
    int a = idx % len, c = idx / len;
    if (a >= c) D[a * (BMAX + 1) + c] -= v[a] * p[c] + p[a] * v[c];
  }
  __syncthreads();
}

// Norm bounds of the band (k_band_rowsum): mx[0] largest absolute row sum, mx[1] the complement of the smallest one
// beside the first column (bits of doubles), mx[2] bit 0: two neighbours further apart than 2^4, bit 1: a row of
// zeros.  One fixed-point unit for the whole band, 2^-61 of mx[0], takes the relative accuracy of a block far below the
// rest if that is decoupled: such a block begins with a jump between neighbours (or beyond a row of zeros),
// and the band stays FP64.  Where the rows fall off slowly FP64 mixes them as well; there the unit has to
// be no coarser than FP64's at the smallest row.  Decoupled blocks at 2^-4, 2^-6, 2^-8 of the rest, order 500: mean
// error of their eigenvalues 0.8, 1.6, 5.4e-15 in fixed point, 0.7e-15 in FP64.  Tight-binding bands of order
// 512 to 16384 have neighbours within 5.2 and rows within 13 to 106: 57 ms at order 8192 instead of 182.
__device__ __forceinline__ bool band_wide(const unsigned long long* mx) {
  const double hi = __longlong_as_double((ll)mx[0]), lo = __longlong_as_double((ll)~mx[1]);
  return mx[1] != 0 && (mx[0] >> 52) < 0x7FF && ((mx[2] & 1) || lo < ((mx[2] & 2) ? 0x1p-4 : 0x1p-8) * hi);
}

__global__ void __launch_bounds__(256) k_bulge(BulgeArgs a) {
  extern __shared__ double sm[];
  double* Bm = sm;                          // BMAX x (BMAX+1), [row][col]
  double* Dm = Bm + BMAX * (BMAX + 1);
  double* vp = Dm + BMAX * (BMAX + 1);      // previous reflector
  double* vc = vp + BMAX;                   // current reflector
  double* xv = vc + BMAX;                   // column to annihilate / scratch
  double* pw = xv + BMAX;
  double* red = pw + BMAX;                  // 4*BMAX + 1
  double* hs = red + 4 * BMAX + 8;          // tau, beta, the two factors of the scale
  __shared__ int abort_flag;
  const int t = threadIdx.x, M = a.M, b = a.b, ldab = a.ldab;
  if (t == 0) abort_flag = 0;
  __syncthreads();
  if (status_bad(a.st) || (a.mx && !band_wide(a.mx))) return;
  for (int s = blockIdx.x; s <= M - 2; s += gridDim.x) {
    const int ns = bulge_steps(M, b, s);
    double taup = 0.0;
    for (int k = 0; k < ns; ++k) {
      if (s > 0 && t == 0) {  // step k of sweep s needs step k+1 of sweep s-1
        int pns = bulge_steps(M, b, s - 1);
        int need = k + 2 < pns ? k + 2 : pns;
        unsigned long long t0 = gclock();
        while (ld_acquire(a.prog + (s - 1)) < need) {
          if (*(volatile int*)(a.st + 1) != 0) { abort_flag = 1; break; }
          if (gclock() - t0 > a.wait_ns) {
            atomicExch(a.st + 1, GEP_ERR_TIMEOUT);
            abort_flag = 1;
            break;
          }
        }
      }
      __syncthreads();
      if (abort_flag) return;
      const int st_k = s + 1 + k * b;
      const int len = (M - st_k) < b ? (M - st_k) : b;
      {
        if (k == 0) {
          for (int i = t; i < len; i += blockDim.x) xv[i] = __ldcg(a.AB + (1 + i) + (size_t)s * ldab);
          __syncthreads();
          house(xv, len, vc, hs, b);
          if (t < len) a.AB[(1 + t) + (size_t)s * ldab] = (t == 0) ? hs[1] : 0.0;
        } else {
          const int stp = st_k - b;  // previous block's first row/column (its length is b)
          for (int idx = t; idx < len * b; idx += blockDim.x) {
            int i = idx % len, q = idx / len;
            Bm[i * (BMAX + 1) + q] = __ldcg(a.AB + (b + i - q) + (size_t)(stp + q) * ldab);
          }
          __syncthreads();
          {  // B <- B H(s,k-1): y = B vp, B -= taup y vp^T
            int i = t & 63, part = t >> 6;
            double y = 0.0;
            if (i < len)
              for (int q = part; q < b; q += 4) y += Bm[i * (BMAX + 1) + q] * vp[q];
            red[part * BMAX + i] = y;
            __syncthreads();
            if (t < len) pw[t] = taup * (red[t] + red[BMAX + t] + red[2 * BMAX + t] + red[3 * BMAX + t]);
            __syncthreads();
            for (int idx = t; idx < len * b; idx += blockDim.x) {
              int ii = idx % len, q = idx / len;
              Bm[ii * (BMAX + 1) + q] -= pw[ii] * vp[q];
            }
            __syncthreads();
          }
          for (int i = t; i < len; i += blockDim.x) xv[i] = Bm[i * (BMAX + 1)];
          __syncthreads();
          house(xv, len, vc, hs, b);
          {  // B(:, 1:) <- H B(:, 1:): u = tau B^T v
            double tk = hs[0];
            int q = t & 63, part = t >> 6;
            double u = 0.0;
            if (q >= 1 && q < b)
              for (int i = part; i < len; i += 4) u += vc[i] * Bm[i * (BMAX + 1) + q];
            red[part * BMAX + q] = u;
            __syncthreads();
            if (t < b) pw[t] = tk * (red[t] + red[BMAX + t] + red[2 * BMAX + t] + red[3 * BMAX + t]);
            __syncthreads();
            for (int idx = t; idx < len * b; idx += blockDim.x) {
              int i = idx % len, qq = idx / len;
              double x;
              if (qq == 0) x = (i == 0) ? hs[1] : 0.0;
              else x = Bm[i * (BMAX + 1) + qq] - vc[i] * pw[qq];
              a.AB[(b + i - qq) + (size_t)(stp + qq) * ldab] = x;
            }
          }
        }
        // D = C(st_k : st_k+len, same) <- H D H
        for (int idx = t; idx < len * len; idx += blockDim.x) {
          int i = idx % len, q = idx / len;
          int lo = i > q ? i : q, hi = i > q ? q : i;
          Dm[i * (BMAX + 1) + q] = __ldcg(a.AB + (lo - hi) + (size_t)(st_k + hi) * ldab);
        }
        __syncthreads();
        double tk = hs[0];
        two_sided(Dm, len, vc, tk, pw, red);
        for (int idx = t; idx < len * len; idx += blockDim.x) {
          int i = idx % len, q = idx / len;
          if (i >= q) a.AB[(i - q) + (size_t)(st_k + q) * ldab] = Dm[i * (BMAX + 1) + q];
        }
      }
      const double tk = hs[0];
      if (a.q2) {  // reflector into diamond (j, k), column c
        int j = s / b, c = s - j * b;
        double* D0 = a.q2 + diamond_index(a.Q, j, k) * diamond_elems(b);
        for (int i = t; i < len; i += blockDim.x) D0[(c + i) + (size_t)c * 2 * b] = vc[i];
        if (t == 0) D0[(size_t)2 * b * b + c] = tk;
      }
      if (t < b) vp[t] = vc[t];
      taup = tk;
      __syncthreads();  // every thread's stores of this step precede the release below
      if (t == 0 && s != a.drop_sweep) {
        __threadfence();
        st_release(a.prog + s, k + 1);
      }
    }
  }
}

// ---- bulge chasing for b = N = 32 or 64: fixed point, warp-specialised
//
// Arithmetic.  The band is held as 64-bit integers q with C = q 2^-sh, sh chosen so that the
// largest absolute row sum of the band (a bound on its 2-norm, which no similarity changes) is
// at most 2^61 (rows too far apart for one unit: band_wide); reflectors have v in Q62 (|v_i| <= 1 by construction), tau in Q61.  The norms
// in play (v^T v <= 2, tau |v| <= 2, w = tau C v - ... at most 2 |C|) keep every intermediate
// below 2^63.  A product drops only the low x low limb: its error is about half a unit, 2^-62
// of the row-sum bound, where an FP64 operation rounds its result at 2^-54; every term is rounded by
// itself (a constant for the floors of a sum would leave noise in rows beyond the matrix and turn
// zeros into 2^-57).  A reflector's scalars come from exact squares (q_reflector).  An FP64 instruction holds a scheduler for 64 clocks on this part; the three
// 32 x 32 -> 64 multiply-adds of a fixed-point product and their shifts take about 20.
//
// Schedule.  A sweep's reflectors form a chain of their own: x of step k + 1 is column 0 of
// B_{k+1} H(s, k), which needs H(s, k) but not the updates of step k.  So the finder warps run
// that chain one step ahead of the appliers, of which one group updates B of the step and the
// other D; they hand over through shared memory (two buffers, mbarriers).  Likewise step k of
// sweep s + 1 needs of step k + 1 of sweep s only the element beta = (H B)(0, 0) before its
// reflector, and the rest of that step (the last row of its D) only before its D update.  Two
// progress counters per sweep publish the two events: prog[s] counts steps whose beta is
// stored, prog[M + s] steps stored completely; one warp of a group polls.
//
// Bound: latency, one find + apply + flag through L2 per sweep.  Measured (the FP64 kernel at
// b = 64 with one role -> this one at b = 64 / b = 32): order 516 14.9 -> 5.4 / 2.6 ms, 2047
// 64 -> 24 / 11 ms, 8192 262 -> 100 / 60 ms (7.3 us a sweep; an FP64 build of the same schedule
// took 222 / 102 ms).
constexpr int BC = 8;  // columns per warp in every role: N / BC finder warps, as many for B and for D
template <int N>
struct BulgeShared {
  ll Bs[2][N][N + 1];  // [column][row] of the step's block
  ll Ds[N][N + 1];     // diagonal block, both triangles
  ll redA[N / BC][N], x0[N];
  ll redU[N / BC][N], redD[N / BC][N];
  int2 yv[2][N], vp[2][N], vc[2][N];  // split into limbs
  ll sc[2][2];                        // tau (Q61), beta
  unsigned long long full_y[2], full_v[2], empty[2];
  int abort_a[2], abort_u[2];
};

__device__ __forceinline__ uint32_t sm32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mb_init(unsigned long long* b, int n) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(sm32(b)), "r"(n) : "memory");
}
__device__ __forceinline__ void mb_arrive(unsigned long long* b) {
  asm volatile("{ .reg .b64 t; mbarrier.arrive.shared::cta.b64 t, [%0]; }" ::"r"(sm32(b)) : "memory");
}
// Bounded wait inside the CTA: gives up when an error has been recorded, or records a timeout.
__device__ bool mb_wait(unsigned long long* b, uint32_t parity, const BulgeArgs& a) {
  unsigned long long t0 = 0;
  for (int it = 0;; ++it) {
    uint32_t ok;
    asm volatile("{ .reg .pred p; mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2; selp.u32 %0, 1, 0, p; }"
                 : "=r"(ok) : "r"(sm32(b)), "r"(parity) : "memory");
    if (ok) return true;
    if ((it & 63) == 63) {
      if (*(volatile int*)(a.st + 1) != 0) return false;
      const unsigned long long now = gclock();
      if (t0 == 0) t0 = now;
      else if (now - t0 > a.wait_ns + 2000000000ull) {
        atomicExch(a.st + 1, GEP_ERR_TIMEOUT);
        return false;
      }
    }
  }
}
// Bounded wait of a warp until *p >= need and *q >= needq (lanes 0 and 1 poll together).
__device__ __forceinline__ bool prog_wait(const int* p, int need, const int* q, int needq, const BulgeArgs& a) {
  const int lane = threadIdx.x & 31, want = lane ? needq : need;
  const int* w = lane ? q : p;
  unsigned long long t0 = 0;
  for (int it = 0;; ++it) {
    const int ok = lane < 2 ? ld_acquire(w) >= want : 1;
    if (__all_sync(0xffffffffu, ok)) {
      __syncwarp();
      return true;
    }
    if ((it & 15) == 15) {
      const unsigned long long now = gclock();
      if (t0 == 0) t0 = now;
      int dead = *(volatile int*)(a.st + 1) != 0;
      if (!dead && now - t0 > a.wait_ns) {
        atomicExch(a.st + 1, GEP_ERR_TIMEOUT);
        dead = 1;
      }
      if (__any_sync(0xffffffffu, dead)) return false;
    }
  }
}
template <int ID, int WARPS>
__device__ __forceinline__ void group_sync() { asm volatile("bar.sync %0, %1;" ::"n"(ID), "n"(32 * WARPS) : "memory"); }

template <int N>
constexpr int bulge_threads() { return 32 * 3 * (N / BC); }

template <int N>
__global__ void __launch_bounds__(bulge_threads<N>()) k_bulge_ws(BulgeArgs a) {
  constexpr int R = N / 32, LD = 2 * N;  // rows per lane, band leading dimension
  constexpr int G = N / BC, C = BC;      // warps of a group, columns per warp
  extern __shared__ __align__(16) unsigned char smraw[];
  BulgeShared<N>& sh = *reinterpret_cast<BulgeShared<N>*>(smraw);
  const int t = threadIdx.x, lane = t & 31, wid = t >> 5, M = a.M;
  ll* AB = reinterpret_cast<ll*>(a.AB);
  if (t == 0) {
    for (int q = 0; q < 2; ++q) {
      mb_init(&sh.full_y[q], 32 * G);
      mb_init(&sh.full_v[q], 32);
      mb_init(&sh.empty[q], 64 * G);
      sh.abort_a[q] = sh.abort_u[q] = 0;
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  if (status_bad(a.st) || band_wide(a.mx)) return;
  int* progA = a.prog;
  int* progF = a.prog + M;
  int g = 0;  // steps of this CTA so far (every role counts the same)
  if (wid < G) {
    // ---------------- finders
    const int w = wid;
    for (int s = blockIdx.x; s <= M - 2; s += gridDim.x) {
      const int ns = bulge_steps(M, N, s), pns = s > 0 ? bulge_steps(M, N, s - 1) : 0;
      int2 v[R], taup = make_int2(0, 0);
#pragma unroll
      for (int r = 0; r < R; ++r) v[r] = make_int2(0, 0);
      for (int k = 0; k < ns; ++k, ++g) {
        const int buf = g & 1;
        if (w == 0) {
          bool ok = s == 0 || prog_wait(progF + s - 1, min(k + 1, pns), progA + s - 1, min(k + 2, pns), a);
          if (ok && g >= 2) ok = mb_wait(&sh.empty[buf], ((uint32_t)(g >> 1) & 1u) ^ 1u, a);
          if (!ok) sh.abort_a[buf] = 1;
        }
        group_sync<1, G>();
        if (sh.abort_a[buf]) return;
        const int st_k = s + 1 + k * N, stp = st_k - N, len = min(M - st_k, N);
        ll x[R];
        if (k == 0) {
#pragma unroll
          for (int r = 0; r < R; ++r) {
            const int i = lane + 32 * r;
            x[r] = i < len ? __ldcg(AB + (1 + i) + (size_t)s * LD) : 0;
          }
        } else {
          ll b[R][C];
          const ll* Bp = AB + (size_t)stp * LD + N + lane + w * C * (LD - 1);
#pragma unroll
          for (int q = 0; q < C; ++q)
#pragma unroll
            for (int r = 0; r < R; ++r) b[r][q] = lane + 32 * r < len ? __ldcg(Bp + 32 * r + q * (LD - 1)) : 0;
          int2 vsel = v[0];
          if (R > 1 && w >= G / R) vsel = v[R - 1];  // the half of v that holds this warp's columns
          ll hh[R], mm[R];
#pragma unroll
          for (int r = 0; r < R; ++r) { hh[r] = 0; mm[r] = 0; }
#pragma unroll
          for (int q = 0; q < C; ++q) {
            int2 vq;
            vq.x = __shfl_sync(0xffffffffu, vsel.x, (w * C + q) & 31);
            vq.y = __shfl_sync(0xffffffffu, vsel.y, (w * C + q) & 31);
#pragma unroll
            for (int r = 0; r < R; ++r) {
              const int2 bb = qsplit(b[r][q]);
              hh[r] += qhh(bb, vq);
              mm[r] += qmid(bb, vq, 1ll << 29) >> 30;
            }
          }
#pragma unroll
          for (int r = 0; r < R; ++r) {
            const int i = lane + 32 * r;
            sh.redA[w][i] = (hh[r] << 2) + mm[r];
            if (w == 0) {
              sh.x0[i] = b[r][0];
              sh.vp[buf][i] = v[r];
            }
          }
          group_sync<1, G>();
#pragma unroll
          for (int r = 0; r < R; ++r) {
            const int i = lane + 32 * r;
            ll ys = 0;
#pragma unroll
            for (int q = 0; q < G; ++q) ys += sh.redA[q][i];
            const ll y = qmul<61>(qsplit(ys), taup);
            x[r] = sh.x0[i] - y;
            if (w == 0) sh.yv[buf][i] = qsplit(y);
          }
#pragma unroll
          for (int r = 0; r < R; ++r)
#pragma unroll
            for (int q = 0; q < C; ++q) sh.Bs[buf][w * C + q][lane + 32 * r] = b[r][q];
        }
        mb_arrive(&sh.full_y[buf]);
        // reflector of x, formed by every finder warp for itself, from the exact sum of the squares:
        // entries far below alpha must not vanish in it
        unsigned sq[6] = {0, 0, 0, 0, 0, 0};
#pragma unroll
        for (int r = 0; r < R; ++r) {
          const unsigned long long ax = lane + 32 * r > 0 ? (unsigned long long)(x[r] < 0 ? -x[r] : x[r]) : 0ull;
          add_square(sq, ax);
        }
        const Sum128 s2 = warp_squares(sq);
        const ll alpha_q = __shfl_sync(0xffffffffu, x[0], 0);
        QReflector o;
        o.m = o.tq = 0;
        o.beta = alpha_q;
        o.up = 0;
        if ((s2.lo | s2.hi) != 0) o = q_reflector(alpha_q, s2);
        const int2 mq = qsplit(o.m);
#pragma unroll
        for (int r = 0; r < R; ++r) v[r] = qsplit(qmul<61>(qsplit(x[r] << o.up), mq));
        const ll beq = o.beta, tauq = o.tq;
        taup = qsplit(tauq);
        if (lane == 0) v[0] = make_int2(0, 1 << 30);
        if (w == 0) {
#pragma unroll
          for (int r = 0; r < R; ++r) sh.vc[buf][lane + 32 * r] = v[r];
          if (lane == 0) {
            sh.sc[buf][0] = tauq;
            sh.sc[buf][1] = beq;
            AB[k == 0 ? 1 + (size_t)s * LD : N + (size_t)stp * LD] = beq;
          }
          mb_arrive(&sh.full_v[buf]);
          if (lane == 0 && s != a.drop_sweep) st_release(progA + s, k + 1);
        }
      }
    }
  } else if (wid < 2 * G) {
    // ---------------- appliers of B: B <- H(s,k) (B H(s,k-1)), lane = column, 8 rows a warp
    const int u = wid - G;
    for (int s = blockIdx.x; s <= M - 2; s += gridDim.x) {
      const int ns = bulge_steps(M, N, s);
      for (int k = 0; k < ns; ++k, ++g) {
        const int buf = g & 1;
        const uint32_t ph = (uint32_t)(g >> 1) & 1u;
        const int st_k = s + 1 + k * N, stp = st_k - N, len = min(M - st_k, N);
        bool ok = mb_wait(&sh.full_y[buf], ph, a);
        ll b[R][C];  // column c = lane + 32 r, rows u C + q
        if (k > 0) {
#pragma unroll
          for (int r = 0; r < R; ++r) {
            const int c = lane + 32 * r;
            const int2 vpc = sh.vp[buf][c];
#pragma unroll
            for (int q = 0; q < C; ++q) b[r][q] = sh.Bs[buf][c][u * C + q] - qmul<62>(sh.yv[buf][u * C + q], vpc);
          }
        }
        if (ok) ok = mb_wait(&sh.full_v[buf], ph, a);
        if (!ok) sh.abort_u[buf] = 1;
        if (k > 0) {
          ll zh[R], zm[R];
#pragma unroll
          for (int r = 0; r < R; ++r) {
            zh[r] = 0;
            zm[r] = 0;
          }
#pragma unroll
          for (int q = 0; q < C; ++q) {
            const int2 vq = sh.vc[buf][u * C + q];
#pragma unroll
            for (int r = 0; r < R; ++r) {
              const int2 bb = qsplit(b[r][q]);
              zh[r] += qhh(bb, vq);
              zm[r] += qmid(bb, vq, 1ll << 29) >> 30;
            }
          }
#pragma unroll
          for (int r = 0; r < R; ++r) sh.redU[u][lane + 32 * r] = (zh[r] << 2) + zm[r];
          group_sync<2, G>();
          const int2 tau = qsplit(sh.sc[buf][0]);
          const ll be = sh.sc[buf][1];
#pragma unroll
          for (int r = 0; r < R; ++r) {
            const int c = lane + 32 * r;
            ll zs = 0;
#pragma unroll
            for (int q = 0; q < G; ++q) zs += sh.redU[q][c];
            const int2 zc = qsplit(qmul<61>(qsplit(zs), tau));
#pragma unroll
            for (int q = 0; q < C; ++q) {
              const int i = u * C + q;
              const ll x = b[r][q] - qmul<62>(zc, sh.vc[buf][i]);
              sh.Bs[buf][c][i] = c == 0 ? (i == 0 ? be : 0) : x;
            }
          }
          group_sync<2, G>();  // stored with lane = row, so that a warp's stores are contiguous
          ll* Bp = AB + (size_t)stp * LD + N + lane + u * C * (LD - 1);
#pragma unroll
          for (int q = 0; q < C; ++q)
#pragma unroll
            for (int r = 0; r < R; ++r) {
              const int i = lane + 32 * r, c = u * C + q;
              if (i < len && (i | c) != 0) Bp[32 * r + q * (LD - 1)] = sh.Bs[buf][c][i];
            }
        } else if (u == 0) {
#pragma unroll
          for (int r = 0; r < R; ++r) {
            const int i = lane + 32 * r;
            if (i > 0 && i < len) AB[(1 + i) + (size_t)s * LD] = 0;
          }
        }
        if (a.q2 && u == G - 1) {  // reflector into diamond (j, k), column c
          const int j = s / N, c = s - j * N;
          double* D0 = a.q2 + diamond_index(a.Q, j, k) * diamond_elems(N);
#pragma unroll
          for (int r = 0; r < R; ++r)
            if (lane + 32 * r < len)
              D0[(c + lane + 32 * r) + (size_t)c * 2 * N] = (double)qjoin(sh.vc[buf][lane + 32 * r]) * 0x1p-62;
          if (lane == 0) D0[(size_t)2 * N * N + c] = qscaled(sh.sc[buf][0], 61);
        }
        mb_arrive(&sh.empty[buf]);
        group_sync<4, 2 * G>();  // the stores of both groups precede the release
        if (sh.abort_u[buf]) return;
      }
    }
  } else {
    // ---------------- appliers of D: D <- H D H on the lower triangle, lane = row, 8 columns a warp
    const int u = wid - 2 * G;
    for (int s = blockIdx.x; s <= M - 2; s += gridDim.x) {
      const int ns = bulge_steps(M, N, s), pns = s > 0 ? bulge_steps(M, N, s - 1) : 0;
      for (int k = 0; k < ns; ++k, ++g) {
        const int buf = g & 1;
        const uint32_t ph = (uint32_t)(g >> 1) & 1u;
        const int st_k = s + 1 + k * N, len = min(M - st_k, N);
        if (u == 0 && s > 0) {
          const int need = min(k + 2, pns);
          if (!prog_wait(progF + s - 1, need, progF + s - 1, need, a)) sh.abort_u[buf] = 1;
        }
        group_sync<3, G>();
        ll dv[R][C];
        ll* Dp = AB + (size_t)st_k * LD + lane + u * C * (LD - 1);
#pragma unroll
        for (int q = 0; q < C; ++q)
#pragma unroll
          for (int r = 0; r < R; ++r) {
            const int i = lane + 32 * r, c = u * C + q;
            dv[r][q] = (i >= c && i < len) ? __ldcg(Dp + 32 * r + q * (LD - 1)) : 0;
          }
#pragma unroll
        for (int q = 0; q < C; ++q)
#pragma unroll
          for (int r = 0; r < R; ++r) {
            const int i = lane + 32 * r, c = u * C + q;
            if (i >= c) {
              sh.Ds[c][i] = dv[r][q];
              sh.Ds[i][c] = dv[r][q];
            }
          }
        if (!mb_wait(&sh.full_v[buf], ph, a)) sh.abort_u[buf] = 1;
        group_sync<3, G>();
        const int2 tau = qsplit(sh.sc[buf][0]);
        int2 vr[R];
        ll hh[R], mm[R];
#pragma unroll
        for (int r = 0; r < R; ++r) {
          vr[r] = sh.vc[buf][lane + 32 * r];
          hh[r] = 0;
          mm[r] = 0;
        }
#pragma unroll
        for (int q = 0; q < C; ++q) {
          const int2 vq = sh.vc[buf][u * C + q];
#pragma unroll
          for (int r = 0; r < R; ++r) {
            const int2 dd = qsplit(sh.Ds[u * C + q][lane + 32 * r]);
            hh[r] += qhh(dd, vq);
            mm[r] += qmid(dd, vq, 1ll << 29) >> 30;
          }
        }
#pragma unroll
        for (int r = 0; r < R; ++r) sh.redD[u][lane + 32 * r] = (hh[r] << 2) + mm[r];
        group_sync<3, G>();
        ll p[R], K = 0;
#pragma unroll
        for (int r = 0; r < R; ++r) {
          ll ps = 0;
#pragma unroll
          for (int q = 0; q < G; ++q) ps += sh.redD[q][lane + 32 * r];
          p[r] = qmul<61>(qsplit(ps), tau);
          K += qmul<62>(qsplit(p[r]), vr[r]);
        }
        const int2 Kh = qsplit(qmul<62>(qsplit(qwarp_sum(K)), tau));  // tau / 2 p^T v
        int2 wv[R];
#pragma unroll
        for (int r = 0; r < R; ++r) wv[r] = qsplit(p[r] - qmul<62>(Kh, vr[r]));
        int2 wsel = wv[0];
        if (R > 1 && u >= G / R) wsel = wv[R - 1];
#pragma unroll
        for (int q = 0; q < C; ++q) {
          const int c = u * C + q;
          int2 wc;
          wc.x = __shfl_sync(0xffffffffu, wsel.x, c & 31);
          wc.y = __shfl_sync(0xffffffffu, wsel.y, c & 31);
          const int2 vq = sh.vc[buf][c];
#pragma unroll
          for (int r = 0; r < R; ++r) {
            const int i = lane + 32 * r;
            if (32 * r + 31 < c) continue;  // the whole warp lies above the diagonal
            const ll x = dv[r][q] - qmul<62>(vr[r], wc) - qmul<62>(wv[r], vq);
            if (i >= c && i < len) Dp[32 * r + q * (LD - 1)] = x;
          }
        }
        mb_arrive(&sh.empty[buf]);
        group_sync<4, 2 * G>();  // the stores of both groups precede the release
        if (sh.abort_u[buf]) return;
        if (u == 0 && lane == 0 && s != a.drop_sweep) st_release(progF + s, k + 1);
      }
    }
  }
}

// Norm bounds of the band matrix for band_wide and band_shift (mx zero on entry).
__global__ void k_band_rowsum(int M, int b, const double* __restrict__ AB, int ldab, unsigned long long* mx,
                              const int* st) {
  if (status_bad(st)) return;
  const int i = blockIdx.x * blockDim.x + threadIdx.x, lane = threadIdx.x & 31;
  // row r beside the first column, and first: its entry there (of row 0: the diagonal)
  auto beside = [&](int r, double& first) {
    double s = 0.0;
    first = r <= b ? fabs(AB[r]) : 0.0;
    for (int o = r == 0 ? 1 : 0; o <= b && r + o < M; ++o) s += fabs(AB[o + (size_t)r * ldab]);
    for (int o = 1; o <= b && o < r; ++o) s += fabs(AB[o + (size_t)(r - o) * ldab]);
    return s;
  };
  double rest = 0.0, first = 0.0;
  if (i < M) rest = beside(i, first);
  unsigned long long v = (unsigned long long)__double_as_longlong(rest + first), bits = i < M && rest == 0.0 ? 2 : 0;
  if (i == 0 && rest == 0.0) rest = first;  // a decoupled first row
  double above = __shfl_up_sync(0xffffffffu, rest, 1), unused;
  if (lane == 0) above = i > 1 && i < M ? beside(i - 1, unused) : rest;
  if (i > 1 && i < M && rest > 0.0 && above > 0.0 && fmin(rest, above) < 0x1p-4 * fmax(rest, above)) bits |= 1;
  unsigned long long u = rest > 0.0 ? ~(unsigned long long)__double_as_longlong(rest) : 0;
  for (int o = 16; o; o >>= 1) {
    const unsigned long long q = __shfl_xor_sync(0xffffffffu, v, o), p = __shfl_xor_sync(0xffffffffu, u, o);
    if (q > v) v = q;
    if (p > u) u = p;
    bits |= __shfl_xor_sync(0xffffffffu, bits, o);
  }
  if (lane == 0) {
    if (v) atomicMax(mx, v);
    if (u) atomicMax(mx + 1, u);
    if (bits) atomicOr(mx + 2, bits);
  }
}

// sh with (largest row sum) 2^sh in (2^60, 2^61]
__device__ __forceinline__ int band_shift(const unsigned long long* mx) {
  const int E = (int)(*mx >> 52);  // sum < 2^(E - 1022)
  return E ? 61 - (E - 1022) : 0;
}

__global__ void k_band_fix(int M, double* AB, int ldab, const unsigned long long* mx, const int* st) {
  if (status_bad(st) || band_wide(mx)) return;
  const int sh = band_shift(mx);
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < (size_t)M * ldab; i += (size_t)gridDim.x * blockDim.x) {
    const double x = AB[i];
    reinterpret_cast<ll*>(AB)[i] = x == 0.0 ? 0 : __double2ll_rn(scale2(x, sh));
  }
}

__global__ void k_band_diag_fix(int M, const double* __restrict__ AB, int ldab, const unsigned long long* mx,
                                double* __restrict__ d, double* __restrict__ e, const int* st) {
  if (status_bad(st)) return;
  const int i = blockIdx.x * blockDim.x + threadIdx.x, sh = band_shift(mx);
  if (i >= M) return;
  if (band_wide(mx)) {
    d[i] = AB[(size_t)i * ldab];
    if (i + 1 < M) e[i] = AB[1 + (size_t)i * ldab];
    return;
  }
  const ll* q = reinterpret_cast<const ll*>(AB);
  const bool finite = (*mx >> 52) < 0x7FF;  // an integer cannot carry a NaN or an infinity of the band
  d[i] = finite ? scale2((double)q[(size_t)i * ldab], -sh) : NAN;
  if (i + 1 < M) e[i] = finite ? scale2((double)q[1 + (size_t)i * ldab], -sh) : NAN;
}

__global__ void k_band_diag(int M, const double* __restrict__ AB, int ldab, double* __restrict__ d,
                            double* __restrict__ e, const int* st) {
  if (status_bad(st)) return;
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= M) return;
  d[i] = AB[(size_t)i * ldab];
  if (i + 1 < M) e[i] = AB[1 + (size_t)i * ldab];
}

// ------------------------------------------------------------------ Q2 application

constexpr int Q2_COLS = 64;  // Z columns per CTA

// Z <- G(j,k) Z for every diamond of wavefront t (blockIdx.x) on a slab of Q2_COLS
// columns (blockIdx.y).  G(j,k) = H(s0,k) ... H(s0+b-1,k) is applied reflector by
// reflector, the last one first.  Each Z column is owned by four lanes of one warp.
__global__ void __launch_bounds__(256) k_q2_apply(int M, int b, int Q, int wt, const double* __restrict__ q2,
                                                  double* __restrict__ Z, int ldz, int ncol, const int* st) {
  extern __shared__ double sm[];
  if (status_bad(st)) return;
  const int kmin = wt - Q > 0 ? wt - Q : 0;
  const int k = kmin + blockIdx.x;
  if (2 * k > wt) return;  // k <= wt / 2 keeps j + k <= Q
  const int j = Q - wt + k;
  if (j < 0 || j > Q || k > Q - j) return;
  const int L = 2 * b - 1;
  const int r0 = 1 + (j + k) * b;
  const int c0 = blockIdx.y * Q2_COLS;
  double* Vs = sm;                      // [c][2b]
  double* Zs = Vs + (size_t)2 * b * b;  // [row][Q2_COLS + 1]
  double* ts = Zs + (size_t)L * (Q2_COLS + 1);
  const double* D0 = q2 + diamond_index(Q, j, k) * diamond_elems(b);
  const int t = threadIdx.x;
  for (int idx = t; idx < 2 * b * b; idx += blockDim.x) Vs[idx] = D0[idx];
  if (t < b) ts[t] = D0[(size_t)2 * b * b + t];
  for (int idx = t; idx < L * Q2_COLS; idx += blockDim.x) {
    int r = idx % L, cc = idx / L;
    int gr = r0 + r, gc = c0 + cc;
    Zs[r * (Q2_COLS + 1) + cc] = (gr < M && gc < ncol) ? Z[gr + (size_t)gc * ldz] : 0.0;
  }
  __syncthreads();
  const int col = t >> 2, part = t & 3;
  for (int c = b - 1; c >= 0; --c) {
    double tc = ts[c];
    if (tc == 0.0) continue;
    const double* v = Vs + (size_t)c * 2 * b;
    double u = 0.0;
    for (int r = c + part; r < c + b; r += 4) u += v[r] * Zs[r * (Q2_COLS + 1) + col];
    u += __shfl_xor_sync(0xffffffffu, u, 1);
    u += __shfl_xor_sync(0xffffffffu, u, 2);
    u *= tc;
    for (int r = c + part; r < c + b; r += 4) Zs[r * (Q2_COLS + 1) + col] -= u * v[r];
    __syncwarp();
  }
  __syncthreads();
  for (int idx = t; idx < L * Q2_COLS; idx += blockDim.x) {
    int r = idx % L, cc = idx / L;
    int gr = r0 + r, gc = c0 + cc;
    if (gr < M && gc < ncol) Z[gr + (size_t)gc * ldz] = Zs[r * (Q2_COLS + 1) + cc];
  }
}

// Dense tiles of Q2.  Tile (J, K) holds the diamonds (j, k) with j in [J TQ, (J+1) TQ)
// and k in [K TQ, (K+1) TQ); diamond (j, k) acts on rows 1 + (j + k) b .. + 2b - 2, so
// the tile acts on the W = 2 TQ b rows starting at 1 + (J + K) TQ b.  A diamond must
// precede (j, k+1) and, where rows overlap, the diamonds (j-1, k'), k' >= k of the next
// lower group: every dependency keeps or lowers j and keeps or raises k, so tiles are
// applied with J descending and K ascending, and inside a tile with j descending and k
// ascending.  U(J, K) is the product of its diamonds in that order, built by applying
// them to the identity, W x TB_COLS columns per CTA, and stored as U - I so that a tile
// is applied as Z(rows) += (U - I) Z(rows).
// Diamonds per tile side: W = 2 TQ b = 512 for b = 32 and 64, the depth of one exact chunk of the
// product kernel.
__host__ __device__ constexpr int tile_q(int b) { return b == 32 ? 8 : 4; }
constexpr int TB_COLS = 32;  // tile columns per CTA in the build (8 lanes per column)
constexpr int TB_LD = TB_COLS + 2;  // (8 rows x 2 columns of a half warp then fall into distinct banks)

// Tile index t (tile rows J ascending, then K) -> (J, K); nK(J) = (Q - J TQ) / TQ + 1.
__device__ __forceinline__ void tile_of_index(int Q, int TQ, int t, int& J, int& K) {
  J = 0;
  for (int nK; t >= (nK = (Q - J * TQ) / TQ + 1); ++J) t -= nK;
  K = t;
}

// The arithmetic is the fixed point of the bulge-chasing kernel (entries of U and v in Q62, all at
// most 1 in magnitude; tau in Q61), about a third of the FP64 issue time and exact to 2^-61 per
// operation.  Eight lanes share a column; a diamond's reflectors are turned into limbs in shared
// memory once per CTA, the next diamond's being fetched meanwhile.
// Bound: integer issue (about 100 instructions a reflector for 8 warps) and its latency.  Measured
// (D&C beside the build, then the back-transformation; b = 32): order 2047 5.8 + 24.6 -> 9.2 +
// 10.1 ms, order 8192 115 + 167 -> 88 + 146 ms.  All tiles are one launch (a launch per tile row
// left most SMs idle).
__global__ void __launch_bounds__(256) k_q2_tile_build(int b, int Q, const double* __restrict__ q2,
                                                       double* __restrict__ U, const int* st) {
  extern __shared__ __align__(16) unsigned char smq[];
  if (status_bad(st)) return;
  const int TQ = tile_q(b), W = 2 * TQ * b;
  int J, K;
  tile_of_index(Q, TQ, blockIdx.x, J, K);
  const int J0 = J * TQ, K0 = K * TQ;
  const int c0 = blockIdx.y * TB_COLS;
  ll* Us = reinterpret_cast<ll*>(smq);                         // [row][TB_LD]
  int2* Vs = reinterpret_cast<int2*>(Us + (size_t)W * TB_LD);  // [c][b]: v of reflector c, its own rows
  int2* ts = Vs + b * b;                                       // [c]
  const int t = threadIdx.x;
  constexpr ll ONE = 1ll << 62;
  for (int idx = t; idx < W * TB_COLS; idx += blockDim.x) {
    int r = idx / TB_COLS, cc = idx % TB_COLS;
    Us[r * TB_LD + cc] = (r == c0 + cc) ? ONE : 0;
  }
  const int col = t >> 3, part = t & 7;
  const int jhi = min(J0 + TQ - 1, Q);
  // rows [rmin, rmax] hold every nonzero of this CTA's columns (identity columns at
  // first): a reflector whose rows miss that range leaves them unchanged and is skipped
  int rmin = c0, rmax = c0 + TB_COLS - 1;
  for (int j = jhi; j >= J0; --j) {
    for (int k = K0; k < K0 + TQ; ++k) {
      if (k > Q - j) continue;
      const int lo = (j + k - J0 - K0) * b;  // tile row of the diamond's row 0
      if (lo + 2 * b - 2 < rmin || lo > rmax) continue;
      const double* D0 = q2 + diamond_index(Q, j, k) * diamond_elems(b);
      __syncthreads();  // the previous diamond's reflectors are no longer read
      for (int idx = t; idx < b * b; idx += blockDim.x) {
        const int c = idx / b, i = idx - c * b;
        const double x = D0[(size_t)c * 2 * b + c + i];
        const ll m = x == 0.0 ? 0 : qint(fabs(x), 62);
        Vs[idx] = qsplit(x < 0.0 ? -m : m);
      }
      if (t < b) {
        const double x = D0[(size_t)2 * b * b + t];
        ts[t] = qsplit(x == 0.0 ? 0 : qint(x, 61));
      }
      __syncthreads();
      for (int c = b - 1; c >= 0; --c) {
        if (lo + c + b - 1 < rmin || lo + c > rmax) continue;
        const int2 tc = ts[c];
        if ((tc.x | tc.y) == 0) continue;
        rmin = min(rmin, lo + c);
        rmax = max(rmax, lo + c + b - 1);
        const int2* v = Vs + c * b;
        ll* u0 = Us + (lo + c) * TB_LD + col;
        ll hh = 0, mm = 0;
#pragma unroll 4
        for (int r = part; r < b; r += 8) {
          const int2 x = qsplit(u0[r * TB_LD]), y = v[r];
          hh += qhh(x, y);
          mm += qmid(x, y, 1ll << 29) >> 30;
        }
        ll d = (hh << 2) + mm;
        d += __shfl_xor_sync(0xffffffffu, d, 1);
        d += __shfl_xor_sync(0xffffffffu, d, 2);
        d += __shfl_xor_sync(0xffffffffu, d, 4);
        const int2 u = qsplit(qmul<62>(qsplit(d), tc));  // Q61
#pragma unroll 4
        for (int r = part; r < b; r += 8) u0[r * TB_LD] -= qmul<61>(u, v[r]);
        __syncwarp();
      }
    }
  }
  __syncthreads();
  double* Ut = U + (size_t)blockIdx.x * W * W;  // U - I, W x W column-major
  for (int idx = t; idx < W * TB_COLS; idx += blockDim.x) {
    int r = idx % W, cc = idx / W;
    if (c0 + cc >= W) continue;
    // (on the diagonal of a tile with reflections U may be -1 and a rounding: one less than -2^63 as an integer)
    const ll u = Us[r * TB_LD + cc];
    const bool dia = r == c0 + cc;
    Ut[r + (size_t)(c0 + cc) * W] = dia && u < 0 ? (double)u * 0x1p-62 - 1.0 : (double)(u - (dia ? ONE : 0)) * 0x1p-62;
  }
}

size_t q2_tile_smem_bytes(int b) {
  return (size_t)2 * tile_q(b) * b * TB_LD * sizeof(ll) + ((size_t)b * b + b) * sizeof(int2);
}

size_t q2_smem_bytes(int b) {
  return ((size_t)2 * b * b + (size_t)(2 * b - 1) * (Q2_COLS + 1) + b) * sizeof(double);
}
size_t bulge_smem_bytes() { return ((size_t)2 * BMAX * (BMAX + 1) + 4 * BMAX + 4 * BMAX + 16) * sizeof(double); }

}  // namespace

// CTAs whose partial sums the panel-QR buffers hold: the per-step kernel's ceil(M / 256),
// or up to 1024 CTAs of 64 rows for the single-launch form.
static size_t pqr_partial_ctas(int M) {
  size_t g256 = ((size_t)M + PQ_ROWS - 1) / PQ_ROWS, g64 = ((size_t)M + 63) / 64;
  if (g64 > 1024) g64 = 1024;
  return g256 > g64 ? g256 : g64;
}

size_t q2_elems(int M, int b) {
  if (M < 2 || b < 1) return 0;
  size_t Q = (size_t)(M - 2) / b;
  return (Q + 1) * (Q + 2) / 2 * diamond_elems(b);
}

size_t band_ws_elems(int M, int b) {
  size_t G = pqr_partial_ctas(M);
  // + the digit planes of the trailing matrix (shared by the C22 products of a panel group)
  size_t reduce = 2 * rr(G * BMAX) + 2 * rr(BMAX) + rr(32) + 4 * rr((size_t)M * b) +
                  2 * rr((size_t)M * 2 * BAND_GROUP * b) + 5 * rr((size_t)2 * b * b) +
                  rr((size_t)2 * BAND_GROUP * b * b) + rr(oz_sym_planes_bytes(M, 9) / sizeof(double) + 1) +
                  rr(oz_sym_part_elems(M, b));
  size_t chase = rr((size_t)2 * b * M) + rr((size_t)M) + rr(1);  // band, progress counters, norm bound
  return reduce > chase ? reduce : chase;
}

namespace {

struct BandWs {
  double *part0, *part1, *prow0, *prow1;
  long long gcap;  // CTAs the partial-sum buffers hold
  int *bar, *wide;
  double *V, *CV, *V1, *W1;
  double *WV, *VW;     // n x 2 G b: [W_0 V_0 W_1 V_1 ...] and [V_0 W_0 V_1 W_1 ...] of a panel group
  double *GV, *T, *Tt, *Pm, *Ym, *Zs;
  void* planes;        // digit planes of C22
  size_t planes_bytes;
  double* parts;       // partial products of C22 V
  size_t part_elems;
};

// QR of the n x b panel P (ld ldp): reflectors stay in P, tau[0..b), explicit V (n x b,
// unit lower trapezoidal) and the compact-WY factor T (b x b).
int panel_factor(gep_handle_t h, int n, int b, double* P, int ldp, double* tau, const BandWs& w, double* V,
                 int eng) {
  const int G = (n + PQ_ROWS - 1) / PQ_ROWS;
  const int nref = n < b ? n : b;
  double *pin = w.part0, *pout = w.part1, *rin = w.prow0, *rout = w.prow1;
  // one cooperative launch when every CTA of the panel can be resident at once
  static DeviceValue resident;
  int coop_per_sm = 0;
  GEP_CHECK(resident.get(current_device(), &coop_per_sm, [](int* v) -> int {
    const size_t smax = pqr_coop_smem_bytes(PQ_ROWS, BMAX);
    GEP_CUDA(cudaFuncSetAttribute(k_pqr_coop, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smax));
    GEP_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(v, k_pqr_coop, PQ_ROWS, smax));
    return GEP_OK;
  }));
  // fewest rows per CTA whose grid is resident at once and fits the partial-sum buffers
  // (a test may force 64, 128 or 256 rows, or the per-column kernel with -1)
  const long long cap = (long long)coop_per_sm * h->sm_count;
  int rp = 0;
  if (h->pqr_rows > 0) {
    const long long g = (n + h->pqr_rows - 1) / h->pqr_rows;
    if (g > cap || g > w.gcap) return GEP_ERR_UNSUPPORTED;
    rp = h->pqr_rows;
  } else if (h->pqr_rows == 0) {
    for (int c = 64; c <= PQ_ROWS; c *= 2) {
      long long g = (n + c - 1) / c;
      if (g <= cap && g <= w.gcap) { rp = c; break; }
    }
  }
  if (rp > 0) {
    const int Gc = (n + rp - 1) / rp;
    const size_t smem = pqr_coop_smem_bytes(rp, BMAX);
    GEP_CUDA(cudaMemsetAsync(w.bar, 0, sizeof(int), h->stream));
    int nn = n, nbb = b, rpp = rp, ld = ldp;
    int* bar = w.bar;
    int* st = h->d_status;
    void* args[] = {&nn, &nbb, &rpp, &P, &ld, &pin, &pout, &rin, &rout, &tau, &bar, &st};
    GEP_CUDA(cudaLaunchCooperativeKernel((void*)k_pqr_coop, dim3(Gc), dim3(PQ_ROWS), args, smem, h->stream));
    GEP_CHECK(check_launch(h));
  } else {
    k_pqr_step<<<G, PQ_ROWS, 0, h->stream>>>(n, b, -1, P, ldp, pin, rin, pout, rout, tau, h->d_status);
    GEP_CHECK(check_launch(h));
    for (int c = 0; c < nref; ++c) {
      double* tp = pin; pin = pout; pout = tp;
      tp = rin; rin = rout; rout = tp;
      k_pqr_step<<<G, PQ_ROWS, 0, h->stream>>>(n, b, c, P, ldp, pin, rin, pout, rout, tau, h->d_status);
      GEP_CHECK(check_launch(h));
    }
  }
  k_panel_v<<<dim3((n + 255) / 256, b), 256, 0, h->stream>>>(n, b, P, ldp, V, h->d_status);
  GEP_CHECK(check_launch(h));
  GEP_CHECK(dgemm(h, 'T', 'N', 'F', b, b, n, 1.0, V, n, V, n, 0.0, w.GV, b, eng));
  return larft_rec(h, b, w.GV, b, tau, w.T, b, w.Tt, GEP_PREC_FP64);
}

// k_panel_qr's launch (b <= 32): V_j into Va and Vb (ld ldv, r0 zero rows first), T into w.T.
// Returns GEP_ERR_UNSUPPORTED when the grid cannot be resident or its partial sums do not fit.
template <int RPW>
int panel_qr_launch(gep_handle_t h, const PanelArgs& a, long long part_elems) {
  const int G = (a.n + PQW * RPW - 1) / (PQW * RPW);
  static DeviceValue resident;
  int per_sm = 0;
  GEP_CHECK(resident.get(current_device(), &per_sm, [](int* v) -> int {
    GEP_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(v, k_panel_qr<RPW>, 32 * (PQW + 1), 0));
    return GEP_OK;
  }));
  if ((long long)G > (long long)per_sm * h->sm_count || 2LL * G * PQN > part_elems) return GEP_ERR_UNSUPPORTED;
  GEP_CUDA(cudaMemsetAsync(a.bar, 0, sizeof(int), h->stream));
  PanelArgs aa = a;
  void* args[] = {&aa};
  GEP_CUDA(cudaLaunchCooperativeKernel((void*)k_panel_qr<RPW>, dim3(G), dim3(32 * (PQW + 1)), args, 0, h->stream));
  return check_launch(h);
}

int panel_qr(gep_handle_t h, int n, int b, double* P, int ldp, double* tau, const BandWs& w, double* Va, double* Vb,
             int r0, int ldv) {
  if (!h->no_clusters && panel_qr_cluster_takes(n, b)) {
    const int rc = panel_qr_cluster(h, n, b, P, ldp, tau, Va, Vb, r0, ldv, w.T, w.wide);
    if (rc != GEP_ERR_UNSUPPORTED) return rc;
  }
  PanelArgs a;
  a.n = n; a.nb = b; a.ldp = ldp; a.r0 = r0; a.ldv = ldv;
  a.P = P; a.tau = tau; a.part = w.part0; a.prow = w.prow0; a.Va = Va; a.Vb = Vb; a.T = w.T;
  a.bar = w.bar; a.st = h->d_status;
  const long long cap = 2 * w.gcap * BMAX;  // part0 and part1 together
  const int rows = n <= 127 * 32 ? 4 : n <= 127 * 128 ? 8 : 16;
  if (rows == 4) return panel_qr_launch<4>(h, a, cap);
  if (rows == 8) return panel_qr_launch<8>(h, a, cap);
  return panel_qr_launch<16>(h, a, cap);
}

// W = X - V (T^T V^T X) / 2 with X = CV T (CV = C22 V, n x b): the two-sided update of
// the trailing matrix is then C22 - W V^T - V W^T.
int panel_w(gep_handle_t h, int n, int b, const double* V, const double* CV, double* W, const BandWs& w, int eng) {
  GEP_CHECK(dgemm(h, 'N', 'N', 'F', n, b, b, 1.0, CV, n, w.T, b, 0.0, W, n, eng));    // X = C22 V T
  GEP_CHECK(dgemm(h, 'T', 'N', 'F', b, b, n, 1.0, V, n, W, n, 0.0, w.Pm, b, eng));    // V^T X
  GEP_CHECK(dgemm(h, 'T', 'N', 'F', b, b, b, 1.0, w.T, b, w.Pm, b, 0.0, w.Ym, b, eng));  // T^T V^T X
  return dgemm(h, 'N', 'N', 'F', n, b, b, -0.5, V, n, w.Ym, b, 1.0, W, n, eng);
}

}  // namespace

// S1b.  C (M x M, lower triangle) -> band of width b in C (lower), reflectors below the
// band, tau1[j] for columns j < M - b (zero where no reflector).  The upper triangle is
// not referenced.  Panels are taken in groups of up to BAND_GROUP: panel j of a group first
// receives the pending updates of panels 0..j-1 on its columns and diagonal block, its
// C^(j) V_j is formed from the group's not yet updated trailing matrix minus the low-rank
// corrections sum_i W_i (V_i^T V_j) + V_i (W_i^T V_j), and all the group's updates are
// applied together as one product of depth 2 G b (512 for G = 4, b = 64: one full exact
// chunk of the product kernel, and one digit split of the trailing matrix per group).
int band_reduce(gep_handle_t h, int M, double* C, int ldc, int b, double* tau1, double* ws, size_t ws_elems,
                int eng) {
  if (b < 1 || b > BMAX) return GEP_ERR_UNSUPPORTED;
  if (ws_elems < band_ws_elems(M, b)) return GEP_ERR_ALLOC;
  if (M <= 0) return GEP_OK;
  GEP_CHECK(set_matrix(h, M, 1, 0.0, 0.0, tau1, M));
  if (M <= b + 1) return GEP_OK;
  size_t Gmax = pqr_partial_ctas(M);
  BandWs w;
  w.gcap = (long long)Gmax;
  double* q = ws;
  auto take = [&](size_t n) { double* p = q; q += rr(n); return p; };
  w.part0 = take(Gmax * BMAX);
  w.part1 = take(Gmax * BMAX);
  w.prow0 = take(BMAX);
  w.prow1 = take(BMAX);
  w.bar = reinterpret_cast<int*>(take(32));
  w.wide = w.bar + 32;
  w.V = take((size_t)M * b);
  w.CV = take((size_t)M * b);
  w.V1 = take((size_t)M * b);
  w.W1 = take((size_t)M * b);
  w.WV = take((size_t)M * 2 * BAND_GROUP * b);
  w.VW = take((size_t)M * 2 * BAND_GROUP * b);
  w.GV = take((size_t)2 * b * b);
  w.T = take((size_t)2 * b * b);
  w.Tt = take((size_t)2 * b * b);
  w.Pm = take((size_t)2 * b * b);
  w.Ym = take((size_t)2 * b * b);
  w.Zs = take((size_t)2 * BAND_GROUP * b * b);
  w.planes_bytes = oz_sym_planes_bytes(M, 9);
  w.planes = take(w.planes_bytes / sizeof(double) + 1);
  w.part_elems = oz_sym_part_elems(M, b);
  w.parts = take(w.part_elems);
  const int levels = eng == GEP_PREC_MIXED_REFINED ? 4 : 9;
  if (b <= PQN) {  // the arithmetic of the panels in a cluster (the sums in V, not yet in use)
    unsigned long long* sum = reinterpret_cast<unsigned long long*>(w.V);
    int* ex = w.wide + 1;
    GEP_CUDA(cudaMemsetAsync(sum, 0, sizeof(unsigned long long) * (size_t)M, h->stream));
    GEP_CUDA(cudaMemsetAsync(w.wide, 0, 2 * sizeof(int), h->stream));
    const int nt = (M + 63) / 64;
    GEP_CHECK(max_exponent(h, M, C, ldc, ex));
    k_row_sums<<<dim3(nt, nt), 256, 0, h->stream>>>(M, C, ldc, ex, sum, h->d_status);
    GEP_CHECK(check_launch(h));
    k_row_spread<<<1, 1024, 0, h->stream>>>(M, sum, ex, w.wide, h->d_status);
    GEP_CHECK(check_launch(h));
  }
  for (int pb = 0; M - pb - b >= 2;) {
    const int n = M - pb - b;
    // panels of this group: panel j (j >= 1) owns columns [(j-1) b, j b) of C22 and its
    // reflectors act on rows [j b, n), which needs n - j b >= 2
    // (groups pay where the trailing matrix is large; below that pairs, whose two C22 products
    // need no cross-panel corrections beyond one pair of small products)
    const int gmin = h->band_group_min >= 0 ? h->band_group_min : (b <= 32 ? BAND_GROUP_MIN_N / 2 : BAND_GROUP_MIN_N);
    const int g = std::min(n >= gmin ? BAND_GROUP : 2, (n - 2) / b + 1);
    double* P = C + (pb + b) + (size_t)pb * ldc;
    double* C22 = C + (pb + b) + (size_t)(pb + b) * ldc;
    // V_j and W_j are kept at full height n (zero above row j b) in WV / VW, so that the
    // pending update of panel i on any block of C22 is the same slice of one product.
    auto wv = [&](int blk) { return w.WV + (size_t)blk * b * n; };
    auto vw = [&](int blk) { return w.VW + (size_t)blk * b * n; };
    // C22 is split into digit planes once for the group on the tensor-core engines: every
    // C^(j) V_j below reads rows j b.. of the planes against the full-height V_j.  The columns
    // the group updates in between (those of panels 1..g-1) meet V_j's zero rows.
    OzSymPlanes planes;
    const bool use_planes = eng != GEP_PREC_FP64 && n >= 128 && b >= 32;
    if (use_planes) GEP_CHECK(oz_split_sym(h, n, C22, ldc, levels, w.planes, w.planes_bytes, &planes));
    for (int j = 0; j < g; ++j) {
      const int r0 = j * b, nr = n - r0;  // panel j's reflectors act on rows [r0, n) of C22
      double* Vj;
      int ldv = nr;
      double* Pj = P;
      if (j > 0) {
        // panel j = C22 columns [(j-1) b, j b), rows [(j-1) b, n): the pending updates of
        // panels 0..j-1 first (its diagonal block on the lower triangle only), then its QR
        const int c0 = r0 - b;
        double* Dj = C22 + c0 + (size_t)c0 * ldc;
        GEP_CHECK(dgemm(h, 'N', 'T', 'L', b, b, 2 * j * b, -1.0, w.WV + c0, n, w.VW + c0, n, 1.0, Dj, ldc, eng));
        GEP_CHECK(dgemm(h, 'N', 'T', 'F', nr, b, 2 * j * b, -1.0, w.WV + r0, n, w.VW + c0, n, 1.0, Dj + b, ldc,
                        eng));
        Pj = Dj + b;
      }
      int rc = GEP_ERR_UNSUPPORTED;
      if (b <= PQN && h->pqr_rows == 0) rc = panel_qr(h, nr, b, Pj, ldc, tau1 + pb + r0, w, wv(2 * j + 1), vw(2 * j), r0, n);
      const bool narrow = rc != GEP_ERR_UNSUPPORTED;  // V_j is in the group buffers
      if (narrow) {
        GEP_CHECK(rc);
        Vj = vw(2 * j) + r0;
        ldv = n;
      } else if (j == 0) {
        GEP_CHECK(panel_factor(h, n, b, P, ldc, tau1 + pb, w, w.V, eng));
        Vj = w.V;
      } else {
        GEP_CHECK(panel_factor(h, nr, b, Pj, ldc, tau1 + pb + r0, w, w.V1, eng));
        Vj = w.V1;
      }
      // V_j at full height into both group buffers (zero rows above r0)
      if (!narrow && r0 > 0) {
        GEP_CHECK(set_matrix(h, r0, b, 0.0, 0.0, wv(2 * j + 1), n));
        GEP_CHECK(set_matrix(h, r0, b, 0.0, 0.0, vw(2 * j), n));
        GEP_CHECK(set_matrix(h, r0, b, 0.0, 0.0, wv(2 * j), n));
        GEP_CHECK(set_matrix(h, r0, b, 0.0, 0.0, vw(2 * j + 1), n));
      }
      if (!narrow) {
        GEP_CHECK(copy_matrix(h, nr, b, Vj, nr, wv(2 * j + 1) + r0, n));
        GEP_CHECK(copy_matrix(h, nr, b, Vj, nr, vw(2 * j) + r0, n));
      }
      // C^(j) V_j = C22(r0:, r0:) V_j - sum_{i<j} (W_i V_i^T + V_i W_i^T)(r0:, r0:) V_j
      if (use_planes && nr >= 128) {
        GEP_CHECK(dgemm_oz_sym_planes(h, planes, r0, b, 1.0, vw(2 * j), n, 0.0, w.CV, nr, w.parts, w.part_elems));
      } else {
        GEP_CHECK(dgemm(h, 'S', 'N', 'F', nr, b, nr, 1.0, C22 + r0 + (size_t)r0 * ldc, ldc, Vj, ldv, 0.0, w.CV, nr,
                        eng));
      }
      if (j > 0) {
        // Zs = [V_0 W_0 .. V_{j-1} W_{j-1}](r0:)^T V_j, CV -= [W_0 V_0 ..](r0:) Zs
        GEP_CHECK(dgemm(h, 'T', 'N', 'F', 2 * j * b, b, nr, 1.0, w.VW + r0, n, Vj, ldv, 0.0, w.Zs, 2 * j * b, eng));
        GEP_CHECK(dgemm(h, 'N', 'N', 'F', nr, b, 2 * j * b, -1.0, w.WV + r0, n, w.Zs, 2 * j * b, 1.0, w.CV, nr,
                        eng));
      }
      if (narrow) {
        GEP_CHECK(dgemm_f64(h, 'T', 'N', 'F', b, b, nr, 1.0, Vj, ldv, w.CV, nr, 0.0, w.Pm, b));  // V^T C22 V
        const auto kernel = nr <= 8 * h->sm_count ? k_panel_w<1> : nr <= 16 * h->sm_count ? k_panel_w<2> : k_panel_w<4>;
        const int rows = nr <= 8 * h->sm_count ? 8 : nr <= 16 * h->sm_count ? 16 : 32;
        kernel<<<std::min((nr + rows - 1) / rows, 2 * h->sm_count), 256, 0, h->stream>>>(
            nr, b, Vj, ldv, w.CV, w.T, w.Pm, wv(2 * j), vw(2 * j + 1), r0, h->d_status);
        GEP_CHECK(check_launch(h));
        continue;
      }
      GEP_CHECK(panel_w(h, nr, b, Vj, w.CV, w.W1, w, eng));
      GEP_CHECK(copy_matrix(h, nr, b, w.W1, nr, wv(2 * j) + r0, n));
      GEP_CHECK(copy_matrix(h, nr, b, w.W1, nr, vw(2 * j + 1) + r0, n));
    }
    // trailing matrix after the group: C22(t0:, t0:) -= [W_0 V_0 ..][V_0 W_0 ..]^T (lower
    // triangle, depth 2 g b), t0 = (g-1) b
    const int t0 = (g - 1) * b, nt = n - t0;
    GEP_CHECK(dgemm(h, 'N', 'T', 'L', nt, nt, 2 * g * b, -1.0, w.WV + t0, n, w.VW + t0, n, 1.0,
                    C22 + t0 + (size_t)t0 * ldc, ldc, eng));
    pb += g * b;
  }
  return GEP_OK;
}

// S1c.  Band of width b in the lower triangle of C -> d, e; reflectors into q2 (may be null).
int band_to_tridiag(gep_handle_t h, int M, const double* C, int ldc, int b, double* d, double* e, double* q2,
                    double* ws, size_t ws_elems) {
  if (b < 1 || b > BMAX) return GEP_ERR_UNSUPPORTED;
  if (ws_elems < band_ws_elems(M, b)) return GEP_ERR_ALLOC;
  if (M <= 0) return GEP_OK;
  const int ldab = 2 * b;
  double* AB = ws;
  int* prog = reinterpret_cast<int*>(ws + rr((size_t)2 * b * M));
  k_band_copy<<<M, ldab, 0, h->stream>>>(M, b, C, ldc, AB, ldab, h->d_status);
  GEP_CHECK(check_launch(h));
  if (M >= 2) {
    GEP_CUDA(cudaMemsetAsync(prog, 0, sizeof(int) * 2 * (size_t)M, h->stream));
    const int Q = (M - 2) / b;
    if (q2) GEP_CUDA(cudaMemsetAsync(q2, 0, q2_elems(M, b) * sizeof(double), h->stream));
    // b = 32 and 64 take the fixed-point kernel unless the rows differ in scale (known on the device only: both
    // kernels are launched and one returns at once, about 5 us), other widths the general one
    const bool fixed = b == 32 || b == 64;
    unsigned long long* mx = reinterpret_cast<unsigned long long*>(prog + rr((size_t)M) * 2);
    static DeviceOnce attributes;
    GEP_CHECK(once_per_device(attributes, []() -> int {
      GEP_CUDA(cudaFuncSetAttribute(k_bulge, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bulge_smem_bytes()));
      GEP_CUDA(cudaFuncSetAttribute(k_bulge_ws<32>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(BulgeShared<32>)));
      GEP_CUDA(cudaFuncSetAttribute(k_bulge_ws<64>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(BulgeShared<64>)));
      return GEP_OK;
    }));
    BulgeArgs a;
    a.M = M; a.b = b; a.ldab = ldab; a.Q = Q; a.AB = AB; a.prog = prog; a.q2 = q2; a.st = h->d_status;
    a.mx = fixed ? mx : nullptr;
    a.wait_ns = h->wait_limit_ns;
    a.drop_sweep = h->fault_drop_sweep;
    if (fixed) {
      GEP_CUDA(cudaMemsetAsync(mx, 0, 3 * sizeof(unsigned long long), h->stream));
      k_band_rowsum<<<(M + 255) / 256, 256, 0, h->stream>>>(M, b, AB, ldab, mx, h->d_status);
      GEP_CHECK(check_launch(h));
      k_band_fix<<<std::min(M, 4 * h->sm_count), 256, 0, h->stream>>>(M, AB, ldab, mx, h->d_status);
      GEP_CHECK(check_launch(h));
    }
    auto chase = [&](const void* kern, int threads, size_t smem) -> int {
      int per_sm = 0;
      GEP_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, threads, smem));
      if (per_sm < 1) return GEP_ERR_UNSUPPORTED;
      // The sweeps form a dependency chain (step k of sweep s waits for step k+1 of sweep
      // s-1): the time is set by the latency of one step, which co-resident CTAs stretch.
      if (per_sm > BULGE_CTAS_PER_SM) per_sm = BULGE_CTAS_PER_SM;
      // Sweep s starts two steps after sweep s-1 and lasts about (M - 2) / b + 1 steps, so
      // about half that many sweeps are in flight at once: CTAs beyond that would only wait,
      // holding SMs that concurrent solves on other streams could use.
      const int grid = std::min({per_sm * h->sm_count, ((M - 2) / b + 1) / 2 + 2, M - 1});
      void* args[] = {&a};
      GEP_CUDA(cudaLaunchCooperativeKernel(kern, dim3(grid), dim3(threads), args, smem, h->stream));
      return check_launch(h);
    };
    if (b == 32) GEP_CHECK(chase((const void*)k_bulge_ws<32>, bulge_threads<32>(), sizeof(BulgeShared<32>)));
    if (b == 64) GEP_CHECK(chase((const void*)k_bulge_ws<64>, bulge_threads<64>(), sizeof(BulgeShared<64>)));
    GEP_CHECK(chase((const void*)k_bulge, 256, bulge_smem_bytes()));
    if (fixed) {
      k_band_diag_fix<<<(M + 255) / 256, 256, 0, h->stream>>>(M, AB, ldab, mx, d, e, h->d_status);
      return check_launch(h);
    }
  }
  k_band_diag<<<(M + 255) / 256, 256, 0, h->stream>>>(M, AB, ldab, d, e, h->d_status);
  return check_launch(h);
}

size_t q2_tile_ws_elems(int M, int b) {
  if (M < 3 || b < 1) return 0;
  return rr((size_t)2 * tile_q(b) * b * (size_t)M);
}

namespace {

// Tiles of every tile row J, one after the other (tile (J, K) at all_tiles_offset(Q, J) + K).
size_t all_tiles_offset(int Q, int J, int TQ) {
  size_t off = 0;
  for (int j = 0; j < J; ++j) off += (size_t)((Q - j * TQ) / TQ + 1);
  return off;
}

int set_tile_build_attr() {
  static DeviceOnce attributes;
  return once_per_device(attributes, []() -> int {
    GEP_CUDA(cudaFuncSetAttribute(k_q2_tile_build, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)q2_tile_smem_bytes(BMAX)));
    return GEP_OK;
  });
}

}  // namespace

size_t q2_all_tiles_elems(int M, int b) {
  if (M < 3 || b < 1) return 0;
  const int Q = (M - 2) / b, TQ = tile_q(b);
  const size_t W = (size_t)2 * TQ * b;
  return all_tiles_offset(Q, Q / TQ + 1, TQ) * W * W;
}

// Builds every dense tile U(J, K) - I of Q2 into U (q2_all_tiles_elems doubles) on `stream`,
// for apply_q2 to use later; it only reads q2, so it may run on a second stream while the
// tridiagonal eigensolver runs on the first.
int build_q2_tiles(gep_handle_t h, cudaStream_t stream, int M, int b, const double* q2, double* U) {
  if (b < 1 || b > BMAX) return GEP_ERR_UNSUPPORTED;
  if (M < 3) return GEP_OK;
  GEP_CHECK(set_tile_build_attr());
  const int Q = (M - 2) / b;
  const int TQ = tile_q(b), W = 2 * TQ * b;
  const size_t tiles = all_tiles_offset(Q, Q / TQ + 1, TQ);
  k_q2_tile_build<<<dim3((unsigned)tiles, (W + TB_COLS - 1) / TB_COLS), 256, q2_tile_smem_bytes(b), stream>>>(
      b, Q, q2, U, h->d_status);
  return check_launch(h);
}

// Where U(J, K) - I can be nonzero, per 128-row block of a W x W tile: the reflectors of the
// tile's diamonds, taken in the order k_q2_tile_build applies them, spread each column's
// nonzero rows over an interval (a reflector whose rows miss the interval leaves the
// column alone, one that meets it widens it to the union).  Row block r then needs only
// the columns whose interval meets its rows.  Every tile has this structure or a subset
// of it (tiles at the edge hold fewer diamonds).
static void q2_tile_kranges(int b, OzKRange* kr) {
  const int TQ = tile_q(b), W = 2 * TQ * b;
  std::vector<int> rmin(W), rmax(W);
  for (int c = 0; c < W; ++c) rmin[c] = rmax[c] = c;
  for (int jj = TQ - 1; jj >= 0; --jj)
    for (int kk = 0; kk < TQ; ++kk)
      for (int c = b - 1; c >= 0; --c) {
        const int r0 = (jj + kk) * b + c, r1 = r0 + b - 1;
        for (int x = 0; x < W; ++x)
          if (r0 <= rmax[x] && r1 >= rmin[x]) {
            rmin[x] = std::min(rmin[x], r0);
            rmax[x] = std::max(rmax[x], r1);
          }
      }
  kr->n = std::min((W + 127) / 128, OZ_KR_MAX);
  for (int r = 0; r < kr->n; ++r) {
    const int a = 128 * r, e = std::min(W, a + 128) - 1;
    int lo = W, hi = 0;
    for (int x = 0; x < W; ++x)
      if (rmin[x] <= e && rmax[x] >= a) {
        lo = std::min(lo, x);
        hi = std::max(hi, x + 1);
      }
    kr->lo[r] = lo < hi ? lo : 0;
    kr->hi[r] = lo < hi ? hi : 0;
  }
}

namespace {

// ---- larger Q2 tiles
//
// Four tiles (2J + a, 2K + b) of order w make one of order 2 w (the same staircase with twice the
// step): U = T01 T00 T11 T10, T_ab at rows (a + b) w / 2.  With U = I + V and the overlaps of w / 2 rows,
//   VA = V10 + V11 + V11(:, :w/2) V10(w/2:, :),  VB = V00 + V01 + V01(:, :w/2) V00(w/2:, :),
//   V = VA + VB + VB(:, w/2:3w/2) VA(w/2:3w/2, :).
// A tile twice as large costs the same flops a row of Z but half the passes over it (digits or residues
// of Z, C in and out), and from order 1024 on the products go through residues.  Order 8192: S3 102 -> 75 ms.

// VA and VB of tiles z: their placed parts (tiles of a row follow each other; nA, nB of them).
__global__ void __launch_bounds__(256) k_q2_place(int w, const double* __restrict__ rowA, int nA,
                                                  const double* __restrict__ rowB, int nB, double* __restrict__ VA,
                                                  double* __restrict__ VB, const int* st) {
  if (status_bad(st)) return;
  const int z = blockIdx.z, c = blockIdx.y, r = blockIdx.x * 256 + threadIdx.x, h = w / 2;
  if (r >= 2 * w) return;
  const size_t ww = (size_t)w * w, o = (size_t)z * 4 * ww + r + (size_t)c * 2 * w;
  auto el = [&](const double* row, int n, int t, int off) {
    const int i = r - off, j = c - off;
    return t < n && i >= 0 && i < w && j >= 0 && j < w ? row[t * ww + i + (size_t)j * w] : 0.0;
  };
  VA[o] = el(rowB, nB, 2 * z, h) + el(rowB, nB, 2 * z + 1, w);
  VB[o] = el(rowA, nA, 2 * z, 0) + el(rowA, nA, 2 * z + 1, h);
}

__global__ void __launch_bounds__(256) k_q2_sum(size_t n, const double* __restrict__ VA, const double* __restrict__ VB,
                                                double* __restrict__ V, const int* st) {
  if (status_bad(st)) return;
  for (size_t i = blockIdx.x * (size_t)256 + threadIdx.x; i < n; i += (size_t)gridDim.x * 256) V[i] = VA[i] + VB[i];
}

// dst: the (nA + 1) / 2 tiles of order 2 w that the tiles of rows 2J (rowA) and 2J + 1 (rowB) make.
int merge_q2_tiles(gep_handle_t h, int w, const double* rowA, int nA, const double* rowB, int nB, double* VA,
                   double* VB, double* dst) {
  const int count = (nA + 1) / 2, hw = w / 2, ld = 2 * w;
  const long long ww = (long long)w * w;
  k_q2_place<<<dim3((2 * w + 255) / 256, 2 * w, count), 256, 0, h->stream>>>(w, rowA, nA, rowB, nB, VA, VB, h->d_status);
  GEP_CHECK(check_launch(h));
  if (nB >= 2)
    GEP_CHECK(dgemm_oz_batched(h, w, w, hw, rowB + ww, w, 2 * ww, rowB + hw, w, 2 * ww, VA + w + (size_t)hw * ld, ld,
                               4 * ww, nB / 2));
  if (nA >= 2)
    GEP_CHECK(dgemm_oz_batched(h, w, w, hw, rowA + ww, w, 2 * ww, rowA + hw, w, 2 * ww, VB + hw, ld, 4 * ww, nA / 2));
  k_q2_sum<<<8 * h->sm_count, 256, 0, h->stream>>>((size_t)count * 4 * ww, VA, VB, dst, h->d_status);
  GEP_CHECK(check_launch(h));
  if (nB >= 1)
    GEP_CHECK(dgemm_oz_batched(h, 3 * hw, 3 * hw, w, VB + (size_t)hw * ld, ld, 4 * ww, VA + hw + (size_t)hw * ld, ld,
                               4 * ww, dst + (size_t)hw * ld, ld, 4 * ww, (nB + 1) / 2));
  return GEP_OK;
}

// Tiles of level L (order W 2^L) out of the tiles of level 0.
struct Q2Levels {
  gep_handle_t h;
  int Q, TQ, W;
  const double* U;
  int nJ(int L) const { return ((Q / TQ + 1) + (1 << L) - 1) >> L; }
  int nK(int L, int J) const {
    if (L == 0) return J * TQ <= Q ? (Q - J * TQ) / TQ + 1 : 0;
    return (nK(L - 1, 2 * J) + 1) / 2;
  }
  size_t tile(int L) const { return (size_t)W * W << (2 * L); }
  // doubles that tiles(L, ..., cnt) takes from its buffer
  size_t need(int L, int cnt) const { return L == 0 ? 0 : 3 * cnt * tile(L) + 2 * need(L - 1, 2 * cnt); }
  // *out: tiles K0 .. K0 + cnt - 1 of row J (those that exist, following each other); buf: need(L, cnt)
  int tiles(int L, int J, int K0, int cnt, double* buf, const double** out, int* have) const {
    *have = std::max(0, std::min(cnt, nK(L, J) - K0));
    if (L == 0) {
      *out = U + (all_tiles_offset(Q, J, TQ) + K0) * tile(0);
      return GEP_OK;
    }
    double* dst = buf;
    double* VA = dst + cnt * tile(L);
    double* VB = VA + cnt * tile(L);
    double* bA = VB + cnt * tile(L);
    double* bB = bA + need(L - 1, 2 * cnt);
    const double *rA = nullptr, *rB = nullptr;
    int nA = 0, nB = 0;
    GEP_CHECK(tiles(L - 1, 2 * J, 2 * K0, 2 * cnt, bA, &rA, &nA));
    if (nK(L - 1, 2 * J + 1) > 2 * K0) GEP_CHECK(tiles(L - 1, 2 * J + 1, 2 * K0, 2 * cnt, bB, &rB, &nB));
    *out = dst;
    return nA > 0 ? merge_q2_tiles(h, W << (L - 1), rA, nA, rB, nB, VA, VB, dst) : GEP_OK;
  }
};

}  // namespace

// Z (M x ncol) <- Q2 Z.  engine FP64: diamonds applied directly on the FP64 cores.
// Otherwise the diamonds are merged into dense W x W tiles U(J, R) and every tile is
// applied as one product Z(rows) <- U Z(rows) on the engine (ws: q2_tile_ws_elems); U_all: the
// tiles, built by build_q2_tiles (on the caller's stream order).
int apply_q2(gep_handle_t h, int M, int b, const double* q2, double* Z, int ldz, int ncol, int engine, double* ws,
             size_t ws_elems, const double* U_all) {
  if (b < 1 || b > BMAX) return GEP_ERR_UNSUPPORTED;
  if (M < 3 || ncol <= 0) return GEP_OK;  // M = 2: the only reflector is the identity
  const int Q = (M - 2) / b;
  if (engine != GEP_PREC_FP64) {
    if (!U_all || ws_elems < q2_tile_ws_elems(M, b)) return GEP_ERR_ALLOC;
    const int TQ = tile_q(b), W = 2 * TQ * b;
    // Levels of merging, where the tiles suit the batched products and the scratch holds them (narrow Z does
    // not pay for the merging).  S3 with 0 / 1 / 2 levels: order 2047 3.82 / 3.86 / 3.86 ms, 3000 9.5 / 8.2 / 8.2,
    // 4000 16.8 / 14.5 / 16.7, 6000 46.5 / 39.2 / 38.8, 8192 102 / 81 / 75, 16384 (b = 64) 651 / 531 / 451; a third
    // level gains nothing (467 at 16384).
    Q2Levels lv{h, Q, TQ, W, U_all};
    int L = engine == GEP_PREC_FP64_EMULATED && W % 256 == 0 && ncol >= 2048 ? (M >= 6000 ? 2 : M >= 2560 ? 1 : 0) : 0;
    // (beside the tiles: a copy of up to 256 rows of Z, and one K panel of digits for products in place)
    const size_t rest = (size_t)256 * ncol;
    auto fits = [&](int l, int c) {
      const size_t w = (size_t)W << l;
      return w <= 2048 && lv.need(l, c) + rest <= ws_elems && 16 * (w + ncol) * w + 4 * (w + ncol) + 4096 <= h->eng_bytes;
    };
    while (L > 0 && !fits(L, 1)) --L;
    int chunk = 1;
    while (L > 0 && chunk < 8 && fits(L, 2 * chunk)) chunk *= 2;
    const int WL = W << L;
    double* Tmp = ws;
    OzKRange kr;
    q2_tile_kranges(b, &kr);
    for (int J = lv.nJ(L) - 1; J >= 0; --J) {
      const int nK = lv.nK(L, J);  // tiles (J, K) with a diamond
      const double* row = nullptr;
      int first = 0, have = 0;
      for (int K = 0; K < nK; ++K) {
        const int r0 = 1 + (J + K) * (WL / 2);
        if (r0 >= M) break;
        if (K >= first + have) {
          first = K;
          GEP_CHECK(lv.tiles(L, J, K, L ? chunk : nK, ws, &row, &have));
        }
        const int Wc = (M - r0) < WL ? (M - r0) : WL;
        const double* Ut = row + (size_t)(K - first) * WL * WL;
        // one K panel of the split-BF16 engine: all of Z(rows) is split into digit planes
        // before its product kernel writes C, so the update may run in place
        const size_t one_panel = (size_t)16 * (Wc + ncol) * ((Wc + 31) / 32 * 32) + (size_t)4 * (Wc + ncol) + 4096;
        if (product_on_tensor_cores(h, 'F', Wc, ncol, Wc, engine) && Wc <= 4096 && one_panel <= h->eng_bytes) {
          GEP_CHECK(dgemm(h, 'N', 'N', 'F', Wc, ncol, Wc, 1.0, Ut, WL, Z + r0, ldz, 1.0, Z + r0, ldz, engine,
                          L ? nullptr : &kr));
        } else {  // Z(rows) += (U - I) copy(Z(rows))
          double* T = L ? ws + lv.need(L, chunk) : Tmp;
          if (L && lv.need(L, chunk) + (size_t)Wc * ncol > ws_elems) return GEP_ERR_ALLOC;
          GEP_CHECK(copy_matrix(h, Wc, ncol, Z + r0, ldz, T, Wc));
          GEP_CHECK(dgemm(h, 'N', 'N', 'F', Wc, ncol, Wc, 1.0, Ut, WL, T, Wc, 1.0, Z + r0, ldz, engine, L ? nullptr : &kr));
        }
      }
    }
    return GEP_OK;
  }
  size_t smem = q2_smem_bytes(b);
  static DeviceOnce attributes;
  GEP_CHECK(once_per_device(attributes, []() -> int {
    GEP_CUDA(cudaFuncSetAttribute(k_q2_apply, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)q2_smem_bytes(BMAX)));
    return GEP_OK;
  }));
  const int slabs = (ncol + Q2_COLS - 1) / Q2_COLS;
  for (int wt = 0; wt <= 2 * Q; ++wt) {
    int kmin = wt - Q > 0 ? wt - Q : 0, kmax = wt / 2;
    if (kmax < kmin) continue;
    k_q2_apply<<<dim3(kmax - kmin + 1, slabs), 256, smem, h->stream>>>(M, b, Q, wt, q2, Z, ldz, ncol,
                                                                      h->d_status);
    GEP_CHECK(check_launch(h));
  }
  return GEP_OK;
}

}  // namespace gep
