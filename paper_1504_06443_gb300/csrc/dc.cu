// SEP solver, stage "D&C" (Table 3): eigenvalues and eigenvectors of the
// symmetric tridiagonal T = tridiag(e, d, e) by divide and conquer.
//
// T is torn at every multiple of LEAF (Cuppen): at split point p the coupling
// beta = e[p-1] is removed from the diagonal on both sides, leaving independent
// leaves solved one warp each (implicit QL with Wilkinson shift in shared
// memory).  Leaves are merged bottom-up, level by level; every kernel of a level
// works on all its merges at once (grid dimension y or x), since a merge alone is
// far too small for the GPU: the merges of a level used to run one after the other,
// about 12 launches each (order 2047: D&C 29.5 -> 5.7 ms, order 64: 2.57 -> 0.48 ms).  Merging two solved
// halves is the rank-one problem D + rho z z^T (z = last row of Q1 and first row
// of Q2 scaled by sign(beta)/sqrt(2), rho = 2|beta|), handled as:
//   1. deflation of negligible z_i and of nearly equal d_i (Givens rotation),
//   2. one root per non-deflated pole of the secular equation
//        f(lambda) = 1 + rho sum_i z_i^2 / (d_i - lambda) = 0,
//      found by a bracketed iteration on a two-pole rational model, with the root
//      stored as (nearest pole, offset) so every d_i - lambda_j is accurate,
//   3. z recomputed from the roots (Loewner formula, Gu & Eisenstat) so the
//      eigenvectors u_j ~ z_i / (d_i - lambda_j) are numerically orthogonal,
//   4. the merged eigenvectors Q [u_j] as one product per child on the GEMM engine
//      (the deflation rotations are folded into the rows of [u_j], so Q stays
//      block diagonal); the products of narrow merges run in one FP64 launch per level.
// Eigenvalues of every block are kept sorted ascending.
#include <math.h>

#include "gep_internal.cuh"

namespace gep {
namespace {

constexpr int LEAF = 8;
constexpr int FP64_WIDTH = 256;  // merges up to this order form their products in FP64, one launch a level
constexpr double EPS = 0x1p-53;

// Arrays of M entries: a merge of rows [lo, hi) uses [lo, hi) of each.
struct DcWs {
  double *Qt, *U, *D, *dd, *zs, *dv, *ndd, *ndz, *dfv, *rc, *rs, *tauR, *lam, *zhat, *rho;
  double *ptau, *pc, *ps;  // the Givens deflation test of each adjacent pair, from the undeflated values
  int *perm, *ndx, *dfx, *ra, *rb, *org, *posr, *posd, *cnt;
  int *nsl, *prot;         // positions (in perm) with z not negligible; pair test outcome
  // the view of merge m (rows [lo, ...)): per-merge scalars are rho[m], cnt[8 m ..]
  __device__ DcWs at(int lo, int m) const {
    DcWs v = *this;
    v.zs += lo; v.dv += lo; v.ndd += lo; v.ndz += lo; v.dfv += lo; v.rc += lo; v.rs += lo; v.tauR += lo;
    v.lam += lo; v.zhat += lo; v.ptau += lo; v.pc += lo; v.ps += lo;
    v.perm += lo; v.ndx += lo; v.dfx += lo; v.ra += lo; v.rb += lo; v.org += lo; v.posr += lo; v.posd += lo;
    v.nsl += lo; v.prot += lo;
    v.rho += m;
    v.cnt += 8 * m;
    return v;
  }
};

__device__ __forceinline__ double warp_sum(double v) {
  for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

__device__ double block_sum(double v, double* red) {
  int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
  v = warp_sum(v);
  __syncthreads();
  if (lane == 0) red[w] = v;
  __syncthreads();
  double s = (threadIdx.x < nw) ? red[threadIdx.x] : 0.0;
  if (w == 0) s = warp_sum(s);
  if (threadIdx.x == 0) red[0] = s;
  __syncthreads();
  double r = red[0];
  __syncthreads();
  return r;
}

__device__ double block_max(double v, double* red) {
  int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
  for (int o = 16; o; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
  __syncthreads();
  if (lane == 0) red[w] = v;
  __syncthreads();
  double s = (threadIdx.x < nw) ? red[threadIdx.x] : 0.0;
  if (w == 0)
    for (int o = 16; o; o >>= 1) s = fmax(s, __shfl_xor_sync(0xffffffffu, s, o));
  if (threadIdx.x == 0) red[0] = s;
  __syncthreads();
  double r = red[0];
  __syncthreads();
  return r;
}

// Exclusive prefix sum of one count per thread; *total gets the sum.  sc: 33 ints.
__device__ int block_scan(int v, int* sc, int* total) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  int x = v;
  for (int o = 1; o < 32; o <<= 1) {
    int y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  __syncthreads();
  if (lane == 31) sc[w] = x;
  __syncthreads();
  if (w == 0) {
    int s = lane < nw ? sc[lane] : 0;
    for (int o = 1; o < 32; o <<= 1) {
      int y = __shfl_up_sync(0xffffffffu, s, o);
      if (lane >= o) s += y;
    }
    sc[lane] = s;
  }
  __syncthreads();
  *total = sc[nw - 1];
  return x - v + (w ? sc[w - 1] : 0);
}

__device__ __forceinline__ double pow2(int e) { return __longlong_as_double((long long)(1023 + e) << 52); }

// Order-preserving integer key of a finite double (compared on the integer pipe).
__device__ __forceinline__ long long order_key(double x) {
  const long long b = __double_as_longlong(x);
  return b ^ ((b >> 63) & 0x7fffffffffffffffll);
}

// Tearing: dd = d with |e[p-1]| removed on both sides of every split point p.
__global__ void k_tear(int M, const double* __restrict__ d, const double* __restrict__ e,
                       double* __restrict__ dd) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= M) return;
  double v = d[i];
  if (i > 0 && i % LEAF == 0) v -= fabs(e[i - 1]);
  if ((i + 1) % LEAF == 0 && i + 1 < M) v -= fabs(e[i]);
  dd[i] = v;
}

// One warp per leaf: implicit QL with Wilkinson shift; lane r owns row r of the eigenvectors
// (shared memory), every lane runs the scalar recurrence (an FP64 instruction costs a warp the
// same for one lane as for 32), the split test is one ballot.  The leaf is scaled by a power of
// two so that a rotation needs one rsqrt instead of a hypot and two divisions.  Sorted
// ascending and written to Z/D at the end.  With leaves of 32 rows, hypot and divisions in
// lane 0 this kernel took 2.46 ms, with 16 rows 0.33 ms; at 8 the extra level of merges costs less than
// the leaves save (D&C of order 64 0.48 -> 0.35 ms, 2047 8.6 -> 6.6 ms).
__global__ void __launch_bounds__(32) k_leaf(int M, const double* __restrict__ dd, const double* __restrict__ e,
                                             double* __restrict__ D, double* __restrict__ Z, int ldz, int* st) {
  __shared__ double Zs[LEAF][33];
  __shared__ double dl[LEAF], el[LEAF];
  __shared__ int ord[LEAF];
  if (status_bad(st)) return;
  const int lane = threadIdx.x, lo = blockIdx.x * LEAF;
  const int n = min(LEAF, M - lo);
  double dv = lane < n ? dd[lo + lane] : 0.0, ev = lane < n - 1 ? e[lo + lane] : 0.0;
  int mx = max((int)((__double_as_longlong(dv) >> 52) & 0x7FF), (int)((__double_as_longlong(ev) >> 52) & 0x7FF));
  for (int o = 16; o; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  // 2^(1023 - mx) and its inverse, kept inside the normal range
  const int sh = max(-1000, min(1000, 1023 - mx));
  const double sc = pow2(sh), isc = pow2(-sh);
  if (lane < LEAF) {
    dl[lane] = dv * sc;
    el[lane] = fabs(ev * sc) < 0x1p-900 ? 0.0 : ev * sc;  // (a rotation of subnormal numbers is not orthogonal)
  }
#pragma unroll
  for (int c = 0; c < LEAF; ++c) Zs[c][lane] = (lane == c) ? 1.0 : 0.0;
  __syncwarp();
  int bad = mx == 0x7FF;  // a NaN or an infinity: the merges order finite numbers only
  for (int l = 0; l < n && !bad; ++l) {
    for (int iter = 0;; ++iter) {
      bool small = true;
      if (lane < n - 1) small = fabs(el[lane]) <= 2.0 * EPS * (fabs(dl[lane]) + fabs(dl[lane + 1]));
      const unsigned mask = __ballot_sync(0xffffffffu, small);
      const int m = l + __ffs(mask >> l) - 1;
      if (m == l) break;
      if (iter > 60) { bad = 1; break; }
      double g, r, s = 1.0, c = 1.0, p = 0.0;
      {
        const double a = 2.0 * el[l];
        g = (dl[l + 1] - dl[l]) / a;
        r = (fabs(g) < 0x1p400) ? sqrt(fma(g, g, 1.0)) : fabs(g);
        g = dl[m] - dl[l] + el[l] / (g + copysign(r, g));
      }
      double zhi = Zs[m][lane];  // column i + 1 of the running rotation
      int i = m - 1;
      bool early = false;
      for (; i >= l; --i) {
        const double ei = el[i], di = dl[i], di1 = dl[i + 1];
        const double f = s * ei, b = c * ei, h = fma(f, f, g * g);
        __syncwarp();
        if (h >= 0x1p-900) {
          const double ri = rsqrt(h);
          r = h * ri;
          s = f * ri;
          c = g * ri;
        } else {
          r = hypot(f, g);
          if (r == 0.0) {
            if (lane == 0) {
              el[i + 1] = 0.0;
              dl[i + 1] = di1 - p;
              el[m] = 0.0;
            }
            early = true;
            break;
          }
          s = f / r;
          c = g / r;
        }
        g = di1 - p;
        const double q = fma(di - g, s, 2.0 * c * b);
        p = s * q;
        if (lane == 0) {
          el[i + 1] = r;
          dl[i + 1] = g + p;
        }
        g = fma(c, q, -b);
        const double zi = Zs[i][lane];
        Zs[i + 1][lane] = fma(s, zi, c * zhi);
        zhi = fma(c, zi, -s * zhi);
      }
      Zs[i + 1][lane] = zhi;  // (after an early stop: the column the last rotation left)
      if (!early && lane == 0) {
        dl[l] -= p;
        el[l] = g;
        el[m] = 0.0;
      }
      __syncwarp();
    }
  }
  if (bad) {
    if (lane == 0) atomicCAS(st, 0, M + lo + 1);
    return;
  }
  if (lane < n) {
    const double v = dl[lane];
    int rank = 0;
    for (int j = 0; j < n; ++j) rank += dl[j] < v || (dl[j] == v && j < lane);
    ord[rank] = lane;
  }
  __syncwarp();
  if (lane < n) {
    for (int j = 0; j < n; ++j) Z[GEP_IX(lo + lane, lo + j, ldz)] = Zs[ord[j]][lane];
    D[lo + lane] = dl[ord[lane]] * isc;
  }
}

// Sorts the first c entries (key v, with companions) ascending when they are not already: the
// lists of k_prep are ascending up to the roundings of a few rotations, so this is a check that
// rarely does more; the sort itself ranks every entry against all (integer compares).
__device__ void sort_list(int c, double* v, double* z, int* ix, double* tv, double* tz, int* ti) {
  int inv = 0;
  for (int x = threadIdx.x + 1; x < c; x += blockDim.x) inv |= order_key(v[x - 1]) > order_key(v[x]);
  if (!__syncthreads_or(inv)) return;
  for (int x = threadIdx.x; x < c; x += blockDim.x) {
    const long long k = order_key(v[x]);
    int r = 0;
    for (int y = 0; y < c; ++y) {
      const long long o = order_key(v[y]);
      r += o < k || (o == k && y < x);
    }
    tv[r] = v[x];
    if (z) tz[r] = z[x];
    ti[r] = ix[x];
  }
  __syncthreads();
  for (int x = threadIdx.x; x < c; x += blockDim.x) {
    v[x] = tv[x];
    if (z) z[x] = tz[x];
    ix[x] = ti[x];
  }
  __syncthreads();
}

// Merge set-up (one CTA per merge): z, sort of the two halves' eigenvalues, deflation.  The
// deflation scan is sequential (a Givens rotation changes the next pair's operands), but
// only a rotated pair's successor needs its test re-evaluated: every pair's test is first
// formed in parallel from the undeflated values, one thread then follows only the chains
// that start at a rotated pair, and the lists are compacted in
// parallel (all set-ups of order 4096: 13.2 -> 0.23 ms).
__global__ void __launch_bounds__(1024) k_prep(int M, int half, const double* __restrict__ e,
                                               const double* __restrict__ D, const double* __restrict__ Z,
                                               int ldz, DcWs ws, int* st) {
  __shared__ double red[32];
  __shared__ int sc[33];
  __shared__ int snr;
  if (__syncthreads_or(status_bad(st))) return;  // (another merge of this launch may be storing it)
  const int lo = blockIdx.x * 2 * half, mid = lo + half, hi = min(M, mid + half);
  const DcWs w = ws.at(lo, blockIdx.x);
  const int tid = threadIdx.x, nt = blockDim.x;
  const int n = hi - lo, n1 = half;
  const double beta = e[mid - 1];
  const double sg = beta < 0.0 ? -1.0 : 1.0;
  auto field = [](double x) { return (int)((__double_as_longlong(x) >> 52) & 0x7FF); };
  int bad = 0;
  double zmax = 0.0, dmax = 0.0, dall = 0.0;  // dmax: of the values that the rank-one term reaches
  for (int t = tid; t < n; t += nt) {
    double z = (t < n1) ? Z[GEP_IX(mid - 1, lo + t, ldz)] : sg * Z[GEP_IX(mid, lo + t, ldz)];
    z *= 0.70710678118654752440;
    w.zs[t] = z;
    double dv = D[lo + t];
    w.dv[t] = dv;
    bad |= max(field(z), field(dv)) == 0x7FF;
    zmax = fmax(zmax, fabs(z));
    dall = fmax(dall, fabs(dv));
    if (z != 0.0) dmax = fmax(dmax, fabs(dv));
  }
  // The orders below are indices into this merge's arrays: what is not a number has none.
  if (__syncthreads_or(bad)) {
    if (tid == 0) atomicCAS(st, 0, M + lo + 1);
    return;
  }
  zmax = block_max(zmax, red);
  dmax = block_max(dmax, red);
  dall = block_max(dall, red);
  // The merge runs on numbers of order one: scaled by the power of two that brings those the rank-one term
  // reaches into [1, 2) (values of a decoupled block of another scale only pass through).
  const int top = field(fmax(dmax, fabs(beta)));
  const int sh = max(-1000, min(top ? 1023 - top : 1000, min(1000, 2000 - field(dall))));  // (top 0: subnormal)
  const double f = pow2(sh);
  const double rho = 2.0 * (fabs(beta) * f);
  for (int t = tid; t < n; t += nt) w.dv[t] *= f;
  __syncthreads();
  const double tol = 8.0 * EPS * 2.0 * fmax(dmax * f, rho * zmax);
  // merge the two ascending runs [0, n1) and [n1, n), the first run's entry first on ties
  for (int x = tid; x < n; x += nt) {
    const double v = w.dv[x];
    int a = (x < n1) ? n1 : 0, b = (x < n1) ? n : n1;  // search the other run
    while (a < b) {
      int c = (a + b) >> 1;
      bool before = (x < n1) ? (w.dv[c] < v) : (w.dv[c] <= v);
      if (before) a = c + 1; else b = c;
    }
    w.perm[(x < n1) ? x + (a - n1) : (x - n1) + a] = x;
  }
  __syncthreads();
  // positions whose z is not negligible, in order; posr marks the deflated positions
  const int chunk = (n + nt - 1) / nt, c0 = min(n, tid * chunk), c1 = min(n, c0 + chunk);
  int cnt = 0, nns;
  for (int q = c0; q < c1; ++q) {
    const bool neg = rho * fabs(w.zs[w.perm[q]]) <= tol;
    w.posr[q] = neg;
    cnt += !neg;
  }
  int o = block_scan(cnt, sc, &nns);
  for (int q = c0; q < c1; ++q)
    if (!w.posr[q]) w.nsl[o++] = q;
  __syncthreads();
  // the rotation test of every adjacent pair, from the undeflated values
  int any = 0;
  for (int m = 1 + tid; m < nns; m += nt) {
    const int pj = w.perm[w.nsl[m - 1]], t = w.perm[w.nsl[m]];
    double zs_ = w.zs[pj], zc = w.zs[t];
    double tau = hypot(zc, zs_);
    double c = zc / tau, sn = -zs_ / tau;
    double tdiff = w.dv[t] - w.dv[pj];
    const int rot = fabs(tdiff * c * sn) <= tol;
    w.prot[m] = rot;
    w.ptau[m] = tau;
    w.pc[m] = c;
    w.ps[m] = sn;
    any |= rot;
  }
  if (tid == 0) snr = 0;
  any = __syncthreads_or(any);
  if (any) {
    // the pairs that rotate, in order (posd), then their chains one after the other
    const int ch = (nns + nt - 1) / nt, m0 = max(1, min(nns, tid * ch)), m1 = min(nns, tid * ch + ch);
    int rc_ = 0, nrot;
    for (int m = m0; m < m1; ++m) rc_ += w.prot[m];
    int ro = block_scan(rc_, sc, &nrot);
    for (int m = m0; m < m1; ++m)
      if (w.prot[m]) w.posd[ro++] = m;
    __syncthreads();
    if (tid == 0) {
      int nr = 0, next = 0;
      for (int x = 0; x < nrot; ++x) {
        int m = w.posd[x];
        if (m < next) continue;  // already decided by the chain before it
        double tau = w.ptau[m], c = w.pc[m], sn = w.ps[m];
        for (;;) {
          const int pj = w.perm[w.nsl[m - 1]], t = w.perm[w.nsl[m]];
          const double dp = w.dv[pj], dt = w.dv[t];
          const double dnew = dp * sn * sn + dt * c * c;
          w.zs[t] = tau;
          w.zs[pj] = 0.0;
          w.ra[nr] = pj; w.rb[nr] = t; w.rc[nr] = c; w.rs[nr] = sn; ++nr;
          w.dv[t] = dnew;
          w.dv[pj] = dp * c * c + dt * sn * sn;
          w.posr[w.nsl[m - 1]] = 1;
          if (++m >= nns) break;
          // t was rotated into: the next pair's test with its new z and d
          const int t2 = w.perm[w.nsl[m]];
          const double zc = w.zs[t2];
          const double ntau = hypot(zc, tau), nc = zc / ntau, ns = -tau / ntau;
          const double tdiff = w.dv[t2] - dnew;
          if (!(fabs(tdiff * nc * ns) <= tol)) break;
          tau = ntau;
          c = nc;
          sn = ns;
        }
        next = m + 1;
      }
      snr = nr;
    }
    __syncthreads();
  }
  // both lists in sorted order of the undeflated values
  int k, kc = 0;
  for (int q = c0; q < c1; ++q) kc += !w.posr[q];
  int ko = block_scan(kc, sc, &k);
  for (int q = c0; q < c1; ++q) {
    const int t = w.perm[q];
    if (w.posr[q]) {
      w.dfx[q - ko] = t;
      w.dfv[q - ko] = w.dv[t];
    } else {
      w.ndx[ko] = t;
      w.ndd[ko] = w.dv[t];
      w.ndz[ko] = w.zs[t];
      ++ko;
    }
  }
  __syncthreads();
  sort_list(k, w.ndd, w.ndz, w.ndx, w.ptau, w.pc, w.perm);
  sort_list(n - k, w.dfv, nullptr, w.dfx, w.ptau, nullptr, w.perm);
  if (tid == 0) {
    w.cnt[0] = k;
    w.cnt[1] = n - k;
    w.cnt[2] = snr;
    w.cnt[3] = sh;
    w.rho[0] = rho;
  }
}

// The deflation rotations applied to the rows of U instead of the columns of Q:
// Q G_0 ... G_{nr-1} U = Q (G_0 (... (G_{nr-1} U))), so Q keeps its block-diagonal
// form and the merge product splits into one product per child.  One thread per column.
__global__ void k_rot_u(int M, int width, double* U, int ldu, DcWs ws, const int* st) {
  if (status_bad(st)) return;
  const int lo = blockIdx.y * width, n = min(width, M - lo);
  const DcWs w = ws.at(lo, blockIdx.y);
  int col = blockIdx.x * blockDim.x + threadIdx.x;
  if (col >= n) return;
  double* u = U + GEP_IX(lo, lo + col, ldu);
  for (int q = w.cnt[2] - 1; q >= 0; --q) {
    int a = w.ra[q], b = w.rb[q];
    double x = u[a], y = u[b], c = w.rc[q], s = w.rs[q];
    u[a] = c * x - s * y;
    u[b] = s * x + c * y;
  }
}

// One warp per root j of the secular equation on the k non-deflated poles.
__global__ void __launch_bounds__(256) k_secular(int width, DcWs ws, const int* st) {
  if (status_bad(st)) return;
  const DcWs w = ws.at(blockIdx.y * width, blockIdx.y);
  int j = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  int k = w.cnt[0];
  if (j >= k) return;
  const double rho = w.rho[0];
  const double* dd = w.ndd;
  const double* zz = w.ndz;
  int org;
  double lo, hi;
  if (j < k - 1) {
    double gap = dd[j + 1] - dd[j];
    double s = 0.0;
    for (int i = lane; i < k; i += 32) {
      double del = (dd[i] - dd[j]) - 0.5 * gap;
      s += zz[i] * zz[i] / del;
    }
    double fmid = 1.0 + rho * warp_sum(s);
    if (fmid >= 0.0) { org = j; lo = 0.0; hi = 0.5 * gap; }
    else { org = j + 1; lo = -0.5 * gap; hi = 0.0; }
  } else {
    double s = 0.0;
    for (int i = lane; i < k; i += 32) s += zz[i] * zz[i];
    org = j; lo = 0.0; hi = rho * warp_sum(s);
  }
  const double dorg = dd[org];
  const double DL = dd[j] - dorg;                          // left pole (relative)
  const double DR = (j < k - 1) ? dd[j + 1] - dorg : 0.0;  // right pole (relative)
  double tau = 0.5 * (lo + hi);
  for (int it = 0; it < 400; ++it) {
    double pL = 0.0, dpL = 0.0, pR = 0.0, dpR = 0.0;
    for (int i = lane; i < k; i += 32) {  // one reciprocal per pole (the FP64 pipe is the bound)
      double r = 1.0 / ((dd[i] - dorg) - tau);
      double t = zz[i] * zz[i] * r;
      if (i <= j) { pL += t; dpL += t * r; }
      else { pR += t; dpR += t * r; }
    }
    pL = rho * warp_sum(pL);
    dpL = rho * warp_sum(dpL);
    pR = rho * warp_sum(pR);
    dpR = rho * warp_sum(dpR);
    double f = 1.0 + pL + pR;
    if (f == 0.0) break;
    if (f > 0.0) hi = tau; else lo = tau;
    double errf = EPS * (8.0 * (1.0 + fabs(pL) + fabs(pR)) + fabs(tau) * (dpL + dpR));
    if (fabs(f) <= errf) break;
    if (hi - lo <= 4.0 * EPS * fmax(fabs(lo), fabs(hi))) break;
    // two-pole rational model around tau, solved for the step eta
    double a = DL - tau;
    double sL = dpL * a * a, cL = pL - dpL * a;
    double eta = NAN;
    if (j < k - 1) {
      double b = DR - tau;
      double sR = dpR * b * b, cR = pR - dpR * b;
      double C0 = 1.0 + cL + cR;
      double B2 = C0 * (a + b) + sL + sR;
      double C2 = C0 * a * b + sL * b + sR * a;
      if (C0 == 0.0) {
        eta = C2 / B2;
      } else {
        double disc = fmax(B2 * B2 - 4.0 * C0 * C2, 0.0);
        double q = 0.5 * (B2 + copysign(sqrt(disc), B2));
        double e1 = q / C0, e2 = (q != 0.0) ? C2 / q : NAN;
        bool ok1 = (tau + e1 > lo) && (tau + e1 < hi);
        bool ok2 = (tau + e2 > lo) && (tau + e2 < hi);
        if (ok1 && ok2) eta = fabs(e1) < fabs(e2) ? e1 : e2;
        else if (ok1) eta = e1;
        else if (ok2) eta = e2;
      }
    } else {
      double C0 = 1.0 + cL;
      if (C0 > 0.0) eta = a + sL / C0;
    }
    double tn = tau + eta;
    if (!(tn > lo && tn < hi)) tn = 0.5 * (lo + hi);
    if (tn == tau) break;
    tau = tn;
  }
  if (lane == 0) {
    w.org[j] = org;
    w.tauR[j] = tau;
    w.lam[j] = dorg + tau;
  }
}

// x <- x 2^-s with |x 2^-s| in [1, 2) (sign kept), e += s; zero and subnormal x are left as
// they are (a zero product stays zero).
__device__ __forceinline__ void renorm_exp(double& x, int& e) {
  const long long bits = __double_as_longlong(x);
  const int E = (int)((bits >> 52) & 0x7FF);
  if (E == 0 || E == 0x7FF) return;
  x = __longlong_as_double((bits & ~(0x7FFll << 52)) | (1023ll << 52));
  e += E - 1023;
}

// Warps 0..k-1 of a merge: Loewner formula zhat_i^2 = ((lam_i - d_i)/rho) prod_{j != i}
// (lam_j - d_i)/(d_j - d_i), one warp per i (lanes over j), and the place of root i in the
// ascending order of all n merged eigenvalues; warps k..n-1: the places of the deflated values.
// One thread per i left most of the GPU idle (992 us at k = 4096), and the order was one
// thread's merge of the two lists; both together at order 4096: 12.1 -> 0.51 ms.
__global__ void __launch_bounds__(256) k_zhat_order(int M, int width, double* __restrict__ D, DcWs ws, const int* st) {
  if (status_bad(st)) return;
  const int lo = blockIdx.y * width, n = min(width, M - lo);
  const DcWs w = ws.at(lo, blockIdx.y);
  const int i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (i >= n) return;
  const int k = w.cnt[0], nd = w.cnt[1];
  const double isc = pow2(-w.cnt[3]);
  if (i >= k) {
    if (lane == 0) {  // after the roots that are not above it (roots first on ties)
      const int m = i - k;
      const double v = w.dfv[m];
      int a = 0, b = k;
      while (a < b) {
        const int c = (a + b) >> 1;
        if (w.lam[c] <= v) a = c + 1; else b = c;
      }
      w.posd[m] = m + a;
      D[lo + m + a] = v * isc;
    }
    return;
  }
  const double di = w.ndd[i];
  // numerator and denominator products kept apart (one division at the end); every eighth
  // factor both are brought back to [1, 2) in magnitude, their binary exponents counted in
  // en, ed, so that neither over- nor underflows
  double pn = 1.0, pd = 1.0;
  if (lane == 0) pn = -((di - w.ndd[w.org[i]]) - w.tauR[i]) / w.rho[0];
  int en = 0, ed = 0, c = 0;
  for (int j = lane; j < k; j += 32) {
    if (j != i) {
      pn *= -((di - w.ndd[w.org[j]]) - w.tauR[j]);
      pd *= w.ndd[j] - di;
    }
    if (++c == 8) {
      c = 0;
      renorm_exp(pn, en);
      renorm_exp(pd, ed);
    }
  }
  renorm_exp(pn, en);
  renorm_exp(pd, ed);
  for (int o = 16; o; o >>= 1) {
    pn *= __shfl_xor_sync(0xffffffffu, pn, o);
    pd *= __shfl_xor_sync(0xffffffffu, pd, o);
    en += __shfl_xor_sync(0xffffffffu, en, o);
    ed += __shfl_xor_sync(0xffffffffu, ed, o);
  }
  if (lane == 0) {
    const double prod = ldexp(pn / pd, en - ed);
    w.zhat[i] = copysign(sqrt(fmax(prod, 0.0)), w.ndz[i]);
    const double v = w.lam[i];
    int a = 0, b = nd;
    while (a < b) {
      const int q = (a + b) >> 1;
      if (w.dfv[q] < v) a = q + 1; else b = q;
    }
    w.posr[i] = i + a;
    D[lo + i + a] = v * isc;
  }
}

// One CTA per column of U: root j's column posr[j] is the normalised z_hat_i / (d_i - lam_j) at
// rows ndx[i], a deflated value's column the unit vector of its row; all other entries zero.
__global__ void __launch_bounds__(256) k_ucols(int M, int width, double* U, int ldu, DcWs ws, const int* st) {
  __shared__ double red[32];
  if (status_bad(st)) return;
  const int lo = blockIdx.y * width, n = min(width, M - lo);
  const DcWs w = ws.at(lo, blockIdx.y);
  const int j = blockIdx.x, k = w.cnt[0];
  if (j >= n) return;
  if (j >= k) {
    double* col = U + GEP_IX(lo, lo + w.posd[j - k], ldu);
    const int one = w.dfx[j - k];
    for (int i = threadIdx.x; i < n; i += blockDim.x) col[i] = i == one ? 1.0 : 0.0;
    return;
  }
  const double dorg = w.ndd[w.org[j]], tj = w.tauR[j];
  double* col = U + GEP_IX(lo, lo + w.posr[j], ldu);
  for (int i = threadIdx.x; i < n - k; i += blockDim.x) col[w.dfx[i]] = 0.0;
  constexpr int KEEP = 8;  // entries a thread keeps in registers between the norm and the store
  double keep[KEEP], s = 0.0;
#pragma unroll
  for (int q = 0; q < KEEP; ++q) {
    const int i = threadIdx.x + q * blockDim.x;
    keep[q] = 0.0;
    if (i < k) {
      keep[q] = w.zhat[i] / ((w.ndd[i] - dorg) - tj);
      s = fma(keep[q], keep[q], s);
    }
  }
  for (int i = threadIdx.x + KEEP * blockDim.x; i < k; i += blockDim.x) {
    double u = w.zhat[i] / ((w.ndd[i] - dorg) - tj);
    s = fma(u, u, s);
    col[w.ndx[i]] = u;
  }
  const double inv = 1.0 / sqrt(block_sum(s, red));
#pragma unroll
  for (int q = 0; q < KEEP; ++q) {
    const int i = threadIdx.x + q * blockDim.x;
    if (i < k) col[w.ndx[i]] = keep[q] * inv;
  }
  for (int i = threadIdx.x + KEEP * blockDim.x; i < k; i += blockDim.x) col[w.ndx[i]] *= inv;
}

// Products of every merge of a narrow level (width <= FP64_WIDTH): Out(rows of a child, all n
// columns) = Z(child, child) U(child rows, :), 16 x 16 output tiles, one output per thread (an
// FP64 FMA holds its scheduler 64 clocks, so shared-memory reads are free beside it).
// Grid: (column tiles, row tiles of a child, child).
__global__ void __launch_bounds__(256) k_merge_prod(int M, int half, const double* __restrict__ Z, int ldz,
                                                    const double* __restrict__ U, int ldu, double* __restrict__ Out,
                                                    int ldo, const int* st) {
  __shared__ double As[FP64_WIDTH / 2][17], Bs[FP64_WIDTH / 2][17];
  if (status_bad(st)) return;
  const int mrg = blockIdx.z >> 1, ch = blockIdx.z & 1;
  const int lo = mrg * 2 * half, n = min(2 * half, M - lo);
  const int r0 = ch ? half : 0, nr = ch ? n - half : half;  // the child's rows inside the merge
  const int tr = blockIdx.y * 16, tc = blockIdx.x * 16;
  if (tr >= nr || tc >= n) return;
  const int t = threadIdx.x;
  const double* Zc = Z + GEP_IX(lo + r0, lo + r0, ldz);
  const double* Uc = U + GEP_IX(lo + r0, lo, ldu);
  for (int idx = t; idx < 16 * nr; idx += 256) {
    const int i = idx & 15, kk = idx >> 4;
    As[kk][i] = tr + i < nr ? Zc[GEP_IX(tr + i, kk, ldz)] : 0.0;
  }
  for (int idx = t; idx < 16 * nr; idx += 256) {
    const int kk = idx % nr, c = idx / nr;
    Bs[kk][c] = tc + c < n ? Uc[GEP_IX(kk, tc + c, ldu)] : 0.0;
  }
  __syncthreads();
  const int i = t & 15, c = t >> 4;
  double acc = 0.0;
#pragma unroll 8
  for (int kk = 0; kk < nr; ++kk) acc = fma(As[kk][i], Bs[kk][c], acc);
  if (tr + i < nr && tc + c < n) Out[GEP_IX(lo + r0 + tr + i, lo + tc + c, ldo)] = acc;
}

__global__ void k_copy_vec(int n, const double* __restrict__ s, double* __restrict__ d, const int* st) {
  if (status_bad(st)) return;
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) d[i] = s[i];
}

DcWs carve(char* base, int M, size_t* used) {
  DcWs w;
  size_t off = 0;
  auto takeD = [&](size_t n) { off = align256(off); double* p = (double*)(base + off); off += n * sizeof(double); return p; };
  auto takeI = [&](size_t n) { off = align256(off); int* p = (int*)(base + off); off += n * sizeof(int); return p; };
  size_t mm = (size_t)M * M, m = (size_t)M, nm = (size_t)M / (2 * LEAF) + 1;
  w.Qt = takeD(mm); w.U = takeD(mm);
  w.D = takeD(m); w.dd = takeD(m); w.zs = takeD(m); w.dv = takeD(m); w.ndd = takeD(m); w.ndz = takeD(m);
  w.dfv = takeD(m); w.rc = takeD(m); w.rs = takeD(m); w.tauR = takeD(m); w.lam = takeD(m); w.zhat = takeD(m);
  w.rho = takeD(nm);
  w.ptau = takeD(m); w.pc = takeD(m); w.ps = takeD(m);
  w.perm = takeI(m); w.ndx = takeI(m); w.dfx = takeI(m); w.ra = takeI(m); w.rb = takeI(m); w.org = takeI(m);
  w.posr = takeI(m); w.posd = takeI(m); w.cnt = takeI(8 * nm);
  w.nsl = takeI(m); w.prot = takeI(m);
  *used = align256(off);
  return w;
}

}  // namespace

size_t dc_ws_bytes(int M) {
  size_t used = 0;
  carve(nullptr, M, &used);
  return used;
}

int tridiag_eig_dc(gep_handle_t h, int M, const double* d, const double* e, double* wout, double* Z,
                   int ldz, double* ws, size_t ws_bytes, int engine) {
  if (M <= 0) return GEP_OK;
  size_t used = 0;
  DcWs w = carve((char*)ws, M, &used);
  if (ws_bytes < used) return GEP_ERR_ALLOC;
  cudaStream_t s = h->stream;
  const int* stc = h->d_status;
  // the eigenvectors alternate between Z and Qt level by level and end in Z
  int levels = 0;
  for (int half = LEAF; half < M; half *= 2) ++levels;
  double *cur = (levels & 1) ? w.Qt : Z, *nxt = (levels & 1) ? Z : w.Qt;
  int ldcur = (levels & 1) ? M : ldz, ldnxt = (levels & 1) ? ldz : M;
  k_tear<<<(M + 255) / 256, 256, 0, s>>>(M, d, e, w.dd);
  GEP_CHECK(check_launch(h));
  k_leaf<<<(M + LEAF - 1) / LEAF, 32, 0, s>>>(M, w.dd, e, w.D, cur, ldcur, h->d_status);
  GEP_CHECK(check_launch(h));
  for (int half = LEAF; half < M; half *= 2) {
    const int width = 2 * half;
    const int nm = (M - half + width - 1) / width;  // merges: those whose second half is not empty
    const int tail = nm * width;                    // rows from here on have no partner on this level
    const int nmax = M < width ? M : width;
    k_prep<<<nm, nmax >= 1024 ? 1024 : (nmax + 31) / 32 * 32, 0, s>>>(M, half, e, w.D, cur, ldcur, w, h->d_status);
    GEP_CHECK(check_launch(h));
    k_secular<<<dim3((nmax + 7) / 8, nm), 256, 0, s>>>(width, w, stc);
    GEP_CHECK(check_launch(h));
    k_zhat_order<<<dim3((nmax + 7) / 8, nm), 256, 0, s>>>(M, width, w.D, w, stc);
    GEP_CHECK(check_launch(h));
    k_ucols<<<dim3(nmax, nm), nmax >= 256 ? 256 : (nmax + 31) / 32 * 32, 0, s>>>(M, width, w.U, M, w, stc);
    GEP_CHECK(check_launch(h));
    k_rot_u<<<dim3((nmax + 127) / 128, nm), 128, 0, s>>>(M, width, w.U, M, w, stc);
    GEP_CHECK(check_launch(h));
    // Q = diag(Q1, Q2): one product per child (half the flops of a dense n x n product)
    if (width <= FP64_WIDTH) {
      k_merge_prod<<<dim3((nmax + 15) / 16, (half + 15) / 16, 2 * nm), 256, 0, s>>>(M, half, cur, ldcur, w.U, M, nxt,
                                                                                    ldnxt, stc);
      GEP_CHECK(check_launch(h));
    } else {
      for (int lo = 0; lo < tail; lo += width) {
        const int mid = lo + half, hi = M < lo + width ? M : lo + width;
        const int n = hi - lo, n1 = half, n2 = hi - mid;
        GEP_CHECK(dgemm(h, 'N', 'N', 'F', n1, n, n1, 1.0, cur + GEP_IX(lo, lo, ldcur), ldcur,
                        w.U + GEP_IX(lo, lo, M), M, 0.0, nxt + GEP_IX(lo, lo, ldnxt), ldnxt, engine));
        GEP_CHECK(dgemm(h, 'N', 'N', 'F', n2, n, n2, 1.0, cur + GEP_IX(mid, mid, ldcur), ldcur,
                        w.U + GEP_IX(mid, lo, M), M, 0.0, nxt + GEP_IX(mid, lo, ldnxt), ldnxt, engine));
      }
    }
    if (tail < M)
      GEP_CHECK(copy_matrix(h, M - tail, M - tail, cur + GEP_IX(tail, tail, ldcur), ldcur,
                            nxt + GEP_IX(tail, tail, ldnxt), ldnxt));
    double* tp = cur; cur = nxt; nxt = tp;
    int tl = ldcur; ldcur = ldnxt; ldnxt = tl;
  }
  k_copy_vec<<<(M + 255) / 256, 256, 0, s>>>(M, w.D, wout, stc);
  return check_launch(h);
}

// ---------------------------------------------------------------- T_evo path
namespace {

__global__ void k_gersh(int M, const double* __restrict__ d, const double* __restrict__ e, double* out) {
  __shared__ double red[32];
  double lo = INFINITY, hi = -INFINITY;
  for (int i = threadIdx.x; i < M; i += blockDim.x) {
    double r = (i > 0 ? fabs(e[i - 1]) : 0.0) + (i + 1 < M ? fabs(e[i]) : 0.0);
    lo = fmin(lo, d[i] - r);
    hi = fmax(hi, d[i] + r);
  }
  double mlo = -block_max(-lo, red);
  double mhi = block_max(hi, red);
  if (threadIdx.x == 0) {
    double span = mhi - mlo;
    out[0] = mlo - 1e-12 * span - 1e-300;
    out[1] = mhi + 1e-12 * span + 1e-300;
  }
}

// Sturm count: eigenvalues of T strictly below x, the sign changes of the leading minors
//     p_{i+1} = (d_i - x) p_i - e_{i-1}^2 p_{i-1}
// of T - xI with T scaled by a power of two to norm at most 1: three FP64 instructions a row
// instead of a division (565 clocks) in the chain of pivots; the same rounding errors per row,
// so the same backward error.  A zero minor counts as a sign change (the pivot of -0), and the
// pair is scaled up again, exactly, before it can underflow (one row grows it at most 3-fold).
// PRE: d and e hold the scaled diagonal and the squares of the scaled off-diagonal.
struct SturmState {
  double p = 1.0, pp = 0.0;
  int cnt = 0;
};

// One row, with every special case.
__device__ __forceinline__ void sturm_row(SturmState& s, double t, double e2) {
  double pn = fma(t, s.p, -(e2 * s.pp));
  const int hp = __double2hiint(s.p);
  int hn = __double2hiint(pn);
  if (((hn & 0x7fffffff) | __double2loint(pn)) == 0) {  // zero: a tiny value of the other sign
    pn = __hiloint2double((~hp & 0x80000000) | ((hp & 0x7ff00000) - (200 << 20)), 0);
    hn = __double2hiint(pn);
  }
  s.cnt += (unsigned)(hn ^ hp) >> 31;
  s.pp = s.p;
  s.p = pn;
  const int E = hn & 0x7ff00000;
  if (E < 0x3ff00000 - (300 << 20) || E > 0x3ff00000 + (300 << 20)) {
    const double f = E > 0x3ff00000 ? 0x1p-300 : (E == 0 ? 0x1p600 : 0x1p300);
    s.p *= f;
    s.pp *= f;
  }
}

// Rows are taken 32 at a time, their data spread over the lanes (the next 32 are on the way), and
// in blocks of 8 without any check but the smallest exponent met: a block that met one below
// 2^-400 (or a zero) is done again row by row.  Every lane of the warp calls this together.
template <bool PRE>
__device__ int sturm(int M, const double* __restrict__ d, const double* __restrict__ e, double x, double sc) {
  const int lane = threadIdx.x & 31;
  SturmState s;
  auto row = [&](int i, double& dv, double& ev) {
    dv = i < M ? d[i] : 0.0;
    ev = i > 0 && i < M ? e[i - 1] : 0.0;
    if (!PRE) {
      dv *= sc;
      ev *= sc;
      ev *= ev;
    }
  };
  double dn, en;
  row(lane, dn, en);
  for (int i0 = 0; i0 < M; i0 += 32) {
    const double dv = dn, ev = en;
    row(i0 + 32 + lane, dn, en);
#pragma unroll
    for (int b = 0; b < 32; b += 8) {
      const SturmState s0 = s;
      unsigned emin = 0xffffffffu;
      if (i0 + b + 8 <= M) {
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          const double t = __shfl_sync(0xffffffffu, dv, b + u) - x, e2 = __shfl_sync(0xffffffffu, ev, b + u);
          const double pn = fma(t, s.p, -(e2 * s.pp));
          const int hn = __double2hiint(pn);
          s.cnt += (unsigned)(hn ^ __double2hiint(s.p)) >> 31;
          emin = min(emin, (unsigned)hn & 0x7ff00000u);
          s.pp = s.p;
          s.p = pn;
        }
        // (8 rows grow the pair at most 2^13-fold: no block overflows from 2^300)
        const int E = __double2hiint(s.p) & 0x7ff00000;
        if (E > 0x3ff00000 + (300 << 20)) {
          s.p *= 0x1p-300;
          s.pp *= 0x1p-300;
        }
      } else {
        emin = 0;
      }
      if (__any_sync(0xffffffffu, emin < 0x3ff00000u - (400u << 20))) {
        s = s0;
        for (int u = 0; u < 8 && i0 + b + u < M; ++u)
          sturm_row(s, __shfl_sync(0xffffffffu, dv, b + u) - x, __shfl_sync(0xffffffffu, ev, b + u));
      }
    }
  }
  return s.cnt;
}

// d and e scaled to norm at most 1 (a power of two), e squared.
__device__ __forceinline__ double bisect_scale(const double* gb) {
  const int E = (int)((__double_as_longlong(fmax(fabs(gb[0]), fabs(gb[1]))) >> 52) & 0x7ff);
  const int k = max(1, min(2046, 2045 - E));  // 2^(1022 - E): norm into [1/2, 1)
  return __longlong_as_double((long long)k << 52);
}
__global__ void k_bisect_prep(int M, const double* __restrict__ d, const double* __restrict__ e,
                              const double* __restrict__ gb, double* __restrict__ ds, double* __restrict__ e2,
                              const int* st) {
  if (status_bad(st)) return;
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= M) return;
  const double sc = bisect_scale(gb);
  ds[i] = d[i] * sc;
  const double es = i + 1 < M ? e[i] * sc : 0.0;
  e2[i] = es * es;
}

// w[k], k < n: the (k+1)-th smallest eigenvalue of T (order M) by multisection on Sturm counts:
// a group of K lanes evaluates K interior points of the bracket at once (log2(K + 1) bits a
// count), K chosen so that every SM's four schedulers have a warp.  The first brackets come from
// the counts of a uniform grid (k_bisect_grid).
template <bool PRE>
__global__ void __launch_bounds__(32) k_bisect(int n, int M, int K, const double* __restrict__ d,
                                               const double* __restrict__ e, const double* __restrict__ gb,
                                               const int* __restrict__ grid_cnt, int ngrid,
                                               double* __restrict__ w, const int* st) {
  if (status_bad(st)) return;
  const int lane = threadIdx.x, sub = lane % K, per = 32 / K;
  const int k = blockIdx.x * per + lane / K;
  const double sc = bisect_scale(gb);
  double a = gb[0] * sc, b = gb[1] * sc;
  const bool live = k < n;
  if (live && ngrid > 0) {  // the grid cell that holds eigenvalue k: counts ascend along the grid
    int lo = 0, hi = ngrid;  // first grid point with a count above k
    while (lo < hi) {
      const int m = (lo + hi) >> 1;
      if (grid_cnt[m] > k) hi = m; else lo = m + 1;
    }
    const double h = (b - a) / (ngrid + 1), a0 = a, b0 = b;
    if (lo < ngrid) b = fma(h, lo + 1.0, a0);
    if (lo > 0) a = fma(h, (double)lo, a0);
    if (!(b <= b0)) b = b0;
  }
  const unsigned gmask = K == 32 ? 0xffffffffu : ((1u << K) - 1u) << (lane / K * K);
  for (int it = 0; it < 200; ++it) {
    const double mid = 0.5 * (a + b);
    const bool done = !live || mid <= a || mid >= b;
    if (__all_sync(0xffffffffu, done)) break;
    double x = K == 1 ? mid : fma((b - a) / (K + 1), sub + 1.0, a);
    if (x <= a || x >= b) x = mid;
    const bool above = sturm<PRE>(M, d, e, x, sc) > k;
    const unsigned m = __ballot_sync(0xffffffffu, above) & gmask;
    const int first = m ? __ffs(m) - 1 : -1;  // lowest point above eigenvalue k
    const double xb = __shfl_sync(0xffffffffu, x, first < 0 ? lane : first);
    const int below = first < 0 ? (lane / K * K + K - 1) : first - 1;
    const double xa = __shfl_sync(0xffffffffu, x, below < 0 ? 0 : below);
    if (!done) {
      if (first >= 0) b = xb;
      if (below >= lane / K * K) a = fmax(a, xa);
      if (a > b) a = b;
    }
  }
  if (live && sub == 0) w[k] = (0.5 * (a + b)) / sc;
}

// Sturm counts at ngrid points of a uniform grid inside the Gershgorin interval.
template <bool PRE>
__global__ void __launch_bounds__(32) k_bisect_grid(int M, const double* __restrict__ d, const double* __restrict__ e,
                                                    const double* __restrict__ gb, int* __restrict__ cnt, int ngrid,
                                                    const int* st) {
  if (status_bad(st)) return;
  const int g = blockIdx.x * 32 + threadIdx.x;
  const double sc = bisect_scale(gb), a = gb[0] * sc, b = gb[1] * sc, h = (b - a) / (ngrid + 1);
  const int c = sturm<PRE>(M, d, e, fma(h, g + 1.0, a), sc);
  if (g < ngrid) cnt[g] = c;
}

}  // namespace

int tridiag_eig_bisect(gep_handle_t h, int M, const double* d, const double* e, double* w, int n) {
  if (M <= 0) return GEP_OK;
  if (n < 0 || n > M) n = M;  // the n lowest eigenvalues w[0..n)
  if (n == 0) return GEP_OK;
  double* gb = (double*)(h->d_status + 8);  // two doubles of the handle's status block
  k_gersh<<<1, 1024, 0, h->stream>>>(M, d, e, gb);
  GEP_CHECK(check_launch(h));
  // four warps an SM (one a scheduler) are free of charge: their lanes share the eigenvalues
  const int lanes = 4 * 32 * h->sm_count;
  int K = 1;
  while (K < 32 && (long long)2 * K * n <= lanes) K *= 2;
  const int blocks = (n + 32 / K - 1) / (32 / K);
  // scratch of the split FP64 products: scaled diagonal, squared off-diagonal, grid counts
  const size_t need = 2 * (size_t)M + (lanes + 1) / 2;
  if (h->d_splitk && need <= SPLITK_DOUBLES) {
    double *ds = h->d_splitk, *e2 = ds + M;
    int* cnt = (int*)(e2 + M);
    const int ng = n > 64 ? lanes : 0;
    k_bisect_prep<<<(M + 255) / 256, 256, 0, h->stream>>>(M, d, e, gb, ds, e2, h->d_status);
    GEP_CHECK(check_launch(h));
    if (ng) {
      k_bisect_grid<true><<<lanes / 32, 32, 0, h->stream>>>(M, ds, e2, gb, cnt, ng, h->d_status);
      GEP_CHECK(check_launch(h));
    }
    k_bisect<true><<<blocks, 32, 0, h->stream>>>(n, M, K, ds, e2, gb, cnt, ng, w, h->d_status);
    return check_launch(h);
  }
  k_bisect<false><<<blocks, 32, 0, h->stream>>>(n, M, K, d, e, gb, nullptr, 0, w, h->d_status);
  return check_launch(h);
}

}  // namespace gep
