// Tridiagonalisation of small matrices, and of the last columns of large ones, in one launch of one cluster.
//
// The trailing matrix (order n <= 512) stays in the registers of 4 to 16 CTAs for the whole
// reduction: CTA k holds the rows l = k mod CL, a warp one or two of them, lane and slot the
// columns 32 t + lane, both triangles.  A column then costs one exchange instead of two grid barriers:
//   every CTA knows column i (thread l holds x_l) and forms the reflector for itself;
//   every warp applies the update of the step before to its rows (while warp 0 forms the
//   reflector's scalars), multiplies them with v and pushes y_l = (A v)_l together with its
//   element of column i + 1 to all CTAs (st.async, counted by an mbarrier of each);
//   every CTA forms w = tau y - (tau / 2) (tau y^T v) v and column i + 1 - v w_1 - w v_1 for itself.
// Unblocked: three products an element and column.  In FP64 they would take 3 n^2 / 32 clocks on 16
// SMs, more than everything else from n = 150 on, so the matrix is held in fixed point, as in the
// bulge chasing: C = q 2^-sh with the largest absolute row sum (a bound on the 2-norm, which no
// similarity changes) in (2^60, 2^61], v in Q62 with v_1 = 1, tau in Q61; ||w|| <= 2 ||C||.  A dense
// matrix of order 500 has entries of about 52 bits in it, so sums are kept ten bits longer than their
// result and an update rounds once (a rounding per product made the vectors of order 500 2.2 times as
// far off as FP64 panels); squares and their sums are exact.
//
// One unit for the whole matrix is no coarser than FP64 only while its rows are of like size: a decoupled or
// weakly coupled block far below the rest would lose its relative accuracy.  So where the row sums lie further
// apart than 2^TRC_SPREAD (without the first column, which only enters the first reflector) the same columns
// are taken in FP64, scaled by a power of two.  Order 500, two blocks: relative error of the small one's
// eigenvalues 9.9e-15, 9.1e-15, 9.4e-15 at 1/4, 1/8, 1/10 of the other's scale in fixed point, 6.5e-15 to
// 1.2e-14 below 1/16 in FP64; the FP64 columns take 0.46 / 0.86 / 1.8 / 5.4 ms at order 64 / 128 / 256 / 500,
// the fixed-point ones 0.23 / 0.38 / 0.79 / 2.5 ms (whole calls).
//
// Bound: the chain of a column (two warp and CTA reductions, the scalars, the push: 2.2 us) and from
// n = 260 on the integer products (7 us a column in all at n = 512).  S1 of the cooperative panels -> here:
// order 64 0.62 -> 0.14 ms, 128 1.28 -> 0.29, 256 2.74 -> 0.67, 500 5.67 -> 2.4, the last 512 columns of
// 1501 6 -> 2.5.  Beyond 512 rows the registers of 16 SMs are full.
#include <cooperative_groups.h>

#include "cluster.cuh"
#include "fixed.cuh"
#include "gep_internal.cuh"

namespace cg = cooperative_groups;

namespace gep {
namespace {

constexpr int TRC_SPREAD = 4;  // row sums further apart than 2^4: FP64
constexpr int TRC_MAX = 512, TRC_WARPS = 16, TRC_THREADS = 32 * TRC_WARPS, TRC_CL = 16;

struct TrcArgs {
  int n, ldc;
  double *C, *d, *e, *tau;  // C: element (0, 0) of the trailing matrix; d, e, tau: of its first column
  int* st;
};

struct TrcShared {
  int2 v[2][TRC_MAX], w[TRC_MAX];
  longlong2 recv[2][TRC_MAX];  // y_l, element (l, i + 1)
  longlong2 ack[TRC_CL];
  unsigned long long bar[2];
  longlong2 mx[TRC_WARPS], xmax[TRC_CL];
  ll xa, tauq, zs[TRC_WARPS];
  ll d[TRC_MAX], e[TRC_MAX], tau[TRC_MAX];  // results, turned into doubles at the end
  unsigned sq[TRC_WARPS][6];                // sums of squares in six parts
  int2 mq;
  int up, zero, done;
};

// Largest values of two numbers over the CTAs of the cluster (not below 0).
__device__ void trc_cluster_max(cg::cluster_group& cl, TrcShared& sh, ll& v0, ll& v1) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int o = 16; o; o >>= 1) {
    const ll q0 = __shfl_xor_sync(0xffffffffu, v0, o), q1 = __shfl_xor_sync(0xffffffffu, v1, o);
    v0 = max(v0, q0);
    v1 = max(v1, q1);
  }
  if (lane == 0) sh.mx[warp] = make_longlong2(v0, v1);
  __syncthreads();
  if (threadIdx.x < cl.num_blocks()) {
    longlong2 m = make_longlong2(0, 0);
    for (int q = 0; q < TRC_WARPS; ++q) m = make_longlong2(max(m.x, sh.mx[q].x), max(m.y, sh.mx[q].y));
    cl.map_shared_rank(sh.xmax, threadIdx.x)[cl.block_rank()] = m;
  }
  cl.sync();
  v0 = v1 = 0;
  for (int q = 0; q < (int)cl.num_blocks(); ++q) {
    v0 = max(v0, sh.xmax[q].x);
    v1 = max(v1, sh.xmax[q].y);
  }
  cl.sync();
}

// Entries of v and w are two limbs, or the words of a double.
__device__ __forceinline__ double trc_dbl(int2 a) { return __hiloint2double(a.y, a.x); }
__device__ __forceinline__ int2 trc_int2(double x) { return make_int2(__double2loint(x), __double2hiint(x)); }
__device__ __forceinline__ double trc_dbl(ll a) { return __longlong_as_double(a); }
__device__ __forceinline__ double trc_sum(double v) {
  for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// The columns, in fixed point or in FP64; a, x: elements times 2^scale.
template <bool F64, int RPW, int NT>
__device__ __forceinline__ void trc_columns(const TrcArgs& p, TrcShared& sh, cg::cluster_group& cl, ll (&a)[RPW][NT], ll x,
                                            int scale, bool finite, int cols) {
  const int CL = (int)cl.num_blocks(), k = (int)cl.block_rank();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, n = p.n, l = tid;
  auto out = [&](ll q) { return scale2(F64 ? trc_dbl(q) : qscaled(q, 0), -scale); };
  // two words to the same place in CTA q, counted by its barrier
  auto push = [&](longlong2* slot, int buf, int q, ll y, ll el) {
    uint32_t rd, rb;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(rd) : "r"(cta_shared(slot)), "r"(q));
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(rb) : "r"(cta_shared(&sh.bar[buf])), "r"(q));
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v2.b64 [%0], {%1, %2}, [%3];" ::"r"(rd),
                 "l"(y), "l"(el), "r"(rb) : "memory");
  };
  auto expect = [&](int i) {
    if (tid == 0)
      asm volatile("{ .reg .b64 t; mbarrier.arrive.expect_tx.shared::cta.b64 t, [%0], %1; }" ::"r"(cta_shared(&sh.bar[i & 1])),
                   "r"(16 * max(n - 1 - i, CL)) : "memory");
  };
  // y and the next column's elements of this warp's rows to every CTA
  auto push_rows = [&](int i, const ll (&y)[RPW], const ll (&el)[RPW]) {
#pragma unroll
    for (int u = 0; u < RPW; ++u) {
      const int r = (warp + TRC_WARPS * u) * CL + k;
      if (r > i && r < n && lane < CL) push(&sh.recv[i & 1][r], i & 1, lane, y[u], el[u]);
    }
    // A CTA whose rows are all done still reports every column: the others may be one column ahead of
    // it, as the two buffers allow, and not more.
    if (n - 1 - i < CL && warp == 0 && lane < CL) {
      const int first = i + 1 + (k - (i + 1) % CL + CL) % CL;  // its next row
      if (first >= n) push(&sh.ack[k], i & 1, lane, 0, 0);
    }
  };
  int i = 0;
  for (; i < cols; ++i) {
    const int buf = i & 1;
    const bool act = l > i && l < n;
    if (l == i) sh.d[i] = x;
    if (i == n - 1) break;
    expect(i);
    // ---- norm of x(i + 2 ..): from the exact squares
    if (F64) {
      const double q = act && l > i + 1 ? trc_dbl(x) : 0.0, s2 = trc_sum(q * q);
      if (lane == 0) sh.zs[warp] = __double_as_longlong(s2);
      if (l == i + 1) sh.xa = x;
    } else {
      const unsigned long long ax = act && l > i + 1 ? (unsigned long long)(x < 0 ? -x : x) : 0ull;
      unsigned q[6] = {0, 0, 0, 0, 0, 0};
      add_square(q, ax);
#pragma unroll
      for (int u = 0; u < 6; ++u) q[u] = __reduce_add_sync(0xffffffffu, q[u]);
      if (lane == 0)
#pragma unroll
        for (int u = 0; u < 6; ++u) sh.sq[warp][u] = q[u];
      if (l == i + 1) sh.xa = x;
    }
    __syncthreads();
    if (F64 && warp == 0) {
      const double s2 = trc_sum(lane < TRC_WARPS ? trc_dbl(sh.zs[lane]) : 0.0), xa = trc_dbl(sh.xa);
      double m = 0.0, tau = 0.0, beta = xa;
      const double n2 = fma(xa, xa, s2);
      const bool some = s2 != 0.0 && !tiny_squares(n2);
      if (some) {
        const double ri = rsqrt(n2);
        beta = -copysign(n2 * ri, xa);
        m = 1.0 / (xa - beta);
        tau = fma(fabs(xa), ri, 1.0);
      }
      if (lane == 0) {
        sh.mq = trc_int2(m);
        sh.tauq = sh.tau[i] = __double_as_longlong(tau);
        sh.zero = !some;
        sh.e[i] = __double_as_longlong(beta);
      }
    } else if (warp == 0) {
      unsigned q[6];
#pragma unroll
      for (int u = 0; u < 6; ++u) q[u] = lane < TRC_WARPS ? sh.sq[lane][u] : 0u;
      const Sum128 S = warp_squares(q);
      const ll xa = sh.xa;
      QReflector o;
      o.m = o.tq = 0;
      o.beta = xa;
      o.up = 0;
      const bool nz = (S.lo | S.hi) != 0;
      if (nz) o = q_reflector(xa, S);
      if (lane == 0) {
        sh.mq = qsplit(o.m);
        sh.tauq = o.tq;
        sh.up = o.up;
        sh.zero = !nz;
        sh.e[i] = o.beta;
        sh.tau[i] = o.tq;
      }
    }
    // ---- the update of the step before
    if (i > 0) {
#pragma unroll
      for (int u = 0; u < RPW; ++u) {
        const int r = (warp + TRC_WARPS * u) * CL + k;
        if (r > i && r < n) {
          const int2 vr = sh.v[buf ^ 1][r], wr = sh.w[r];
#pragma unroll
          for (int t = 0; t < NT; ++t) {
            if (32 * t + 31 <= i) continue;
            const int j = 32 * t + lane;
            const int2 vj = sh.v[buf ^ 1][j], wj = sh.w[j];
            if (F64) {  // (row above column first, so that both triangles round alike)
              const double x1 = trc_dbl(r > j ? vr : wr), y1 = trc_dbl(r > j ? wj : vj);
              const double x2 = trc_dbl(r > j ? wr : vr), y2 = trc_dbl(r > j ? vj : wj);
              a[u][t] = __double_as_longlong(fma(-x2, y2, fma(-x1, y1, trc_dbl(a[u][t]))));
              continue;
            }
            // (one rounding; with v_r^2 + v_j^2 <= 1 beside v_1 the four middle products stay below 2^63)
            a[u][t] -= ((qhh(vr, wj) + qhh(wr, vj)) << 2) + (qmid(vr, wj, qmid(wr, vj, 1ll << 29)) >> 30);
          }
        }
      }
    }
    __syncthreads();
    // ---- v
    const int2 tq = qsplit(sh.tauq);
    const double td = trc_dbl(sh.tauq);
    ll v = 0;
    if (act && !sh.zero) {
      if (F64) v = __double_as_longlong(l == i + 1 ? 1.0 : trc_dbl(x) * trc_dbl(sh.mq));
      else v = l == i + 1 ? 1ll << 62 : qmul<61>(qsplit(x << sh.up), sh.mq);
    }
    const int2 vl = F64 ? trc_int2(trc_dbl(v)) : qsplit(v);
    sh.v[buf][l] = vl;
    __syncthreads();
    // ---- y = A v on this warp's rows, pushed to every CTA with the element of column i + 1
    ll yr[RPW], nx[RPW];
#pragma unroll
    for (int u = 0; u < RPW; ++u) {
      const int r = (warp + TRC_WARPS * u) * CL + k;
      yr[u] = nx[u] = 0;
      if (r > i && r < n) {
        ll hh = 0, mm = 0, c1 = 0;
        double yd = 0.0;
#pragma unroll
        for (int t = 0; t < NT; ++t) {
          c1 |= a[u][t] & (t == ((i + 1) >> 5) ? -1ll : 0ll);
          if (32 * t + 31 <= i) continue;
          if (F64) {
            yd = fma(trc_dbl(a[u][t]), trc_dbl(sh.v[buf][32 * t + lane]), yd);
            continue;
          }
          const int2 q = qsplit(a[u][t]), vj = sh.v[buf][32 * t + lane];
          hh += qhh(q, vj);
          mm += qmid(q, vj, (((ll)q.x * vj.x) >> 32) + (1ll << 19)) >> 20;  // 10 bits more than a unit
        }
        yr[u] = F64 ? __double_as_longlong(trc_sum(yd)) : qwarp_sum((hh << 2) + ((mm + 512) >> 10));
        nx[u] = __shfl_sync(0xffffffffu, c1, (i + 1) & 31);
      }
    }
    push_rows(i, yr, nx);
    if (act && l % CL == k)  // (while the others push)
      p.C[GEP_IX(l, i, p.ldc)] = !finite ? NAN : l == i + 1 ? out(sh.e[i]) : F64 ? trc_dbl(v) : qscaled(v, 62);
    const bool ok = cluster_wait<false>(cta_shared(&sh.bar[buf]), (uint32_t)(i >> 1) & 1u, p.st);
    // ---- w and column i + 1
    const ll y = act ? sh.recv[buf][l].x : 0, raw = act ? sh.recv[buf][l].y : 0;
    const ll pl = F64 ? __double_as_longlong(td * trc_dbl(y)) : qmul<61>(qsplit(y), tq);
    {
      const ll s = F64 ? __double_as_longlong(trc_sum(trc_dbl(pl) * trc_dbl(v))) : qwarp_sum(qmul<62>(qsplit(pl), vl));
      if (lane == 0) sh.zs[warp] = s;
    }
    const ll y1 = sh.recv[buf][i + 1].x;
    if (!__syncthreads_and(ok)) {
      ++i;
      break;
    }
    if (F64) {
      const double al = 0.5 * td * trc_sum(lane < TRC_WARPS ? trc_dbl(sh.zs[lane]) : 0.0);
      const double w = fma(-al, trc_dbl(v), trc_dbl(pl)), w1 = fma(td, trc_dbl(y1), -al);
      sh.w[l] = trc_int2(act ? w : 0.0);
      x = act ? __double_as_longlong(fma(-trc_dbl(v), w1, trc_dbl(raw)) - w) : 0;
    } else {
      const int2 al = qsplit(qmul<62>(qsplit(qwarp_sum(lane < TRC_WARPS ? sh.zs[lane] : 0)), tq));
      const ll w = pl - qmul<62>(al, vl), w1 = qmul<61>(qsplit(y1), tq) - qjoin(al);
      sh.w[l] = qsplit(act ? w : 0);
      x = act ? raw - qmul<62>(vl, qsplit(sh.zero ? 0 : w1)) - w : 0;
    }
  }
  __syncthreads();
  if (k == 0 && l < cols) {
    p.d[l] = finite ? out(sh.d[l]) : NAN;
    if (l + 1 < n) {
      p.e[l] = finite ? out(sh.e[l]) : NAN;
      p.tau[l] = !finite ? NAN : F64 ? trc_dbl(sh.tau[l]) : qscaled(sh.tau[l], 61);
    }
  }
  // No CTA leaves before every push into its shared memory has landed.  After a timeout the CTAs may have
  // left the loop a column apart: those behind push the columns they are behind, for their bytes.
  const int done = i;  // columns that this CTA has pushed
  if (tid == 0) sh.done = done;
  cl.sync();
  const int last = __reduce_max_sync(0xffffffffu, lane < CL ? *cl.map_shared_rank(&sh.done, lane) : 0);
  const ll none[RPW] = {};
  for (int c = max(done - 1, 0); c < last; ++c) {
    if (c >= done) {
      expect(c);
      push_rows(c, none, none);
    }
    cluster_wait<true>(cta_shared(&sh.bar[c & 1]), (uint32_t)(c >> 1) & 1u, p.st);
  }
  cl.sync();
}

// RPW rows a warp, NT slots of 32 columns: n <= 32 NT and n <= 16 RPW CL.
template <int RPW, int NT>
__global__ void __launch_bounds__(TRC_THREADS, 1) k_trd_cluster(TrcArgs p) {
  __shared__ TrcShared sh;
  cg::cluster_group cl = cg::this_cluster();
  const int CL = (int)cl.num_blocks(), k = (int)cl.block_rank();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, n = p.n, l = tid;
  const bool bad = status_bad(p.st);  // (every thread of the cluster passes through the same barriers)
  if (tid == 0)
    for (int b = 0; b < 2; ++b)
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(cta_shared(&sh.bar[b])) : "memory");
  if (tid == 0) asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  for (int j = tid; j < TRC_MAX; j += TRC_THREADS) sh.v[0][j] = sh.v[1][j] = sh.w[j] = make_int2(0, 0);

  // rows as bits of doubles; their largest exponent
  ll a[RPW][NT];
  int em = 0;
#pragma unroll
  for (int u = 0; u < RPW; ++u) {
    const int r = (warp + TRC_WARPS * u) * CL + k;
#pragma unroll
    for (int t = 0; t < NT; ++t) {
      const int j = 32 * t + lane;
      a[u][t] = r < n && j < n ? __double_as_longlong(p.C[GEP_IX(r > j ? r : j, r > j ? j : r, p.ldc)]) : 0;
      em = max(em, (int)((a[u][t] >> 52) & 0x7FF));
    }
  }
  cl.sync();  // every CTA of the cluster runs, its barriers are initialised: its shared memory may be reached
  ll emx = em, low = 0;
  trc_cluster_max(cl, sh, emx, low);
  const int emax = (int)emx;
  const bool finite = emax < 0x7FF;
  // row sums with every element below 2^53, then the shift that puts the largest into (2^60, 2^61]; and the
  // smallest sum of a row of the matrix without its first column (of the first row: beside the diagonal)
  const int sh0 = 1075 - emax;
  ll rs = 0;
  low = 0;  // 2^62 - smallest
#pragma unroll
  for (int u = 0; u < RPW; ++u) {
    const int r = (warp + TRC_WARPS * u) * CL + k;
    ll s = 0, any = 0, first = 0, corner = 0;
#pragma unroll
    for (int t = 0; t < NT; ++t) {
      const ll m = a[u][t] & ~(1ll << 63), q = qfix(m, sh0);
      s += q;
      if (t == 0 && lane == 0) {
        first = q;
        corner = m;
      } else {
        any |= m;
      }
    }
    s = qwarp_sum(s);
    rs = max(rs, s);
    const ll rest = s - __shfl_sync(0xffffffffu, first, 0);
    if (__any_sync(0xffffffffu, any != 0)) low = max(low, (1ll << 62) - rest);
    else if (r == 0 && __shfl_sync(0xffffffffu, corner, 0) != 0) low = max(low, (1ll << 62) - s);  // its diagonal alone
  }
  trc_cluster_max(cl, sh, rs, low);
  const bool wide = finite && low > 0 && (1ll << 62) - low < rs >> TRC_SPREAD;
  const int scale = wide ? 1023 - emax : sh0 + (rs > 0 ? __clzll(rs) - 3 : 0);
  auto scaled = [&](double q) { return wide ? __double_as_longlong(scale2(q, scale)) : qfix(__double_as_longlong(q), scale); };
#pragma unroll
  for (int u = 0; u < RPW; ++u)
#pragma unroll
    for (int t = 0; t < NT; ++t) a[u][t] = scaled(trc_dbl(a[u][t]));
  const ll x = l < n ? scaled(p.C[l]) : 0;
  cl.sync();  // every element is read before the first reflector is stored
  const int cols = bad ? 0 : n;
  if (wide) trc_columns<true, RPW, NT>(p, sh, cl, a, x, scale, finite, cols);
  else trc_columns<false, RPW, NT>(p, sh, cl, a, x, scale, finite, cols);
}

template <int RPW, int NT>
int trc_launch(gep_handle_t h, const TrcArgs& a, int cl) {
  static DeviceOnce attributes;
  GEP_CHECK(once_per_device(attributes, []() -> int {
    GEP_CUDA(cudaFuncSetAttribute((const void*)k_trd_cluster<RPW, NT>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
    return GEP_OK;
  }));
  static DeviceValue fits;  // (one cluster size per instance but the smallest)
  if (!cluster_fits(fits, (const void*)k_trd_cluster<RPW, NT>, NT == 2 ? 4 : cl, TRC_THREADS, 0))
    return GEP_ERR_UNSUPPORTED;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(cl);
  cfg.blockDim = dim3(TRC_THREADS);
  cfg.stream = h->stream;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = cl;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  GEP_CUDA(cudaLaunchKernelEx(&cfg, k_trd_cluster<RPW, NT>, a));
  return check_launch(h);
}

}  // namespace

// Whether tridiag_cluster takes a trailing matrix of order n.
bool tridiag_cluster_takes(int n) { return n <= TRC_MAX; }

// Reduces the n x n symmetric matrix in the lower triangle of C to tridiagonal form: d, e, tau and the
// reflectors below the subdiagonal, as tridiag_1stage stores them.  GEP_ERR_UNSUPPORTED before any work
// where the cluster cannot be resident.
int tridiag_cluster(gep_handle_t h, int n, double* C, int ldc, double* d, double* e, double* tau) {
  if (n <= 0) return GEP_OK;
  if (n > TRC_MAX) return GEP_ERR_UNSUPPORTED;
  TrcArgs a;
  a.n = n; a.ldc = ldc; a.C = C; a.d = d; a.e = e; a.tau = tau; a.st = h->d_status;
  // 16 rows a CTA: a warp each
  if (n <= 64) return trc_launch<1, 2>(h, a, n <= 16 ? 1 : n <= 32 ? 2 : 4);
  if (n <= 128) return trc_launch<1, 4>(h, a, 8);
  if (n <= 256) return trc_launch<1, 8>(h, a, 16);
  return trc_launch<2, 16>(h, a, 16);
}

}  // namespace gep
