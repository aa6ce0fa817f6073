// QR factorisation of a panel of at most 32 columns with its T factor in one cluster of 16 CTAs, fixed point.
//
// As k_panel_qr (band.cu): warp w of a CTA holds RPW consecutive rows, lane j column j, and one exchange a
// column carries the partial dots of the next pivot column with all columns (those to its right
// give w = v^T P, those to its left the Gram entries of T) and the next pivot row.  The exchange
// goes through distributed shared memory instead of a grid barrier, and since only 16 SMs then share
// the rows, the rows are 64-bit fixed point: column j is held as q 2^-s_j with its 2-norm (which no
// reflector changes) at most 2^60, reflectors in Q62 with v_1 = 1, tau in Q61; dots are exact 128-bit
// sums, so that a pivot column that has become tiny still gives an orthogonal reflector.  The
// scalars of a reflector are formed by warp 0 of every CTA; an extra warp of CTA 0 accumulates T in FP64.
//
// A column's unit is fair to rows of like size only: where the row sums of the matrix lie further apart than 2^4
// (band.cu's scan) the same exchange carries FP64 numbers, columns scaled by powers of two.
//
// A column: every CTA pushes its sums (and the owner of the pivot row that row) to all 16
// (st.async, counted by an mbarrier of each); warp 0 adds them up and forms the scalars and, lane by lane,
// tau w_j; the row warps apply the reflector and form the next dots.  All CTAs push for every column, so
// none is more than one ahead and two buffers do.
// Bound: the chain of a column (exchange, scalars, two CTA reductions: 2.3 us), then integer issue, about
// 140 clocks a row of a warp and column.  Per panel of 32 columns, k_panel_qr (grid barriers) -> here:
// 500 rows 130 -> 85 us, 1000 rows 135 -> 101 us, 2000 rows 150 -> 134 us; with 16 rows a warp 3000 rows take 210 us
// against 160, so longer panels stay there.  S1b at order 516 4.57 -> 2.68 ms, 1024 8.9 -> 5.8, 2047 15.7 -> 14.2,
// 4000 38.6 -> 37.0.
#include <cooperative_groups.h>

#include <type_traits>

#include "cluster.cuh"
#include "fixed.cuh"
#include "gep_internal.cuh"

namespace cg = cooperative_groups;

namespace gep {
namespace {

constexpr int QC = 16, QW = 16, QN = 32;  // CTAs, row warps, columns
constexpr int QTHREADS = 32 * (QW + 1);

struct QrArgs {
  int n, nb, ldp, r0, ldv;
  double *P, *tau, *Va, *Vb, *T;
  const int* wide;  // nonzero: FP64
  int* st;
};

__device__ __forceinline__ double qr_dbl(ll a) { return __longlong_as_double(a); }
__device__ __forceinline__ double qr_dbl(int2 a) { return __hiloint2double(a.y, a.x); }
__device__ __forceinline__ int2 qr_int2(double x) { return make_int2(__double2loint(x), __double2hiint(x)); }

// Exact sum of products of numbers split into balanced limbs.
struct Dot128 {
  ll hh = 0, mh = 0, ml = 0, l0 = 0;
  __device__ __forceinline__ void add(int2 a, int2 b) {
    hh += (ll)a.y * b.y;
    const ll l = (ll)a.x * b.x, m = (ll)a.y * b.x + ((ll)a.x * b.y + (l >> 32));
    l0 += (unsigned)l;
    mh += m >> 32;
    ml += (unsigned)m;
  }
  __device__ __forceinline__ Sum128 get() const {  // hh 2^64 + (mh 2^32 + ml) 2^32 + l0
    Sum128 r, t;
    r.hi = hh + mh + (ml >> 32);
    r.lo = ml << 32;
    t.hi = 0;
    t.lo = l0;
    return add128(r, t);
  }
};

struct QrShared {
  Sum128 part[QW][QN + 1];   // sums of the warps (read two columns of all warps at a time)
  Sum128 recv[2][QC][QN];    // sums of the CTAs
  ll rrow[2][QN];            // pivot row, received
  ll prow[QN];               // pivot row, at its owner
  unsigned long long bar[2];
  int emx[QC][QN];
  int2 tw[QN], mq;           // tau w_j; m of the reflector
  ll beta;
  double T[QN][QN + 1];
  ll g[2][QN], tq[2];        // Gram entries of the column (Q60), tau (Q61)
  int up, done, fail;        // fail: column + 1 whose wait gave up, 0 for none
};

// Named barriers: 1 all warps, 2 the row warps.
__device__ __forceinline__ void all_sync() { asm volatile("bar.sync 1, %0;" ::"n"(QTHREADS) : "memory"); }
__device__ __forceinline__ void row_sync() { asm volatile("bar.sync 2, %0;" ::"n"(32 * QW) : "memory"); }

template <int RPW>
__global__ void __cluster_dims__(QC, 1, 1) __launch_bounds__(QTHREADS, 1) k_panel_qr_cluster(QrArgs p) {
  constexpr int ROWS = QW * RPW;
  extern __shared__ __align__(16) unsigned char smraw[];
  QrShared& sh = *reinterpret_cast<QrShared*>(smraw);
  double* tile = reinterpret_cast<double*>(smraw + (sizeof(QrShared) + 15) / 16 * 16);  // [column][ROWS + 1]
  cg::cluster_group cl = cg::this_cluster();
  const int k = (int)cl.block_rank(), tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int n = p.n, nb = p.nb, nref = n < nb ? n : nb;
  const bool bad = status_bad(p.st), worker = warp < QW, use_fp64 = *p.wide != 0;
  if (tid == 0) {
    for (int b = 0; b < 2; ++b)
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(cta_shared(&sh.bar[b])) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    sh.fail = 0;
  }
  for (int idx = tid; idx < QN * (QN + 1); idx += QTHREADS) (&sh.T[0][0])[idx] = 0.0;
  for (int idx = k * QTHREADS + tid; !bad && idx < p.r0 * nb; idx += QC * QTHREADS) {
    const size_t o = (size_t)(idx / p.r0) * p.ldv + idx % p.r0;
    p.Va[o] = 0.0;
    p.Vb[o] = 0.0;
  }
  // ---- rows, and the scale of every column
  const int rb = k * ROWS, row0 = rb + warp * RPW;
  for (int idx = tid; idx < ROWS * QN; idx += QTHREADS) {
    const int r = idx % ROWS, j = idx / ROWS;
    tile[j * (ROWS + 1) + r] = rb + r < n && j < nb ? p.P[rb + r + (size_t)j * p.ldp] : 0.0;
  }
  cl.sync();  // every CTA of the cluster runs, its barriers are initialised: its shared memory may be reached
  ll a[RPW];
  int em = 0;
#pragma unroll
  for (int u = 0; u < RPW; ++u) {
    a[u] = worker ? __double_as_longlong(tile[lane * (ROWS + 1) + warp * RPW + u]) : 0;
    em = max(em, (int)((a[u] >> 52) & 0x7FF));
  }
  if (worker) sh.part[warp][lane].lo = em;
  __syncthreads();
  if (warp == 0) {
    for (int w = 1; w < QW; ++w) em = max(em, (int)sh.part[w][lane].lo);
    for (int q = 0; q < QC; ++q) cl.map_shared_rank(&sh, q)->emx[k][lane] = em;
  }
  cl.sync();
  for (int q = 0; q < QC; ++q) em = max(em, sh.emx[q][lane]);
  const int sh0 = 1075 - em;  // entries below 2^53
  const bool finite = em < 0x7FF;
  {
    Dot128 d;
#pragma unroll
    for (int u = 0; u < RPW; ++u) {
      const int2 q = qsplit(qfix(a[u], sh0));
      d.add(q, q);
    }
    if (worker) sh.part[warp][lane] = d.get();
  }
  __syncthreads();
  if (warp == 0) {
    Sum128 s = sh.part[0][lane];
    for (int w = 1; w < QW; ++w) s = add128(s, sh.part[w][lane]);
    for (int q = 0; q < QC; ++q) cl.map_shared_rank(&sh, q)->recv[0][k][lane] = s;
  }
  cl.sync();
  int scale;
  {
    Sum128 s = sh.recv[0][0][lane];
    for (int q = 1; q < QC; ++q) s = add128(s, sh.recv[0][q][lane]);
    const int bits = s.hi ? 128 - __clzll(s.hi) : 64 - __clzll(s.lo);  // norm^2 < 2^bits
    scale = use_fp64 ? 1023 - em : sh0 + 60 - (bits + 1) / 2;
  }
#pragma unroll
  for (int u = 0; u < RPW; ++u) a[u] = use_fp64 ? __double_as_longlong(scale2(qr_dbl(a[u]), scale)) : qfix(a[u], scale);
  cl.sync();  // recv is read everywhere before the first push

  auto expect = [&](int c) {
    if (tid == 0)
      asm volatile("{ .reg .b64 t; mbarrier.arrive.expect_tx.shared::cta.b64 t, [%0], %1; }" ::"r"(cta_shared(&sh.bar[c & 1])),
                   "r"(QC * QN * 16 + QN * 8) : "memory");
  };
  // warp w pushes the sums of columns 2 w and 2 w + 1, one CTA a lane pair, and the owner the pivot row
  auto push = [&](int c, Sum128 s) {
    const int col = 2 * warp + (lane & 1);
    uint32_t rd, rb;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(rd) : "r"(cta_shared(&sh.recv[c & 1][k][col])), "r"(lane >> 1));
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(rb) : "r"(cta_shared(&sh.bar[c & 1])), "r"(lane >> 1));
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v2.b64 [%0], {%1, %2}, [%3];" ::"r"(rd),
                 "l"(s.lo), "l"(s.hi), "r"(rb) : "memory");
    if (c / ROWS == k) {
      asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(rd) : "r"(cta_shared(&sh.rrow[c & 1][col])), "r"(lane >> 1));
      asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.b64 [%0], %1, [%2];" ::"r"(rd),
                   "l"(sh.prow[col]), "r"(rb) : "memory");
    }
  };
  bool run = !bad;
  ll xk = 0;  // lane u: the pivot column in the warp's row u
  int c = -1;
  auto columns = [&](auto arithmetic) {
    constexpr bool wide = decltype(arithmetic)::value;
    for (; run && c < nref; ++c) {
      const int nc = c + 1;
      if (c >= 0) {
        if (warp == 0) {
          const bool ok = cluster_wait<false>(cta_shared(&sh.bar[c & 1]), (uint32_t)(c >> 1) & 1u, p.st);
          const Sum128(*rv)[QN] = sh.recv[c & 1];
          if (wide) {
            double s = 0.0;
#pragma unroll
            for (int q = 0; q < QC; ++q) s += qr_dbl(rv[q][lane].lo);
            const double pr = qr_dbl(sh.rrow[c & 1][lane]);
            const double xn2 = __shfl_sync(0xffffffffu, s, c), alpha = __shfl_sync(0xffffffffu, pr, c);
            double tt = 0.0, sl = 0.0, be = alpha;
            const double n2 = fma(alpha, alpha, xn2);
            if (xn2 > 0.0 && !tiny_squares(n2)) {
              const double ri = rsqrt(n2);
              be = -copysign(n2 * ri, alpha);
              sl = 1.0 / (alpha - be);
              tt = fma(fabs(alpha), ri, 1.0);
            }
            const double w = fma(sl, s, pr);  // v^T P(:, j); for j < c the Gram entry v_j^T v
            sh.tw[lane] = qr_int2(lane > c ? tt * w : 0.0);
            sh.g[c & 1][lane] = __double_as_longlong(w);
            if (lane == 0) {
              sh.mq = qr_int2(sl);
              sh.beta = __double_as_longlong(be);
              sh.tq[c & 1] = __double_as_longlong(tt);
            }
          } else {
            Sum128 s = rv[0][lane];
#pragma unroll
            for (int q = 1; q < QC; ++q) s = add128(s, rv[q][lane]);
            const ll pr = sh.rrow[c & 1][lane];
            const unsigned long long xlo = (unsigned long long)__shfl_sync(0xffffffffu, s.lo, c);
            const ll xhi = __shfl_sync(0xffffffffu, s.hi, c), al_q = __shfl_sync(0xffffffffu, pr, c);
            ll tw = 0, g = pr >> 2;
            QReflector o;
            o.m = o.tq = 0;
            o.beta = al_q;
            o.up = 0;
            if ((xhi | (ll)xlo) != 0) {
              Sum128 x2;
              x2.hi = xhi;
              x2.lo = (ll)xlo;
              o = q_reflector(al_q, x2);
              // to the right: w = p + S / (alpha - beta), tau w; to the left: the Gram entry, Q60.  In the unit
              // of x 2^up the divisor is 2^123 / m, so S is taken times 2^-(61 - up).
              const int sft = lane < c ? 63 - o.up : 61 - o.up;
              const ll t = sft ? (ll)(((unsigned long long)s.hi << (64 - sft)) | ((unsigned long long)s.lo >> sft)) : s.lo;
              g = (lane < c ? pr >> 2 : pr) + qmul<62>(qsplit(t), qsplit(o.m));
              if (lane > c) tw = qmul<61>(qsplit(g), qsplit(o.tq));
            }
            sh.tw[lane] = qsplit(tw);
            sh.g[c & 1][lane] = g;
            if (lane == 0) {
              sh.mq = qsplit(o.m);
              sh.up = o.up;
              sh.beta = o.beta;
              sh.tq[c & 1] = o.tq;
            }
          }
          if (lane == 0 && !ok) sh.fail = c + 1;
        }
        all_sync();
        if (sh.fail == c + 1) break;  // (a warp still here may already see the next column's)
        if (worker) {
          const int2 tw = sh.tw[lane];
          const ll be = sh.beta;
          if (wide) {
            const double vk = qr_dbl(xk) * qr_dbl(sh.mq), t = qr_dbl(tw);
#pragma unroll
            for (int u = 0; u < RPW; ++u) {
              const int r = row0 + u;
              const double v = __shfl_sync(0xffffffffu, vk, u);
              if (r > c) a[u] = __double_as_longlong(lane == c ? v : fma(-v, t, qr_dbl(a[u])));
              else if (r == c) a[u] = lane == c ? be : __double_as_longlong(qr_dbl(a[u]) - t);
            }
          } else {
            // lane u forms v of the warp's row u
            const int2 vk = qsplit(qmul<61>(qsplit(xk << sh.up), sh.mq));
#pragma unroll
            for (int u = 0; u < RPW; ++u) {
              const int r = row0 + u;
              int2 v;
              v.x = __shfl_sync(0xffffffffu, vk.x, u);
              v.y = __shfl_sync(0xffffffffu, vk.y, u);
              if (r > c) a[u] = lane == c ? qjoin(v) : a[u] - qmul<62>(v, tw);
              else if (r == c) a[u] = lane == c ? be : a[u] - qjoin(tw);
            }
          }
        } else if (k == 0) {  // column c of T: T(0:c, c) = -tau T(0:c, 0:c) G(0:c, c)
          const double tt = wide ? qr_dbl(sh.tq[c & 1]) : qscaled(sh.tq[c & 1], 61);
          const double gl = lane >= c ? 0.0 : wide ? qr_dbl(sh.g[c & 1][lane]) : qscaled(sh.g[c & 1][lane], 60);
          if (lane == 0) p.tau[c] = finite ? tt : NAN;
          double s = 0.0;
          for (int q = 0; q < c; ++q) s = fma(sh.T[lane][q], __shfl_sync(0xffffffffu, gl, q), s);
          sh.T[lane][c] = lane < c ? -tt * s : (lane == c ? tt : 0.0);
          __syncwarp();
        }
      }
      if (nc >= nref) break;
      if (worker) {
        expect(nc);
        Dot128 d;
        double f = 0.0;
        xk = 0;
#pragma unroll
        for (int u = 0; u < RPW; ++u) {
          const int r = row0 + u;
          if (wide) {
            const double x = __shfl_sync(0xffffffffu, qr_dbl(a[u]), nc);
            if (lane == u) xk = r > nc ? __double_as_longlong(x) : 0;
            if (r > nc) f = fma(x, qr_dbl(a[u]), f);
            else if (r == nc) sh.prow[lane] = a[u];
            continue;
          }
          const int2 q = qsplit(a[u]);
          int2 x;
          x.x = __shfl_sync(0xffffffffu, q.x, nc);
          x.y = __shfl_sync(0xffffffffu, q.y, nc);
          if (lane == u) xk = r > nc ? qjoin(x) : 0;
          if (r > nc) d.add(x, q);
          else if (r == nc) sh.prow[lane] = a[u];
        }
        sh.part[warp][lane] = d.get();
        if (wide) sh.part[warp][lane].lo = __double_as_longlong(f);
        row_sync();
        // warp w adds columns 2 w and 2 w + 1 over the warps
        Sum128 s = sh.part[lane >> 1][2 * warp + (lane & 1)];
#pragma unroll
        for (int o = 2; o < 32; o <<= 1) {
          Sum128 t;
          t.lo = __shfl_xor_sync(0xffffffffu, s.lo, o);
          t.hi = __shfl_xor_sync(0xffffffffu, s.hi, o);
          if (wide) s.lo = __double_as_longlong(qr_dbl(s.lo) + qr_dbl(t.lo));
          else s = add128(s, t);
        }
        push(nc, s);
      }
    }
  };
  if (use_fp64) columns(std::true_type());
  else columns(std::false_type());
  __syncthreads();
  if (!bad) {
    // R back through the column's scale, reflectors from Q62
    if (worker)
#pragma unroll
      for (int u = 0; u < RPW; ++u) {
        const int r = row0 + u;
        const double x = r > lane ? (use_fp64 ? qr_dbl(a[u]) : qscaled(a[u], 62))
                                  : scale2(use_fp64 ? qr_dbl(a[u]) : qscaled(a[u], 0), -scale);
        tile[lane * (ROWS + 1) + warp * RPW + u] = finite ? x : NAN;
      }
    __syncthreads();
    for (int idx = tid; idx < ROWS * nb; idx += QTHREADS) {
      const int lr = idx % ROWS, j = idx / ROWS, r = rb + lr;
      if (r >= n) continue;
      const double x = tile[j * (ROWS + 1) + lr], v = r > j ? x : (r == j ? 1.0 : 0.0);
      p.P[r + (size_t)j * p.ldp] = x;
      const size_t o = (size_t)j * p.ldv + p.r0 + r;
      p.Va[o] = v;
      p.Vb[o] = v;
    }
    if (k == 0)
      for (int idx = tid; idx < nb * nb; idx += QTHREADS) p.T[idx] = sh.T[idx % nb][idx / nb];
  }
  // No CTA leaves before every push into its shared memory has landed.  After a timeout the CTAs may have
  // left the loop a column apart: those behind push the columns they are behind, for their bytes.
  const int done = c + 1;  // columns that this CTA has pushed
  if (tid == 0) sh.done = done;
  cl.sync();
  const int last = __reduce_max_sync(0xffffffffu, lane < QC ? *cl.map_shared_rank(&sh.done, lane) : 0);
  Sum128 none;
  none.lo = none.hi = 0;
  for (int q = max(done - 1, 0); q < last; ++q) {
    if (q >= done && worker) {
      expect(q);
      push(q, none);
    }
    cluster_wait<true>(cta_shared(&sh.bar[q & 1]), (uint32_t)(q >> 1) & 1u, p.st);
  }
  cl.sync();
}

template <int RPW>
int qr_launch(gep_handle_t h, const QrArgs& a) {
  constexpr int smem = (int)((sizeof(QrShared) + 15) / 16 * 16 + sizeof(double) * QN * (QW * RPW + 1));
  static DeviceOnce attributes;
  GEP_CHECK(once_per_device(attributes, []() -> int {
    GEP_CUDA(cudaFuncSetAttribute(k_panel_qr_cluster<RPW>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
    GEP_CUDA(cudaFuncSetAttribute(k_panel_qr_cluster<RPW>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    return GEP_OK;
  }));
  static DeviceValue fits;
  if (!cluster_fits(fits, (const void*)k_panel_qr_cluster<RPW>, QC, QTHREADS, smem)) return GEP_ERR_UNSUPPORTED;
  k_panel_qr_cluster<RPW><<<QC, QTHREADS, smem, h->stream>>>(a);
  return check_launch(h);
}

}  // namespace

// Panels that panel_qr_cluster takes: 8 rows a warp (see the times above).
bool panel_qr_cluster_takes(int n, int nb) { return nb <= QN && n <= QC * QW * 8; }

// QR of the n x nb panel P (ld ldp): R and the reflectors in P, tau, V at full height (r0 zero rows first, ld
// ldv) in Va and Vb, T (nb x nb).  *wide (device): FP64.  GEP_ERR_UNSUPPORTED before any work where the cluster cannot be resident.
int panel_qr_cluster(gep_handle_t h, int n, int nb, double* P, int ldp, double* tau, double* Va, double* Vb, int r0,
                     int ldv, double* T, const int* wide) {
  if (!panel_qr_cluster_takes(n, nb)) return GEP_ERR_UNSUPPORTED;
  QrArgs a;
  a.n = n; a.nb = nb; a.ldp = ldp; a.r0 = r0; a.ldv = ldv;
  a.P = P; a.tau = tau; a.Va = Va; a.Vb = Vb; a.T = T; a.wide = wide; a.st = h->d_status;
  if (n <= QC * QW) return qr_launch<1>(h, a);
  if (n <= QC * QW * 2) return qr_launch<2>(h, a);
  if (n <= QC * QW * 4) return qr_launch<4>(h, a);
  return qr_launch<8>(h, a);
}

}  // namespace gep
