// 64-bit fixed-point arithmetic of the reduction kernels (band.cu, tridiag_cluster.cu): an FP64
// instruction holds a scheduler of this part for 64 clocks, a fixed-point product about 20.
#pragma once
#include <math.h>

namespace gep {
namespace {

typedef long long ll;

// A fixed-point number as two balanced limbs, value = hi 2^32 + lo with lo in [-2^31, 2^31).
__device__ __forceinline__ int2 qsplit(ll a) {
  const int lo = (int)a;
  return make_int2(lo, (int)(a >> 32) - (lo >> 31));
}
__device__ __forceinline__ ll qjoin(int2 a) { return ((ll)a.y << 32) + a.x; }
__device__ __forceinline__ ll qhh(int2 a, int2 b) { return (ll)a.y * b.y; }
__device__ __forceinline__ ll qmid(int2 a, int2 b, ll c) { return (ll)a.y * b.x + ((ll)a.x * b.y + c); }
// a b 2^-S, rounded (the low x low limb product, at most half a unit, is dropped)
template <int S>
__device__ __forceinline__ ll qmul(int2 a, int2 b) {
  return (qhh(a, b) << (64 - S)) + (qmid(a, b, 1ll << (S - 33)) >> (S - 32));
}

// Sum over the warp (it has to fit 64 bits) by three 32-bit warp reductions.
__device__ __forceinline__ ll qwarp_sum(ll v) {
  const unsigned lo = __reduce_add_sync(0xffffffffu, (unsigned)v & 0xFFFFFu);
  const unsigned mi = __reduce_add_sync(0xffffffffu, (unsigned)(v >> 20) & 0xFFFFFu);
  const int hi = __reduce_add_sync(0xffffffffu, (int)(v >> 40));
  return ((ll)hi << 40) + ((ll)mi << 20) + lo;
}
// The double nearest to a non-negative integer (half up: truncation would lengthen every
// reflector by the same sign, a growth of the spectrum by 2^-59 a sweep).
__device__ __forceinline__ double qdouble(unsigned long long x) {
  if (x == 0) return 0.0;
  const int lz = __clzll((ll)x);
  const unsigned long long y = x << lz;
  return __longlong_as_double((ll)(((unsigned long long)(1085 - lz) << 52) + (y >> 11) + ((y >> 10) & 1ull)));
}
// x 2^e as an integer, for a positive normal x with x 2^e < 2^63 (rounded half up).
__device__ __forceinline__ ll qint(double x, int e) {
  const ll bits = __double_as_longlong(x);
  const int sh = (int)(bits >> 52) - 1075 + e;
  const ll m = (bits & 0xFFFFFFFFFFFFFll) | (1ll << 52);
  return sh >= 0 ? m << sh : (sh > -54 ? (m + (1ll << (-sh - 1))) >> -sh : 0);
}
__device__ __forceinline__ double scale2(double x, int e) {  // x 2^e, e within +-2100
  const int a = e / 2, c = e - a;
  return x * __longlong_as_double((ll)(1023 + a) << 52) * __longlong_as_double((ll)(1023 + c) << 52);
}

// v 2^-sh as a double (correctly rounded; sh within the normal range).
__device__ __forceinline__ double qscaled(ll v, int sh) {
  if (v == 0) return 0.0;
  const double m = qdouble((unsigned long long)(v < 0 ? -v : v));
  return __longlong_as_double((__double_as_longlong(m) - ((ll)sh << 52)) | (v & (1ll << 63)));
}

// x 2^sh rounded to an integer, from the bits of a finite x (|x| 2^sh < 2^62).
__device__ __forceinline__ ll qfix(ll bits, int sh) {
  const int E = (int)((bits >> 52) & 0x7FF);
  if (E == 0) return 0;
  const ll m = (bits & 0xFFFFFFFFFFFFFll) | (1ll << 52);
  const int s = E - 1075 + sh;
  const ll q = s >= 0 ? m << s : (s > -54 ? (m + (1ll << (-s - 1))) >> -s : 0);
  return bits < 0 ? -q : q;
}

struct alignas(16) Sum128 {
  ll lo, hi;  // hi 2^64 + lo (lo unsigned)
};
__device__ __forceinline__ Sum128 add128(Sum128 a, Sum128 b) {
  Sum128 r;
  asm("add.cc.s64 %0, %2, %4;\n\taddc.s64 %1, %3, %5;"
      : "=l"(r.lo), "=l"(r.hi) : "l"(a.lo), "l"(a.hi), "l"(b.lo), "l"(b.hi));
  return r;
}

// Exact sums of squares of numbers up to 2^61 in six parts of 22, 22, 20 and 20, 20, 18 bits, for 32-bit
// warp reductions (sums of up to 512 squares).
__device__ __forceinline__ void add_square(unsigned (&q)[6], unsigned long long ax) {
  const unsigned long long hi = __umul64hi(ax, ax), lo = ax * ax;
  q[0] += (unsigned)lo & 0x3FFFFFu;
  q[1] += (unsigned)(lo >> 22) & 0x3FFFFFu;
  q[2] += (unsigned)(lo >> 44);
  q[3] += (unsigned)hi & 0xFFFFFu;
  q[4] += (unsigned)(hi >> 20) & 0xFFFFFu;
  q[5] += (unsigned)(hi >> 40);
}
__device__ __forceinline__ Sum128 warp_squares(const unsigned (&p)[6]) {
  ll q[6];
#pragma unroll
  for (int u = 0; u < 6; ++u) q[u] = __reduce_add_sync(0xffffffffu, p[u]);
  Sum128 S, t;  // q0 + q1 2^22 + q2 2^44 + (q3 + q4 2^20 + q5 2^40) 2^64, every part below 2^32
  const ll mid = q[1] + (q[0] >> 22), top = q[2] + (mid >> 22);
  S.lo = (q[0] & 0x3FFFFF) | ((mid & 0x3FFFFF) << 22);
  S.hi = q[3] + (q[4] << 20) + (q[5] << 40);
  t.lo = top << 44;
  t.hi = top >> 20;
  return add128(S, t);
}

// Scalars of the reflector that sends x = (alpha, x1 ..) to (beta, 0 ..), from alpha and the exact
// S = sum of the squares of x1 .. (> 0; alpha^2 + S < 2^124):
//   v_i = (x_i 2^up) m 2^-61 in Q62 (v_0 = 1), m signed; tau = tq 2^-61; beta.
// 1 / sqrt and 1 / x start from the FP32 functions (about 21 bits) and take one third-order step each,
// y (1 + e / 2 + 3 e^2 / 8) with e = 1 - x y^2 and r (1 + e + e^2) with e = 1 - x r, in integers: the
// same in FP64 is a chain of a dozen dependent instructions, 1700 clocks.
struct QReflector {
  ll m, tq, beta;
  int up;
};
__device__ __forceinline__ QReflector q_reflector(ll alpha, Sum128 S) {
  typedef unsigned long long ull;
  QReflector o;
  const ull al = (ull)(alpha < 0 ? -alpha : alpha);
  Sum128 q;
  q.lo = (ll)(al * al);
  q.hi = (ll)__umul64hi(al, al);
  q = add128(q, S);
  const ull hi = (ull)q.hi, lo = (ull)q.lo;
  const int t = (hi ? __clzll((ll)hi) : 64 + __clzll((ll)lo)) & ~1;  // 4 .. 126
  // x = M 2^-64 in [1/4, 1), the norm is sqrt(x) 2^(64 - t / 2)
  const ull M = t >= 64 ? lo << (t - 64) : (hi << t) | (lo >> (64 - t));
  o.up = t / 2 - 2;
  const float yf = rsqrtf((float)(unsigned)(M >> 32) * 0x1p-32f);
  const ll Y0 = (ll)__float2uint_rn(yf * 0x1p23f) << 38;                 // Q61, in (1, 2]
  const ull Y2 = (ull)Y0 << 1;
  const ll E = (1ll << 60) - (ll)__umul64hi(M, __umul64hi(Y2, Y2));      // Q60
  const ll e2 = __mul64hi(E << 2, E << 2);
  const ull Y = (ull)(Y0 + __mul64hi(Y0, ((E >> 1) + ((3 * e2) >> 3)) << 4)) << 1;  // Q62
  const ull s = __umul64hi(M, Y);                                        // sqrt(x), Q62
  const ull aq = al << o.up;                                             // |alpha| in the same unit
  o.tq = (1ll << 61) + (ll)__umul64hi(aq << 1, Y);
  const ull d = min(aq + s, (1ull << 63) - 1);                           // at least 2^61
  const float rf = 1.0f / ((float)(unsigned)(d >> 31) * 0x1p-32f);
  const ull R0 = (ull)__float2uint_rn(rf * 0x1p21f) << 39;               // Q60, in (1, 4]
  const ll F = (1ll << 60) - (ll)__umul64hi(d << 1, R0);
  const ll f2 = __mul64hi(F << 2, F << 2);
  const ll R = (ll)R0 + __mul64hi((ll)R0, (F + f2) << 4);
  o.m = alpha < 0 ? -R : R;
  const ll nrm = o.up > 0 ? (ll)((s + (1ull << (o.up - 1))) >> o.up) : (ll)s;
  o.beta = alpha < 0 ? nrm : -nrm;
  return o;
}

}  // namespace
}  // namespace gep
