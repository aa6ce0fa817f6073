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
// a^2 2^-63, the low limb's square (never negative, so not a rounding error) included.
__device__ __forceinline__ ll qsquare(int2 a) {
  return (qhh(a, a) << 1) + (qmid(a, a, (1ll << 30) + (((ll)a.x * a.x) >> 32)) >> 31);
}
// x 2^e as an integer, for a positive normal x with x 2^e < 2^63 (rounded half up).
__device__ __forceinline__ ll qint(double x, int e) {
  const ll bits = __double_as_longlong(x);
  const int sh = (int)(bits >> 52) - 1075 + e;
  const ll m = (bits & 0xFFFFFFFFFFFFFll) | (1ll << 52);
  return sh >= 0 ? m << sh : (sh > -54 ? (m + (1ll << (-sh - 1))) >> -sh : 0);
}
// 1 / sqrt(x) and 1 / x for normal x: the hardware's seeds (about 20 bits) and one third-order
// step each, y += y e (1/2 + 3/8 e) with e = 1 - x y^2, and r += r (e + e^2) with e = 1 - x r.
__device__ __forceinline__ double qrsqrt(double x) {
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double e = fma(-x * y, y, 1.0);
  return fma(y * e, fma(0.375, e, 0.5), y);
}
__device__ __forceinline__ double qrcp(double x) {
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
  const double e = fma(-x, r, 1.0);
  return fma(r, fma(e, e, e), r);
}

__device__ __forceinline__ double scale2(double x, int e) {  // x 2^e, e within +-2100
  const int a = e / 2, c = e - a;
  return x * __longlong_as_double((ll)(1023 + a) << 52) * __longlong_as_double((ll)(1023 + c) << 52);
}

}  // namespace
}  // namespace gep
