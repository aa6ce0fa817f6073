// Shared by the product kernels on the tensor cores (gemm_oz.cu, gemm_res.cu): PTX wrappers of
// mbarriers, TMA, tcgen05 and TMEM, bounded waits, and the integer forms of FP64 scaling and rounding.
#pragma once
#include <cuda.h>
#include <math.h>

#include <atomic>

#include "gep_internal.cuh"

namespace gep {
namespace {

// ------------------------------------------------------------------ numbers

// Biased exponent field of |x| (0 for zero / subnormal).
__device__ __forceinline__ int exp_field(double x) { return (int)((__double_as_longlong(x) >> 52) & 0x7FF); }

// A row of op(A) or a column of op(B) that holds a NaN or an infinity: integers cannot carry it, so the
// epilogues store NaN wherever one of the two raw exponents of an output says so.
__device__ __forceinline__ bool nonfinite(int raw_a, int raw_b) { return max(raw_a, raw_b) == 0x7FF; }
constexpr long long NAN_BITS = 0x7FF8ll << 48;

// Row scale exponent from the largest biased exponent m of the row: e with max |x| < 2^(e-1)
// when xbit = 1 (for a normal x with biased exponent E, |x| < 2^(E-1022)), so that the
// leading digit lies in [-64, 64] like the others; xbit = 0 (the FP32-grade setting, whose
// few levels stay exact with a leading digit in [-128, 128]) keeps max |x| < 2^e.  0 for an
// all-zero row.
__device__ __forceinline__ int scale_exp(int m, int xbit) { return m ? m - 1022 + xbit : 0; }

// F = round(x 2^(7S - e)) as a signed integer (|F| < 2^(7S)), from the IEEE bits: the
// magnitude is rounded half away from zero (error at most half a unit of the last digit).
// The row's own exponent e keeps the left shift at most 3.
__device__ __forceinline__ long long to_fixed(double x, int e, int S) {
  const long long bits = __double_as_longlong(x);
  const int E = (int)((bits >> 52) & 0x7FF);
  if (E == 0) return 0;
  const unsigned long long m = ((unsigned long long)bits & 0xFFFFFFFFFFFFFull) | (1ull << 52);
  const int sh = E - 1075 + 7 * S - e;
  unsigned long long qv;
  if (sh >= 0) qv = m << sh;
  else if (sh > -54) qv = (m + (1ull << (-sh - 1))) >> (-sh);
  else qv = 0;  // below half a unit of the last digit
  return (bits < 0) ? -(long long)qv : (long long)qv;
}

// FP32 bit pattern of the small integer d + bias (|d + bias| <= 256): 1.5 * 2^23 + d is a
// float of the binade [2^23, 2^24) whose last bits are d, and subtracting 1.5 * 2^23 leaves
// d exactly; with at most 9 significant bits its upper half is its BF16 pattern.
__device__ __forceinline__ unsigned f32_bits_of_int(int d, int bias) {
  return (unsigned)__float_as_int(__int_as_float(0x4B400000 + bias + d) - 12582912.0f);
}

// ------------------------------------------------------------------ PTX helpers

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ unsigned long long gtimer() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("{ .reg .b64 st; mbarrier.arrive.shared::cta.b64 st, [%0]; }" ::"r"(bar) : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("{ .reg .b64 st; mbarrier.arrive.expect_tx.shared::cta.b64 st, [%0], %1; }" ::"r"(bar), "r"(bytes)
               : "memory");
}

__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{ .reg .pred p; mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2; selp.u32 %0, 1, 0, p; }"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}

// Bounded wait: gives up after ~4 s of wall time and records a timeout.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, int* st) {
  if (mbar_try(bar, parity)) return true;
  unsigned long long t0 = gtimer();
  for (;;) {
    if (mbar_try(bar, parity)) return true;
    if (gtimer() - t0 > 4000000000ull) {
      atomicExch(st + 1, GEP_ERR_TIMEOUT);
      return false;
    }
    if (*(volatile int*)(st + 1) != 0) return false;  // another CTA already gave up
  }
}

__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap* map, int c0, int c1, int c2, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
      ::"r"(dst), "l"((unsigned long long)map), "r"(c0), "r"(c1), "r"(c2), "r"(bar)
      : "memory");
}

__device__ __forceinline__ void prefetch_map(const CUtensorMap* map) {
  asm volatile("prefetch.tensormap [%0];" ::"l"((unsigned long long)map) : "memory");
}

// Shared-memory matrix descriptor: K-major, 64-byte swizzle, 8-row groups 512 B apart.
__device__ __forceinline__ uint64_t sdesc_sw64(uint32_t addr) {
  uint64_t d = 0;
  d |= (uint64_t)((addr & 0x3FFFF) >> 4);   // start address
  d |= (uint64_t)1 << 16;                   // leading byte offset (unused for swizzled K-major)
  d |= (uint64_t)(512 >> 4) << 32;          // stride byte offset
  d |= (uint64_t)1 << 46;                   // descriptor version (sm_100 family)
  d |= (uint64_t)4 << 61;                   // layout: SWIZZLE_64B
  return d;
}

// The same with 128-byte swizzle: 8-row groups of 1024 B.
__device__ __forceinline__ uint64_t sdesc_sw128(uint32_t addr) {
  uint64_t d = 0;
  d |= (uint64_t)((addr & 0x3FFFF) >> 4);
  d |= (uint64_t)1 << 16;
  d |= (uint64_t)(1024 >> 4) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)2 << 61;                   // layout: SWIZZLE_128B
  return d;
}

// Instruction descriptor, kind::f16: D f32, A/B bf16, both K-major, M = 128, N = n.
__device__ __forceinline__ uint32_t idesc_bf16(int n) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
}

__device__ __forceinline__ void umma(uint32_t dtmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{ .reg .pred p; setp.ne.b32 p, %4, 0; tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p; }"
      ::"r"(dtmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(acc)
      : "memory");
}

__device__ __forceinline__ void umma_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }

// 32 lanes x 16 consecutive 32-bit columns of TMEM from taddr; waits for the load
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float* v) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float* v) {
  uint32_t r[32];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
      "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
        "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
        "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}

__device__ __forceinline__ void tmem_ld8(uint32_t taddr, float* v) {
  uint32_t r[8];
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 8; ++i) v[i] = __uint_as_float(r[i]);
}

template <int N>
__device__ __forceinline__ void tmem_ld(uint32_t taddr, float* v) {
  if constexpr (N == 8) tmem_ld8(taddr, v);
  else if constexpr (N == 16) tmem_ld16(taddr, v);
  else tmem_ld32(taddr, v);
}

// Bits of the double nearest to (A + B 2^-64) 2^(e - 63) (the bits beyond the 64 leading ones are
// dropped before rounding half up: an error of 2^-11 of half a unit), built with integer operations
// only: an FP64 instruction holds a scheduler 64 clocks, an FP64 compare included, so the whole
// epilogue has none but the addition of beta C.
__device__ __forceinline__ long long fixed128_to_bits(long long A, unsigned long long B, int e) {
  const long long neg = A >> 63;
  A = (A ^ neg) + (neg != 0 && B == 0 ? 1 : 0);  // magnitude
  B = (B ^ (unsigned long long)neg) - (unsigned long long)neg;
  if (A == 0) {  // all of the value lies in B
    if (B == 0) return 0;
    A = (long long)(B >> 1);
    B <<= 63;
    e -= 63;
    if (A == 0) { A = 1; B = 0; --e; }  // B was 1
  }
  const int lz = __clzll(A);  // 1 .. 63
  const unsigned long long m = ((unsigned long long)A << lz) | (B >> (64 - lz));
  const unsigned long long q = (m >> 11) + ((m >> 10) & 1ull);
  const int ex = e - lz + 1023;
  if (ex <= 0 || ex >= 2046) {  // outside the normal range: let FP64 arithmetic handle it
    const double v = ldexp((double)q, e - lz - 52);
    return __double_as_longlong(neg ? -v : v);
  }
  return (long long)(((unsigned long long)(ex - 1) << 52) + q) | (neg & (1ll << 63));
}

// The same of (hi 2^D + lo) 2^adj (0 <= D < 64).  With the fused split: 128^3 47 -> 28 us,
// 2000 x 2000 x 64 101 -> 54 us, 512 x 8192 x 512 180 -> 156 us, 4096^3 3107 -> 3067 us.
__device__ __forceinline__ long long fixed_to_bits(long long hi, long long lo, int D, int adj) {
  const long long A = hi + (lo >> D);                                          // T = A 2^D + B 2^(D - 64)
  const unsigned long long B = D ? (unsigned long long)lo << (64 - D) : 0ull;  // the low D bits, left-aligned
  return fixed128_to_bits(A, B, 63 + D + adj);
}

// ------------------------------------------------------------------ host

// cuTensorMapEncodeTiled is a driver-API call; it is resolved at run time through the
// runtime's entry-point query so the library does not link libcuda directly (it then
// loads on machines without a GPU driver, e.g. for symbol checks).
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
  static std::atomic<EncodeTiledFn> fn{nullptr};
  if (!fn.load()) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn.store((EncodeTiledFn)p);
  }
  return fn.load();
}

}  // namespace
}  // namespace gep
