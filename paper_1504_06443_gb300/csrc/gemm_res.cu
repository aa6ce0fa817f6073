// Large FP64-accurate products C = alpha op(A) op(B) + beta C through residues: the second scheme of
// Ozaki, Uchino and Imamura (products of integer matrices modulo coprime numbers, joined by the Chinese
// remainder theorem) on the BF16 tensor cores.
//
// Every row of op(A) and column of op(B) becomes integers F = round(x 2^(56 - e)), |F| <= 2^55, as for
// the digit planes of gemm_oz.cu.  The integer product X = sum_k F^A F^B, |X| <= K 2^110, is determined
// by its residues modulo 16 coprime numbers m_i <= 256 with product P > 2^125.4 while
// K <= 2^14: one BF16 plane product per number instead of the 36 digit products, and X is exact
// (the digit scheme drops the levels below 2^-54 of the scale).  Balanced residues are at most 128 in
// magnitude, so FP32 accumulation in TMEM is exact over 1024 of K; after each such chunk the sums are
// reduced modulo m_i and kept as bytes.  The planes of op(B) are scaled by (P / m_i)^-1 mod m_i, so
// that the byte t_i of output and modulus is already the CRT weight:
//     X = sum_i t_i (P / m_i) - q P,   q = nearest integer of sum_i t_i / m_i.
//
// Three steps: residues of both operands (k_res_split), the 16 products (k_res_gemm: one item per
// modulus and 256 x 256 tile of a CTA pair, bytes out), the reconstruction (k_res_crt: 128-bit integers, then the
// double nearest to the value, alpha and beta).  Against the digit planes the operands take twice the bytes
// and every output 32 bytes more, so this pays where K is large: see res_product_wins.
//
// 4096^3: 3067 us with digit planes, 1657 us here: exponents 50, residues 230, products 1154 (1.9 PFLOP/s of
// BF16, the rate of a plain library product), reconstruction 149.  Error against the exact product: that of one rounding.
#include <cuda_bf16.h>

#include "tc_common.cuh"

namespace gep {
namespace {

typedef unsigned __int128 u128;

constexpr int NMOD = 16;
constexpr int kMod[NMOD] = {256, 255, 253, 251, 247, 241, 239, 233, 229, 227, 223, 217, 211, 199, 197, 193};

constexpr u128 mod_product() {
  u128 p = 1;
  for (int i = 0; i < NMOD; ++i) p *= (u128)kMod[i];
  return p;
}
constexpr u128 kP = mod_product();
constexpr u128 mod_weight(int i) { return kP / (u128)kMod[i]; }
// (P / m_i)^-1 mod m_i
constexpr int weight_inverse(int i) {
  const int w = (int)(mod_weight(i) % (u128)kMod[i]);
  for (int y = 1; y < kMod[i]; ++y)
    if (w * y % kMod[i] == 1) return y;
  return 0;
}
constexpr bool weights_ok() {
  for (int i = 0; i < NMOD; ++i)
    if (weight_inverse(i) == 0) return false;
  return true;
}
static_assert(weights_ok(), "moduli must be coprime");
constexpr unsigned pow2_mod(int e, int y, int m) {  // 2^e y mod m
  unsigned r = (unsigned)(y % m);
  for (int i = 0; i < e; ++i) r = r * 2 % (unsigned)m;
  return r;
}
constexpr unsigned byte_coeffs(int first, int y, int m) {  // 2^(8 b) y mod m for bytes first .. first + 3
  unsigned c = 0;
  for (int b = 0; b < 4; ++b) c |= pow2_mod(8 * (first + b), y, m) << (8 * b);
  return c;
}
// ------------------------------------------------------------------ residues of an operand

template <int I>
struct Idx {
  static constexpr int v = I;
};
template <int I, class F>
__device__ __forceinline__ void for_moduli(F&& f) {
  if constexpr (I < NMOD) {
    f(Idx<I>{});
    for_moduli<I + 1>(f);
  }
}

// FP32 pattern (its upper half: BF16) of the balanced residue of y F modulo m_I, from U = F + 2^56:
// the bytes of U times 2^(8b) y mod m_I, at most 2^19 in all, so that the quotient by the rounded-up
// reciprocal is exact.
template <int I, bool WEIGHTED>
__device__ __forceinline__ unsigned residue_bits(unsigned long long U) {
  constexpr int m = kMod[I], y = WEIGHTED ? weight_inverse(I) : 1, half = m / 2;
  constexpr unsigned c_lo = byte_coeffs(0, y, m), c_hi = byte_coeffs(4, y, m);
  constexpr unsigned c0 = (m - pow2_mod(56, y, m)) % m + half;
  constexpr unsigned recip = (unsigned)(((1ull << 32) + m - 1) / m);
  const unsigned v = __dp4a((unsigned)U, c_lo, __dp4a((unsigned)(U >> 32), c_hi, c0));
  const unsigned q = __umulhi(v, recip);
  return f32_bits_of_int((int)(v - q * m), -half);
}

// Largest exponent field of each row of X(r, k), K contiguous (k_res_exp_rows: a warp per row) or rows
// contiguous (k_res_exp_cols: 256 rows and a 64-deep slab a CTA; raw zero on entry).
__global__ void __launch_bounds__(256) k_res_exp_rows(int R, int K, const double* __restrict__ X, long long sr,
                                                      int* __restrict__ raw, const int* st) {
  if (status_bad(st)) return;
  const int r = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (r >= R) return;
  int m = 0;
#pragma unroll 4
  for (int k = lane; k < K; k += 32) m = max(m, exp_field(X[(size_t)r * sr + k]));
  for (int o = 16; o; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
  if (lane == 0) raw[r] = m;
}

__global__ void __launch_bounds__(256) k_res_exp_cols(int R, int K, const double* __restrict__ X, long long sk,
                                                      int* __restrict__ raw, const int* st) {
  if (status_bad(st)) return;
  const int r = blockIdx.x * 256 + threadIdx.x;
  if (r >= R) return;
  const int k0 = blockIdx.y * 64, k1 = min(K, k0 + 64);
  int m = 0;
#pragma unroll 8
  for (int k = k0; k < k1; ++k) m = max(m, exp_field(X[r + k * sk]));
  if (m) atomicMax(raw + r, m);
}

// Residue planes out[i][r][k] (BF16, Kpad a multiple of 64, zero from K on) of the operand X(r, k).
// A CTA takes 32 rows x 64 of K through shared memory; a thread 8 consecutive k of one row, so that
// every plane gets 128-byte row segments.  About 8 integer instructions a residue: 4096 x 4096 takes
// as long as its 40 bytes an element.
template <bool WEIGHTED>
__global__ void __launch_bounds__(256) k_res_split(int R, int K, int Kpad, const double* __restrict__ X, long long sr,
                                                   long long sk, const int* __restrict__ raw,
                                                   unsigned short* __restrict__ out, const int* st) {
  __shared__ double t[32][65];
  if (status_bad(st)) return;
  const int r0 = blockIdx.y * 32, k0 = blockIdx.x * 64;
  if (sk == 1) {
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int idx = threadIdx.x + 256 * u, q = idx >> 6, kk = idx & 63;
      t[q][kk] = r0 + q < R && k0 + kk < K ? X[(size_t)(r0 + q) * sr + k0 + kk] : 0.0;
    }
  } else {
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int idx = threadIdx.x + 256 * u, q = idx & 31, kk = idx >> 5;
      t[q][kk] = r0 + q < R && k0 + kk < K ? X[(size_t)(r0 + q) * sr + (size_t)(k0 + kk) * sk] : 0.0;
    }
  }
  __syncthreads();
  const int q = threadIdx.x >> 3, c8 = (threadIdx.x & 7) * 8, r = r0 + q;
  if (r >= R) return;
  const int e = scale_exp(raw[r], 1);
  unsigned long long U[8];
#pragma unroll
  for (int u = 0; u < 8; ++u) U[u] = (unsigned long long)(to_fixed(t[q][c8 + u], e, 8) + (1ll << 56));
  unsigned short* o = out + (size_t)r * Kpad + k0 + c8;
  const size_t plane = (size_t)R * Kpad;
  for_moduli<0>([&](auto ix) {
    constexpr int I = decltype(ix)::v;
    unsigned f[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) f[u] = residue_bits<I, WEIGHTED>(U[u]);
    uint4 w;
    w.x = __byte_perm(f[0], f[1], 0x7632);
    w.y = __byte_perm(f[2], f[3], 0x7632);
    w.z = __byte_perm(f[4], f[5], 0x7632);
    w.w = __byte_perm(f[6], f[7], 0x7632);
    *reinterpret_cast<uint4*>(o + (size_t)I * plane) = w;
  });
}

// ------------------------------------------------------------------ the products

// A pair of CTAs (two SMs) computes a 256 x 256 tile: each stages 128 rows of A and 128 of the 256 columns
// of B, and the pair's MMA reads B from both.
constexpr int RM = 256, RN = 256, RK = 64, RSTAGES = 6, RCH = 1024;
constexpr int REPI = 16;                      // epilogue warps of a CTA
constexpr int RTHREADS = 64 + 32 * REPI;
constexpr uint32_t RA_BYTES = RM / 2 * RK * 2, RB_BYTES = RN / 2 * RK * 2, RSTAGE_BYTES = RA_BYTES + RB_BYTES;
constexpr size_t RSMEM = (size_t)RSTAGES * RSTAGE_BYTES + 1024;
constexpr int RGROUP = 4;                     // row tiles per group of the tile order

__constant__ float c_mod[NMOD] = {256, 255, 253, 251, 247, 241, 239, 233, 229, 227, 223, 217, 211, 199, 197, 193};

__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}

// Address of the same shared variable in the pair's CTA of this rank.
__device__ __forceinline__ uint32_t pair_addr(uint32_t addr, int rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ uint32_t leader_addr(uint32_t addr) { return pair_addr(addr, 0); }

__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.aligned;\n\tbarrier.cluster.wait.aligned;" ::: "memory");
}

__device__ __forceinline__ void mbar_arrive_cluster(uint32_t bar) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
}

// TMA load into this CTA's shared memory that reports to a barrier of either CTA of the pair
__device__ __forceinline__ void tma_load_3d_pair(uint32_t dst, const CUtensorMap* map, int c0, int c1, int c2,
                                                 uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.cta_group::2.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], "
      "[%1, {%2, %3, %4}], [%5];"
      ::"r"(dst), "l"((unsigned long long)map), "r"(c0), "r"(c1), "r"(c2), "r"(bar)
      : "memory");
}

__device__ __forceinline__ void umma_pair(uint32_t dtmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{ .reg .pred p; setp.ne.b32 p, %4, 0; tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p; }"
      ::"r"(dtmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(acc)
      : "memory");
}

// arrives on the barrier at this offset in both CTAs once the MMAs so far are done
__device__ __forceinline__ void umma_commit_pair(uint32_t bar) {
  asm volatile(
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
      ::"r"(bar), "h"((unsigned short)3)
      : "memory");
}

// A wait for work in flight: a bad status does not cut it short, its limit does.
__device__ __forceinline__ void mbar_wait_bounded(uint32_t bar, uint32_t parity, int* st) {
  unsigned long long t0 = gtimer();
  while (!mbar_try(bar, parity))
    if (gtimer() - t0 > 2000000000ull) {
      atomicExch(st + 1, GEP_ERR_TIMEOUT);
      return;
    }
}

struct ResArgs {
  int m, kpad, gx, gy, ntile;    // ntile: tiles of one modulus that are computed
  int lower, j0;                 // lower: only tiles that reach the diagonal; j0: global column of column 0
  unsigned char* out;            // residues + 128: [NMOD][m][ldr], columns contiguous
  int ldr;
  int* st;
};

// Tile t of a modulus.  Full: groups of RGROUP row tiles, row fastest (its A and B planes are then
// shared in L2 by the tiles that run together).  Lower: column after column, from the diagonal down.
__device__ __forceinline__ void res_tile(const ResArgs& p, int t, int& tm, int& tn) {
  if (p.lower) {
    for (int c = 0;; ++c) {
      const int r0 = (p.j0 + c * RN) / RM, cnt = p.gx - r0;
      if (t < cnt || c == p.gy - 1) {
        tm = (r0 + t) * RM;
        tn = c * RN;
        return;
      }
      t -= max(cnt, 0);
    }
  }
  const int per_group = RGROUP * p.gy, first = t / per_group * RGROUP, gm = min(p.gx - first, RGROUP);
  const int local = t - first / RGROUP * per_group;
  tm = (first + local % gm) * RM;
  tn = local / gm * RN;
}

// One item per modulus and tile, modulus slowest; pair c takes the items c, c + pairs, ....  In each CTA warp 0
// loads 64-deep steps of its halves (TMA, 128-byte swizzle, ring of six; both CTAs' copies report to the
// first CTA's barrier), warp 1 of the first CTA issues the MMAs (256 x 256 x 16) into one of two TMEM
// buffers, a chunk of 1024 each, and 16 warps of each CTA reduce the other buffer modulo m_i meanwhile
// (four instructions an element and chunk; reduced fully and packed after every chunk they slowed the
// MMAs: 16 x 4096 x 2048 x 2048 380 us, now 307).  The pair halves the shared-memory traffic of B, which bounds one
// CTA with 128 x 256 tiles.  Waits are bounded as in k_oz_gemm; the CTAs of a pair may give up at different
// steps, so before they retire each learns how many steps the other has loaded and both are brought level.
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(RTHREADS, 1)
    k_res_gemm(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, ResArgs p) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  __shared__ __align__(8) unsigned long long bars[2 * RSTAGES + 5];
  __shared__ uint32_t tmem_slot;
  __shared__ int skip, issued;  // issued: steps whose copies this CTA has started
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rank = (int)cluster_rank(), pair = blockIdx.x >> 1, npairs = gridDim.x >> 1;
  unsigned char* smem = (unsigned char*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  const uint32_t bar_full = smem_u32(&bars[0]), bar_empty = smem_u32(&bars[RSTAGES]);
  const uint32_t bar_accf = smem_u32(&bars[2 * RSTAGES]), bar_acce = smem_u32(&bars[2 * RSTAGES + 2]);
  const uint32_t bar_done = smem_u32(&bars[2 * RSTAGES + 4]);
  const int nsteps = p.kpad / RK, nch = (p.kpad + RCH - 1) / RCH;
  constexpr int SPC = RCH / RK;

  if (threadIdx.x == 0) {
    skip = status_bad(p.st) ? 1 : 0;
    issued = 0;
    for (int s = 0; s < RSTAGES; ++s) {
      mbar_init(bar_full + 8 * s, 1);
      mbar_init(bar_empty + 8 * s, 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(bar_accf + 8 * b, 1);
      mbar_init(bar_acce + 8 * b, 2 * REPI);
    }
    mbar_init(bar_done, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    prefetch_map(&tmA);
    prefetch_map(&tmB);
  }
  __syncthreads();
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(&tmem_slot))
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();  // the other CTA's barriers are initialised, its TMEM is allocated
  tc_fence_after();
  const uint32_t tmem = tmem_slot;
  int pair_skip;  // the first CTA's view of the status decides for the pair
  asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(pair_skip) : "r"(leader_addr(smem_u32(&skip))) : "memory");
  const int nitems = pair_skip ? 0 : NMOD * p.ntile;

  if (warp == 0) {
    if (lane == 0) {
      int g = 0;
      bool ok = true;
      for (int w = pair; ok && w < nitems; w += npairs) {
        const int md = w / p.ntile;
        int tm, tn;
        res_tile(p, w - md * p.ntile, tm, tn);
        for (int step = 0; step < nsteps; ++step, ++g) {
          const int sidx = g % RSTAGES;
          ok = mbar_wait(bar_empty + 8 * sidx, ((uint32_t)(g / RSTAGES) & 1u) ^ 1u, p.st);
          if (!ok) break;
          const uint32_t dst = smem_u32(smem + (size_t)sidx * RSTAGE_BYTES);
          const uint32_t full = leader_addr(bar_full + 8 * sidx);
          if (rank == 0) mbar_expect_tx(bar_full + 8 * sidx, 2 * RSTAGE_BYTES);
          tma_load_3d_pair(dst, &tmA, step * RK, tm + rank * (RM / 2), md, full);
          tma_load_3d_pair(dst + RA_BYTES, &tmB, step * RK, tn + rank * (RN / 2), md, full);
        }
      }
      issued = g;
    }
  } else if (warp == 1) {
    if (lane == 0 && rank == 0) {
      const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(RN >> 3) << 17) | ((uint32_t)(RM >> 4) << 24);
      bool ok = true;
      int g = 0, gc = 0;
      for (int w = pair; ok && w < nitems; w += npairs) {
        for (int c = 0, step = 0; c < nch; ++c, ++gc) {
          const int buf = gc & 1;
          ok = mbar_wait(bar_acce + 8 * buf, ((uint32_t)(gc >> 1) & 1u) ^ 1u, p.st);
          if (!ok) break;
          tc_fence_after();
          const int send = min(nsteps, step + SPC);
          for (int sic = 0; step < send; ++step, ++sic, ++g) {
            const int sidx = g % RSTAGES;
            ok = mbar_wait(bar_full + 8 * sidx, (uint32_t)(g / RSTAGES) & 1u, p.st);
            if (!ok) break;
            tc_fence_after();
            const uint32_t abase = smem_u32(smem + (size_t)sidx * RSTAGE_BYTES);
            const uint64_t a0 = sdesc_sw128(abase), b0 = sdesc_sw128(abase + RA_BYTES);
#pragma unroll
            for (int kk = 0; kk < RK / 16; ++kk)
              umma_pair(tmem + (uint32_t)(buf * RN), a0 + (uint64_t)(kk * 2), b0 + (uint64_t)(kk * 2), idesc,
                        (sic | kk) ? 1u : 0u);
            umma_commit_pair(bar_empty + 8 * sidx);
          }
          if (!ok) break;
          umma_commit_pair(bar_accf + 8 * buf);
        }
      }
      umma_commit_pair(bar_done);
      mbar_wait_bounded(bar_done, 0, p.st);
    }
  } else {
    // warp w reads TMEM lanes 32 (w % 4) .., columns 64 ((w - 2) / 4) ..
    const int q = warp & 3, cg = (warp - 2) >> 2;
    bool ok = true;
    int gc = 0;
    for (int w = pair; ok && w < nitems; w += npairs) {
      const int md = w / p.ntile;
      int tm, tn;
      res_tile(p, w - md * p.ntile, tm, tn);
      const float m = c_mod[md], inv = 1.0f / m;
      float acc[64];  // sums of the chunks' residues
#pragma unroll
      for (int j = 0; j < 64; ++j) acc[j] = 0.0f;
      for (int c = 0; c < nch; ++c, ++gc) {
        const int buf = gc & 1;
        ok = mbar_wait(bar_accf + 8 * buf, (uint32_t)(gc >> 1) & 1u, p.st);
        if (!ok) break;
        tc_fence_after();
        const uint32_t ta = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(buf * RN + cg * 64);
#pragma unroll
        for (int sl = 0; sl < 4; ++sl) {
          float v[16];
          tmem_ld16(ta + 16 * sl, v);
          // v (|v| <= 2^24, exact) - m rint(v / m): at most m / 2 + 2
#pragma unroll
          for (int j = 0; j < 16; ++j)
            acc[16 * sl + j] += fmaf(-(fmaf(v[j], inv, 12582912.0f) - 12582912.0f), m, v[j]);
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive_cluster(leader_addr(bar_acce + 8 * buf));
      }
      if (!ok) break;
      const int row = tm + rank * (RM / 2) + q * 32 + lane;
      if (row < p.m) {
        uint4* o = reinterpret_cast<uint4*>(p.out + ((size_t)md * p.m + row) * p.ldr + tn + cg * 64);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          unsigned w[4];
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            unsigned f[4];
#pragma unroll
            for (int x = 0; x < 4; ++x) {
              const float a = acc[16 * j + 4 * u + x];
              // 1.5 2^23 + 128 + residue: the low byte is the residue + 128 (256 wraps to the residue -128)
              f[x] = __float_as_uint(fmaf(-(fmaf(a, inv, 12582912.0f) - 12582912.0f), m, a) + 12583040.0f);
            }
            w[u] = __byte_perm(__byte_perm(f[0], f[1], 0x0040), __byte_perm(f[2], f[3], 0x0040), 0x5410);
          }
          o[j] = make_uint4(w[0], w[1], w[2], w[3]);
        }
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();  // both counts stand, and no MMA reads the stages any more
  // Every copy lands before the CTAs retire.  A step's barrier (the first CTA's) completes with the copies
  // of both: where one CTA gave up earlier, the second loads what it is behind (its stages are free), the
  // first expects what the second is ahead.
  if (threadIdx.x == 0) {
    const int mine = issued;
    int other;
    asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(other) : "r"(pair_addr(smem_u32(&issued), rank ^ 1)) : "memory");
    if (rank == 1) {
      for (int s = mine; s < other; ++s) {
        const uint32_t dst = smem_u32(smem + (size_t)(s % RSTAGES) * RSTAGE_BYTES);
        const uint32_t full = leader_addr(bar_full + 8 * (s % RSTAGES));
        tma_load_3d_pair(dst, &tmA, 0, 0, 0, full);
        tma_load_3d_pair(dst + RA_BYTES, &tmB, 0, 0, 0, full);
      }
    } else {
      for (int s = max(mine - RSTAGES, 0); s < max(mine, other); ++s) {
        if (s >= mine) mbar_expect_tx(bar_full + 8 * (s % RSTAGES), RSTAGE_BYTES);
        mbar_wait_bounded(bar_full + 8 * (s % RSTAGES), (uint32_t)(s / RSTAGES) & 1u, p.st);
      }
    }
  }
  __syncthreads();
  cluster_sync_all();  // no copy, MMA or arrival of the pair is in flight any more
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, 512;" ::"r"(tmem) : "memory");
  }
}

// ------------------------------------------------------------------ reconstruction

struct CrtArgs {
  int m, n, lower, j0, ldr, ldc, amode, bmode;
  const unsigned char* res;  // [NMOD][m][ldr]
  const int *ea, *eb;
  double alpha, beta;
  double* C;                 // column j0 of C
  int* st;
};

// Byte b of the weights of moduli 4 g .. 4 g + 3.
constexpr unsigned weight_bytes(int g, int b) {
  unsigned c = 0;
  for (int i = 0; i < 4; ++i) c |= (unsigned)((mod_weight(4 * g + i) >> (8 * b)) & 255) << (8 * i);
  return c;
}
// The biased bytes add 128 sum_i P / m_i, here modulo P.
constexpr u128 bias_mod_p() {
  u128 s = 0;
  for (int i = 0; i < NMOD; ++i) s = (s + mod_weight(i)) % kP;
  for (int i = 0; i < 7; ++i) s = s * 2 % kP;
  return s;
}
constexpr u128 kBias = bias_mod_p();

template <int B>
__device__ __forceinline__ unsigned weight_sum(const unsigned (&t)[4]) {
  constexpr unsigned w0 = weight_bytes(0, B), w1 = weight_bytes(1, B), w2 = weight_bytes(2, B), w3 = weight_bytes(3, B);
  return __dp4a(t[0], w0, __dp4a(t[1], w1, __dp4a(t[2], w2, __dp4a(t[3], w3, 0u))));
}

// Word B .. B + 3 of the sum of the weights: four byte sums of at most 2^20.
template <int B>
__device__ __forceinline__ unsigned long long weight_word(const unsigned (&t)[4]) {
  const unsigned lo = weight_sum<B>(t) + (weight_sum<B + 1>(t) << 8);
  unsigned hi = weight_sum<B + 2>(t);
  if constexpr (B + 3 < 15) hi += weight_sum<B + 3>(t) << 8;  // the weights have 118 bits
  return (unsigned long long)lo + ((unsigned long long)hi << 16);
}

// A CTA takes 32 rows x 32 columns: a thread four columns of a row (one word of every plane, 32-byte row
// segments), transposed by bytes into four moduli a word, so that byte b of sum_i t_i P / m_i is
// four 4-way byte products.  The doubles go through shared memory, since C runs down the columns.
// Bound: the integer work, about 330 issue slots an element (4096 x 4096 149 us; with 64 64-bit
// multiply-adds an element 194 us).
__global__ void __launch_bounds__(256) k_res_crt(CrtArgs p) {
  __shared__ double tile[32][33];
  if (status_bad(p.st)) return;
  const int r0 = blockIdx.y * 32, c0 = blockIdx.x * 32;
  if (p.lower && r0 + 31 < p.j0 + c0) return;
  {
    const int i = threadIdx.x >> 3, j4 = (threadIdx.x & 7) * 4, row = min(r0 + i, p.m - 1);
    const unsigned char* r = p.res + (size_t)row * p.ldr + c0 + j4;
    const size_t plane = (size_t)p.m * p.ldr;
    unsigned t[4][4];  // [column][moduli 4 g ..]
#pragma unroll
    for (int g = 0; g < 4; ++g) {
      unsigned x[4];
#pragma unroll
      for (int i4 = 0; i4 < 4; ++i4) x[i4] = *reinterpret_cast<const unsigned*>(r + (4 * g + i4) * plane);
      const unsigned a = __byte_perm(x[0], x[1], 0x5140), b = __byte_perm(x[2], x[3], 0x5140);
      const unsigned c = __byte_perm(x[0], x[1], 0x7362), d = __byte_perm(x[2], x[3], 0x7362);
      t[0][g] = __byte_perm(a, b, 0x5410);
      t[1][g] = __byte_perm(a, b, 0x7632);
      t[2][g] = __byte_perm(c, d, 0x5410);
      t[3][g] = __byte_perm(c, d, 0x7632);
    }
    const int ra = p.ea[row], ea = scale_exp(ra, 1) - 112 + 127;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const unsigned long long w0 = weight_word<0>(t[u]), w1 = weight_word<4>(t[u]) + (w0 >> 32),
                               w2 = weight_word<8>(t[u]) + (w1 >> 32), w3 = weight_word<12>(t[u]) + (w2 >> 32);
      const u128 sum = (u128)((w0 & 0xffffffffull) | (w1 << 32)) | (u128)((w2 & 0xffffffffull) | (w3 << 32)) << 64;
      // (sum - bias) / P is within 0.1 of an integer; the top word gives it to 2^-19
      constexpr float scale = (float)((double)(1ull << 40) / (double)(unsigned long long)(kP >> 64));  // 2^104 / P
      constexpr float shift = (float)((double)(unsigned long long)(kBias >> 64) / (double)(unsigned long long)(kP >> 64));
      const int q = __float2int_rn(fmaf((float)(unsigned)(w3 >> 8), scale, -shift));
      const u128 X = sum - kBias - (u128)(unsigned)q * kP;  // modulo 2^128, signed
      const int rb = p.eb[min(c0 + j4 + u, p.n - 1)];
      tile[j4 + u][i] = __longlong_as_double(
          nonfinite(ra, rb) ? NAN_BITS : fixed128_to_bits((long long)(unsigned long long)(X >> 64), (unsigned long long)X,
                                                          ea + scale_exp(rb, 1)));
    }
  }
  __syncthreads();
  const int i = r0 + (threadIdx.x & 31);
  if (i >= p.m) return;
  const long long flip = p.amode < 0 ? 1ll << 63 : 0ll;
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int jl = (threadIdx.x >> 5) + 8 * u, j = c0 + jl;
    if (j >= p.n || (p.lower && i < p.j0 + j)) continue;
    double out = __longlong_as_double(__double_as_longlong(tile[jl][threadIdx.x & 31]) ^ flip);
    double* c = p.C + (size_t)j * p.ldc + i;
    if (p.amode == 0) out *= p.alpha;
    if (p.bmode == 1) out += *c;
    else if (p.bmode == 2) out = fma(p.beta, *c, out);
    *c = out;
  }
}

// ------------------------------------------------------------------ host

int encode_res_map(CUtensorMap* map, const void* base, int kpad, int rows, int box_rows) {
  cuuint64_t dims[3] = {(cuuint64_t)kpad, (cuuint64_t)rows, (cuuint64_t)NMOD};
  cuuint64_t strides[2] = {(cuuint64_t)kpad * 2, (cuuint64_t)kpad * 2 * (cuuint64_t)rows};
  cuuint32_t box[3] = {(cuuint32_t)RK, (cuuint32_t)box_rows, 1};
  cuuint32_t estr[3] = {1, 1, 1};
  EncodeTiledFn enc = encode_fn();
  if (!enc) {
    fprintf(stderr, "gep: cuTensorMapEncodeTiled not available from the driver\n");
    return GEP_ERR_CUDA;
  }
  CUresult r = enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box, estr,
                   CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) {
    fprintf(stderr, "gep: cuTensorMapEncodeTiled failed (%d)\n", (int)r);
    return GEP_ERR_CUDA;
  }
  return GEP_OK;
}

int split_operand(gep_handle_t h, bool weighted, int R, int K, int Kpad, const double* X, long long sr, long long sk,
                  int* raw, unsigned short* out) {
  if (sk == 1) {
    k_res_exp_rows<<<(R * 32 + 255) / 256, 256, 0, h->stream>>>(R, K, X, sr, raw, h->d_status);
  } else {
    GEP_CUDA(cudaMemsetAsync(raw, 0, sizeof(int) * (size_t)R, h->stream));
    k_res_exp_cols<<<dim3((R + 255) / 256, (K + 63) / 64), 256, 0, h->stream>>>(R, K, X, sk, raw, h->d_status);
  }
  GEP_CHECK(check_launch(h));
  const dim3 grid(Kpad / 64, (R + 31) / 32);
  if (weighted) k_res_split<true><<<grid, 256, 0, h->stream>>>(R, K, Kpad, X, sr, sk, raw, out, h->d_status);
  else k_res_split<false><<<grid, 256, 0, h->stream>>>(R, K, Kpad, X, sr, sk, raw, out, h->d_status);
  return check_launch(h);
}

constexpr int RKP_MAX = 4096;  // K panel

// K panel and column block that fit the scratch: planes of m rows and nb columns and the bytes of
// m x nb outputs.  The panel is halved before the block gets narrower than a quarter of it.
struct ResPlan {
  int kp = 0, nb = 0;
};
size_t res_bytes(int m, int nb, int kp) {
  const size_t ldr = (size_t)(nb + RN - 1) / RN * RN;
  return align256((size_t)2 * NMOD * m * kp) + align256((size_t)2 * NMOD * nb * kp) +
         align256((size_t)NMOD * ldr * m) + align256(sizeof(int) * (size_t)m) + align256(sizeof(int) * (size_t)nb);
}
ResPlan res_plan(int m, int n, int k, size_t cap) {
  ResPlan r;
  for (int kp = (min(k, RKP_MAX) + RK - 1) / RK * RK;; kp = (kp / 2 + RK - 1) / RK * RK) {
    if (kp < 512) return ResPlan();
    int nb = min((n + RN - 1) / RN * RN, 1 << 15);
    while (nb > RN && res_bytes(m, nb, kp) > cap) nb -= RN;
    if (nb >= n || nb >= 1024) {
      if (res_bytes(m, min(nb, n), kp) > cap) continue;
      r.kp = kp;
      r.nb = nb;
      return r;
    }
  }
}

// Whether the rx x cx matrix X and the rc x cc matrix C share an element (blocks of one array: exactly;
// different leading dimensions: whether their address ranges meet).  Products in place keep the digit
// planes, which read all of an operand before the first write of C.
bool overlap(const double* X, int ldx, int rx, int cx, const double* C, int ldc, int rc, int cc) {
  if (ldx != ldc) return X < C + (size_t)cc * ldc && C < X + (size_t)cx * ldx;
  const long long d = C - X;
  long long dc = d / ldc, dr = d % ldc;
  if (dr < 0) { dr += ldc; --dc; }
  for (int s = 0; s < 2; ++s, dr -= ldc, ++dc)
    if (dr < rx && dr + rc > 0 && dc < cx && dc + cc > 0) return true;
  return false;
}

}  // namespace

// The faster of the two forms of a product on the tensor cores, by their measured costs (us):
//   digit planes:  10 and 30 a K panel for launches and splits, 4 a panel + 0.05 k per wave of 128 x 64
//                  tiles, the operands' digits;
//   residues:      15, 10 a K panel and 35 for each of its column blocks, 0.0051 k per wave of (256 x 256 tile,
//                  modulus) on the pairs of CTAs, 9 ps an operand element (its 40 bytes) and 13 ps an output and
//                  K panel (16 bytes in, C, the CRT).
// Both by the K panels and column blocks that the scratch allows.  Fitted to 40 shapes and scratches, within a tenth:
// 1024 x 1024 x 4096 with 64 / 128 / 256 / 512 MB: digits 339 / 323 / 282 us, residues 615 / 393 / 279 / 225;
// 4096^3 with 256 MB 3414 / 2883, 3000 x 3000 x 9000 with 128 / 256 MB 4391 / 6017 and 4290 / 3634.
// Digits / residues: 512^3 76 / 74, 1024 x 1024 x 512 77 / 97, 4096 x 256 x 1024 133 / 146,
// 4096 x 4096 x 512 476 / 471, 1024^3 120 / 120, 8192 x 512 x 1024 322 / 260, 2048^3 510 / 328, 256 x 256 x 4096
// 267 / 110, 4096^3 3130 / 1657, lower triangle 8192 x 8192 x 2048 3674 / 2026.
bool res_product_wins(gep_handle_t h, char uplo, int m, int n, int k) {
  if (k < 512) return false;
  const bool lower = uplo == 'L' || uplo == 'l';
  const double half = lower ? 0.5 : 1.0, mn = half * m * n, op = ((double)m + n) * k;
  const double digit_tiles = half * ((m + 127) / 128) * ((n + 63) / 64);
  double res_tiles = (double)((m + RM - 1) / RM) * ((n + RN - 1) / RN);
  if (lower) res_tiles = 0.5 * (res_tiles + (n + RN - 1) / RN);
  const ResPlan pl = res_plan(m, n, k, h->eng_ws ? h->eng_bytes : 0);
  if (pl.kp == 0) return false;
  const double panels = (k + pl.kp - 1) / pl.kp, blocks = (n + pl.nb - 1) / pl.nb;
  const double digit_k = fmin(RKP_MAX, (h->eng_bytes - 1024.0) / (16.0 * ((double)m + n))), digit_panels = ceil(k / digit_k);
  const double digits = 10.0 + 30.0 * digit_panels +
                        ceil(digit_tiles / h->sm_count) * (4.0 * digit_panels + 0.05 * k) + 5e-6 * op;
  const double residues = 15.0 + panels * (10.0 + 35.0 * blocks) +
                          blocks * ceil(NMOD * res_tiles / blocks / (h->sm_count / 2)) * 0.0051 * k + 9e-6 * op +
                          13e-6 * mn * panels;
  return residues < 0.97 * digits;
}

// Scratch that lets the residue products run in K panels of RKP_MAX and column blocks of 2048.
size_t res_workspace_bytes(int m, int n, int k) {
  const int kp = (min(k, RKP_MAX) + RK - 1) / RK * RK;
  return res_bytes(m, min((n + RN - 1) / RN * RN, 2048), kp);
}

int dgemm_res(gep_handle_t h, char ta, char tb, char uplo, int m, int n, int k, double alpha, const double* A, int lda,
              const double* B, int ldb, double beta, double* C, int ldc) {
  const bool TA = (ta == 'T' || ta == 't'), TB = (tb == 'T' || tb == 't'), lower = uplo == 'L' || uplo == 'l';
  const long long sra = TA ? lda : 1, ska = TA ? 1 : lda, srb = TB ? 1 : ldb, skb = TB ? ldb : 1;
  const ResPlan pl = res_plan(m, n, k, h->eng_ws ? h->eng_bytes : 0);
  if (pl.kp == 0) return GEP_ERR_ALLOC;
  // C <- C + A C: in one K panel, a column block of B is split before its block of C is written
  const bool in_place = B == C && ldb == ldc && !TB && m == k && pl.kp >= k;
  if (overlap(A, lda, TA ? k : m, TA ? m : k, C, ldc, m, n) ||
      (!in_place && overlap(B, ldb, TB ? n : k, TB ? k : n, C, ldc, m, n)))
    return GEP_ERR_UNSUPPORTED;
  static DeviceOnce attributes;
  GEP_CHECK(once_per_device(attributes, []() -> int {
    GEP_CUDA(cudaFuncSetAttribute(k_res_gemm, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)RSMEM));
    return GEP_OK;
  }));
  const int nbw = min(pl.nb, n), ldr = (nbw + RN - 1) / RN * RN;
  char* p = h->eng_ws;
  unsigned short* As = (unsigned short*)p;
  p += align256((size_t)2 * NMOD * m * pl.kp);
  unsigned short* Bs = (unsigned short*)p;
  p += align256((size_t)2 * NMOD * nbw * pl.kp);
  unsigned char* res = (unsigned char*)p;
  p += align256((size_t)NMOD * ldr * m);
  int* ea = (int*)p;
  p += align256(sizeof(int) * (size_t)m);
  int* eb = (int*)p;
  for (int kb = 0; kb < k; kb += pl.kp) {
    const int kc = min(pl.kp, k - kb), kpad = (kc + RK - 1) / RK * RK;
    GEP_CHECK(split_operand(h, false, m, kc, kpad, A + (size_t)kb * ska, sra, ska, ea, As));
    CUtensorMap mA, mB;
    GEP_CHECK(encode_res_map(&mA, As, kpad, m, RM / 2));
    for (int j0 = 0; j0 < n; j0 += pl.nb) {
      const int nb = min(pl.nb, n - j0);
      if (lower && j0 >= m) break;
      GEP_CHECK(split_operand(h, true, nb, kc, kpad, B + (size_t)kb * skb + (size_t)j0 * srb, srb, skb, eb, Bs));
      GEP_CHECK(encode_res_map(&mB, Bs, kpad, nb, RN / 2));
      ResArgs a;
      a.m = m; a.kpad = kpad; a.lower = lower; a.j0 = j0; a.out = res; a.ldr = ldr; a.st = h->d_status;
      a.gx = (m + RM - 1) / RM;
      a.gy = (nb + RN - 1) / RN;
      a.ntile = a.gx * a.gy;
      if (lower) {
        a.ntile = 0;
        for (int c = 0; c < a.gy; ++c) a.ntile += max(0, a.gx - (j0 + c * RN) / RM);
      }
      int slot = -1;
      if (h->prof_on) {
        if (h->prof_used < h->prof_cap) {
          slot = h->prof_used++;
          cudaEventRecord(h->prof_ev[2 * slot], h->stream);
          const double f = 2.0 * m * nb * (double)kc * (lower ? 0.5 : 1.0);
          h->prof_f64eq[slot] = f;
          h->prof_flops[slot] = f * NMOD;
          h->prof_mnk[3 * slot] = m;
          h->prof_mnk[3 * slot + 1] = nb;
          h->prof_mnk[3 * slot + 2] = kc;
        } else {
          h->prof_skipped++;
        }
      }
      k_res_gemm<<<2 * min(NMOD * a.ntile, h->sm_count / 2), RTHREADS, RSMEM, h->stream>>>(mA, mB, a);
      GEP_CHECK(check_launch(h));
      if (slot >= 0) cudaEventRecord(h->prof_ev[2 * slot + 1], h->stream);
      CrtArgs c;
      c.m = m; c.n = nb; c.lower = lower; c.j0 = j0; c.ldr = ldr; c.ldc = ldc; c.res = res; c.ea = ea; c.eb = eb;
      c.alpha = alpha; c.beta = kb == 0 ? beta : 1.0; c.C = C + (size_t)j0 * ldc; c.st = h->d_status;
      c.amode = alpha == 1.0 ? 1 : alpha == -1.0 ? -1 : 0;
      c.bmode = c.beta == 0.0 ? 0 : c.beta == 1.0 ? 1 : 2;
      k_res_crt<<<dim3((nb + 31) / 32, (m + 31) / 32), 256, 0, h->stream>>>(c);
      GEP_CHECK(check_launch(h));
    }
  }
  return GEP_OK;
}

}  // namespace gep
