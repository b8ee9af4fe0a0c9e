// Device helpers of the tensor-core kernels: mbarriers, TMA loads, tcgen05 (TMEM allocation, loads, MMA), digit
// splitting and the integer conversions of exact digit sums.
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cstdint>

namespace librpa {
namespace {

// ------------------------------------------------------------------ digits

__device__ __forceinline__ int biased_exp(double v) { return (int)((__double_as_longlong(v) >> 52) & 0x7FF); }

// v 2^e, exact while the result is a normal number (integer instructions; else through FP64)
__device__ __forceinline__ double scale_pow2(double v, int e) {
  const int ex = biased_exp(v);
  if (ex > 0 && ex < 2047 && (unsigned)(ex + e - 1) < 2046u)
    return __longlong_as_double(__double_as_longlong(v) + ((long long)e << 52));
  return (__double_as_longlong(v) << 1) == 0 ? v : scalbn(v, e);
}

// balanced base-256 digits of x = v 2^-E (|x| < 1): x ~ sum_s d_s 2^{-7-8(s-1)}, |d_s| <= 128, as FP32 integers.
// W = x 2^{7+8(S-1)} rounded (half up in magnitude); with 128 added at every lower digit's place the digits are the
// bytes of the sum less 128, and a byte b becomes a float by the bits of 2^23 + b.
template <int S>
__device__ __forceinline__ void make_digits(double v, int E, float (&d)[S]) {
  const long long bits = __double_as_longlong(v);
  const int ex = (int)((bits >> 52) & 0x7FF);
  const int r = 1075 + E - 7 - 8 * (S - 1) - ex;   // |W| = mant 2^-r
  const unsigned long long mant = ((unsigned long long)bits & 0xFFFFFFFFFFFFFull) | (1ull << 52);
  unsigned long long u;
  if (S < 7)   // r > 0 since |x| < 1
    u = ((mant >> (r - 1 & 63)) + 1) >> 1;
  else   // r >= -10
    u = r + 10 == 0 ? mant << 10 : (((mant << 10) >> (r + 9 & 63)) + 1) >> 1;
  if (ex == 0 || r > 53) u = 0;   // zero (subnormals are far below any row scale of interest), or below half a unit
  long long W = bits < 0 ? -(long long)u : (long long)u;
  unsigned lo, hi = 0;
  int top;
  if constexpr (S <= 5) {   // |W| < 2^40
    constexpr unsigned long long kBias = S == 1 ? 0ull : 0x80808080ull >> (8 * (5 - S));
    W += (long long)kBias;
    lo = (unsigned)(unsigned long long)W;
    top = (int)(W >> (8 * (S - 1)));
  } else {   // the lower digits apart, so that the sum of W near 2^63 does not overflow
    static_assert(S <= 5 || S == 8, "make_digits: planes");
    const unsigned long long l = ((unsigned long long)W & 0xFFFFFFFFFFFFFFull) + 0x80808080808080ull;
    lo = (unsigned)l;
    hi = (unsigned)(l >> 32);
    top = (int)(W >> 56) + (int)(l >> 56);
  }
  d[0] = __int_as_float(top + 0x4B400000) - 12582912.f;
#pragma unroll
  for (int s = 1; s < S; ++s) {
    const int byte = S - 1 - s;   // place of digit s
    d[s] = __uint_as_float(__byte_perm(byte < 4 ? lo : hi, 0x4B000000u, 0x7440 + (byte & 3))) - 8388736.f;
  }
}

__device__ __forceinline__ unsigned pack_bf16(float a, float b) {
  __nv_bfloat162 v = __floats2bfloat162_rn(a, b);   // small integers: exact
  return *reinterpret_cast<unsigned *>(&v);
}

// ------------------------------------------------------------------ tcgen05 / TMA / mbarrier

constexpr uint64_t WAIT_NS = 2000000000ull;   // 2 s

// one lane of a converged warp (the compiler then knows that a single thread issues the TMA copies and MMAs)
__device__ __forceinline__ bool elect_one() {
  uint32_t p;
  asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}\n" : "=r"(p));
  return p != 0;
}

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void prefetch_l1(const void *p) { asm volatile("prefetch.global.L1 [%0];" ::"l"(p)); }

__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t *bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ uint64_t global_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
// bounded wait: false after ~limit_ns, or as soon as *abort is set (abort may be NULL: the
// waits that drain a CTA's own copies and MMAs before it exits never give up early)
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, uint32_t parity, uint64_t limit_ns,
                                          const volatile int *abort = nullptr) {
  if (mbar_try_wait(bar, parity)) return true;
  const uint64_t t0 = global_ns();
  while (true) {
    if (mbar_try_wait(bar, parity)) return true;
    if (abort && *abort) return false;
    if (global_ns() - t0 > limit_ns) return false;
  }
}

__device__ __forceinline__ void tma_load_3d(void *dst, const CUtensorMap *map, uint64_t *bar, int x, int y, int z) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
      ::"r"(smem_u32(dst)), "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z), "r"(smem_u32(bar))
      : "memory");
}

__device__ __forceinline__ void tma_load_4d(void *dst, const CUtensorMap *map, uint64_t *bar, int x, int y, int z, int w) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], [%6];"
      ::"r"(smem_u32(dst)), "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z), "r"(w), "r"(smem_u32(bar))
      : "memory");
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

__device__ __forceinline__ void tmem_alloc(uint32_t *slot, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(slot)), "r"(ncols)
               : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}


// instruction descriptor: D = F32, A and B K-major, M = 128, N = n; A/B format 1 = BF16 (kind::f16)
// or 2 = TF32 (kind::tf32)
__host__ __device__ constexpr uint32_t idesc(uint32_t n, bool tf32) {
  return (1u << 4) | ((tf32 ? 2u : 1u) << 7) | ((tf32 ? 2u : 1u) << 10) | ((n >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
}

__device__ __forceinline__ void umma(uint32_t d, uint64_t a, uint64_t b, uint32_t desc, uint32_t acc) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n"
      ::"r"(d), "l"(a), "l"(b), "r"(desc), "r"(acc)
      : "memory");
}
// the same, always adding to the accumulator
__device__ __forceinline__ void umma_add(uint32_t d, uint64_t a, uint64_t b, uint32_t desc) {
  asm volatile("{\n .reg .pred p;\n setp.eq.u32 p, 0, 0;\n tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n"
               ::"r"(d), "l"(a), "l"(b), "r"(desc)
               : "memory");
}
__device__ __forceinline__ void umma_tf32(uint32_t d, uint64_t a, uint64_t b, uint32_t desc, uint32_t acc) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n}\n"
      ::"r"(d), "l"(a), "l"(b), "r"(desc), "r"(acc)
      : "memory");
}
__device__ __forceinline__ void umma_commit(uint64_t *bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
               : "memory");
}
// 4, 8, 12 or 16 columns of the warp's 32 TMEM lanes; the registers are valid after tmem_ld_wait on them
__device__ __forceinline__ void tmem_ld4(uint32_t taddr, uint32_t *r) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(taddr));
}
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t *r) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr));
}
template <int N>
__device__ __forceinline__ void tmem_ld(uint32_t taddr, uint32_t (&r)[N]) {
  static_assert(N == 4 || N == 8 || N == 12 || N == 16, "tmem_ld: columns");
  if constexpr (N >= 8) tmem_ld8(taddr, r);
  if constexpr (N == 16) tmem_ld8(taddr + 8, r + 8);
  if constexpr (N == 12) tmem_ld4(taddr + 8, r + 8);
  if constexpr (N == 4) tmem_ld4(taddr, r);
}
template <int N>
__device__ __forceinline__ void tmem_ld_wait(uint32_t (&r)[N]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int j = 0; j < N; ++j) asm volatile("" : "+r"(r[j]));   // no use of r[j] moves above the wait
}

// shared-memory matrix descriptor: K-major, 64-byte swizzle, 8-row groups `sbo` bytes apart
__device__ __forceinline__ uint64_t smem_desc64(uint32_t saddr, uint32_t sbo = 512) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFF) >> 4);
  d |= (uint64_t)(16 >> 4) << 16;     // leading byte offset (unused for swizzled K-major)
  d |= (uint64_t)(sbo >> 4) << 32;    // stride byte offset
  d |= (uint64_t)1 << 46;             // descriptor version
  d |= (uint64_t)4 << 61;             // SWIZZLE_64B
  return d;
}

// the same with 128-byte swizzle (8-row groups of 1024 bytes)
__device__ __forceinline__ uint64_t smem_desc128(uint32_t saddr) {
  return (uint64_t)((saddr & 0x3FFFF) >> 4) | (uint64_t)1 << 16 | (uint64_t)(1024 >> 4) << 32 | (uint64_t)1 << 46 |
         (uint64_t)2 << 61;
}

__device__ __forceinline__ void mbar_arrive(uint64_t *bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

// ------------------------------------------------------------------ epilogue conversions
// The FP64 pipe of GB300 runs at about 1/64 of its FP32 rate, so the epilogue builds its FP64 (and
// FP32-pair) outputs from the exact integer digit sums with integer instructions: normalise by the
// leading-one position, round to nearest even, and put the scale 2^sh into the exponent field.
// Straight-line but for results outside the normal range (rare), so that a thread's sums interleave.

// mant (53 bits, or 2^53 after rounding up) 2^(e - 1075) with e the biased exponent; neg: sign bit
__device__ __forceinline__ double make_f64(unsigned long long neg, unsigned long long mant, int e) {
  double v = __longlong_as_double((long long)(((unsigned long long)(e - 1) << 52) + mant));
  if ((unsigned)(e - 1) >= 2045u) {   // subnormal, overflow or next to it: scale [1, 2) in two exact steps
    asm volatile("");   // a branch: predicated, its FP64 instructions would cost every element
    const int k = min(1100, max(-1080, e - 1023)), k1 = k / 2, k2 = k - k1;
    v = __longlong_as_double((long long)((1022ull << 52) + mant));
    v = v * __longlong_as_double((long long)(k1 + 1023) << 52) * __longlong_as_double((long long)(k2 + 1023) << 52);
  }
  return __longlong_as_double(__double_as_longlong(v) | (long long)neg);
}

// a 2^sh as FP64, rounded to nearest even
__device__ __forceinline__ double i64_to_f64(long long a, int sh) {
  const unsigned long long neg = (unsigned long long)a & 0x8000000000000000ull;
  const unsigned long long u = (unsigned long long)(a < 0 ? -a : a);
  const int lz = __clzll((long long)u);
  const unsigned long long m = u << (lz & 63);                         // leading one at bit 63
  unsigned long long mant = m >> 11;                                   // 53 significant bits
  mant += ((unsigned)(m & 0x7FFull) + 0x3FFu + (unsigned)(mant & 1ull)) >> 11;
  const double v = make_f64(neg, mant, 1086 - lz + sh);                // biased exponent: 1023 + (63 - lz) + sh
  return a == 0 ? 0.0 : v;
}

// a 2^sh as an unevaluated pair of FP32 numbers (hi, lo): hi = the value rounded to 24 bits, lo =
// the remainder rounded to 24 bits (about 48 significant bits)
__device__ __forceinline__ float2 i64_to_f32x2(long long a, int sh) {
  const unsigned neg = a < 0 ? 0x80000000u : 0u;
  const unsigned long long u = (unsigned long long)(a < 0 ? -a : a);
  const int lz = __clzll((long long)u);
  const unsigned long long m = u << (lz & 63);                         // value = m 2^(sh - lz)
  const unsigned hm = (unsigned)(m >> 40);                             // 24 significant bits
  long long r = (long long)(m & 0xFFFFFFFFFFull);
  const unsigned up = (r > 0x8000000000ll || (r == 0x8000000000ll && (hm & 1u))) ? 1u : 0u;
  r -= (long long)up << 40;                                            // the remainder of a rounded-up hi is negative
  const int e = sh - lz;
  float hi = __uint_as_float(((unsigned)(e + 189) << 23) + hm + up);   // biased exponent 127 + 63 + e, less the leading one
  // r = rh 2^20 + rl, both exact in FP32: one rounding
  float lo = fmaf((float)(int)(r >> 20), 1048576.f, (float)(int)(r & 0xFFFFFll)) * __uint_as_float((unsigned)(e + 127) << 23);
  if (e < -126 || e > 63) {   // outside the FP32 range of a direct scaling: through FP64
    asm volatile("");
    const double v = i64_to_f64(a < 0 ? -a : a, sh);
    hi = __double2float_rn(v);
    lo = __double2float_rn(v - (double)hi);
  }
  if (a == 0) hi = lo = 0.f;
  return make_float2(__uint_as_float(__float_as_uint(hi) ^ neg), __uint_as_float(__float_as_uint(lo) ^ neg));
}

// (hi 2^32 + lo) 2^sh as FP64, rounded to nearest even (|hi|, |lo| < 2^62): the two words are carried
// into one sign and a 96-bit magnitude, whose leading 64 bits (with a sticky bit) are rounded
__device__ __forceinline__ double i96_to_f64(long long hi, long long lo, int sh) {
  hi += lo >> 32;
  unsigned l = (unsigned)(unsigned long long)lo;
  const unsigned long long neg = (unsigned long long)hi & 0x8000000000000000ull;
  if (neg) {
    l = 0u - l;
    hi = l ? ~hi : -hi;
  }
  // the leading one of the 96 bits: in hi, or (hi = 0) in l
  const unsigned long long h = (unsigned long long)hi;
  const int lz = h ? __clzll((long long)h) : 64 + __clz((int)l);
  // x = the bits of (h : l : 0) below the first min(lz, 64) ones
  unsigned long long m = h << (lz & 63);
  const unsigned long long l64 = (unsigned long long)l << 32;
  if (lz >= 64)
    m = l64 << (lz - 64 & 63);
  else
    m |= lz ? l64 >> (64 - lz) : 0ull;
  const unsigned rest = lz < 32 ? l << lz : 0u;   // bits of l below the leading 64
  unsigned long long mant = m >> 11;
  mant += ((unsigned)(m & 0x7FFull) + 0x3FFu + ((unsigned)(mant & 1ull) | (rest ? 1u : 0u))) >> 11;
  const double v = make_f64(neg, mant, 1086 + 32 - lz + sh);
  return h == 0 && l == 0 ? 0.0 : v;
}

}  // namespace
}  // namespace librpa
