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

// balanced base-256 digits of x = v 2^-E (|x| < 1): x ~ sum_s d_s 2^{-7-8(s-1)}, |d_s| <= 128
template <int S>
__device__ __forceinline__ void make_digits(double v, int E, int (&d)[S]) {
  const long long bits = __double_as_longlong(v);
  const int ex = (int)((bits >> 52) & 0x7FF);
#pragma unroll
  for (int s = 0; s < S; ++s) d[s] = 0;
  if (ex == 0) return;   // zero (subnormals are far below any row scale of interest)
  const long long mant = (bits & 0xFFFFFFFFFFFFFLL) | (1LL << 52);
  const int r = 1075 + E - 7 - 8 * (S - 1) - ex;   // W = mant 2^-r, r > 0 since |x| < 1
  long long W = 0;
  if (r <= 0)
    W = mant << (-r);
  else if (r < 62)
    W = (mant + (1LL << (r - 1))) >> r;
  if (bits < 0) W = -W;
#pragma unroll
  for (int s = S - 1; s >= 1; --s) {
    const long long dg = ((W + 128) & 255) - 128;
    d[s] = (int)dg;
    W = (W - dg) >> 8;
  }
  d[0] = (int)W;
}

// ------------------------------------------------------------------ tcgen05 / TMA / mbarrier

constexpr uint64_t WAIT_NS = 2000000000ull;   // 2 s

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

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
// 16 columns of the warp's 32 TMEM lanes; the registers are valid after tmem_ld_wait on them
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
}
__device__ __forceinline__ void tmem_ld_wait(uint32_t (&r)[16]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                 "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15])
               :
               : "memory");
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
  if (e <= 0 || e >= 2046) {   // subnormal, overflow or next to it: scale [1, 2) in two exact steps
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
