// FP64 values as balanced base-256 digits, exact in BF16, for exact products on
// mma.sync (expand.cuh, finalize.cu): a digit product is at most 2^14, so sums of a
// bounded number of them are exact in the FP32 accumulators.
#pragma once
#include <cstdint>

namespace tts {
namespace digit {

constexpr int kExpZero = -4000;  // exponent that stands for a zero

__device__ __forceinline__ uint32_t s_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void ldsm4(uint32_t a, uint32_t* r) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(a));
}
__device__ __forceinline__ void mma(float* c, const uint32_t* a, const uint32_t* b) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
               "{%0,%1,%2,%3};" : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
               : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}
// The same with c = 0 on entry (no registers cleared first).
__device__ __forceinline__ void mma0(float* c, const uint32_t* a, const uint32_t* b) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
               "{%10,%10,%10,%10};" : "=f"(c[0]), "=f"(c[1]), "=f"(c[2]), "=f"(c[3])
               : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]), "f"(0.0f));
}

// Exponent e with |x| < 2^e (kExpZero for zero and subnormal numbers, which count as zero).
__device__ __forceinline__ int exp_of(double x) {
  const int e = (__double2hiint(x) >> 20) & 0x7ff;
  return e == 0 ? kExpZero : e - 1022;
}
__device__ __forceinline__ bool nonfinite(double x) { return ((__double2hiint(x) >> 20) & 0x7ff) == 0x7ff; }
// Infinite, NaN or subnormal: not what the digits hold.
__device__ __forceinline__ bool undigital(double x) {
  const unsigned e = ((unsigned)__double2hiint(x) >> 20) & 0x7ffu;
  return e - 1u >= 0x7feu && x != 0.0;
}

// round(x 2^(B - E)), |x| < 2^E, in integer arithmetic.
template <int B>
__device__ __forceinline__ long long fixed(double x, int E) {
  const long long bits = __double_as_longlong(x);
  const int e = (int)((bits >> 52) & 0x7ff);
  if (e == 0) return 0;
  const unsigned long long m = ((unsigned long long)bits & 0xfffffffffffffull) | (1ull << 52);
  static_assert(B <= 61, "q and its balanced digits fit 64 bits");
  const int s = 1075 + E - B - e;   // >= 53 - B
  if (s > 54) return 0;
  const long long q = (long long)(s > 0 ? (m + (1ull << (s - 1))) >> s : B > 53 ? m << -s : m);
  return bits < 0 ? -q : q;
}

// The P balanced base-256 digits of q (most significant first) as BF16 bit
// patterns: the bytes of q + 0x80..80, less 128 each.
template <int P>
__device__ __forceinline__ void digits(long long q, uint32_t (&d)[P]) {
  unsigned long long b = (unsigned long long)q;
#pragma unroll
  for (int i = 0; i < P; ++i) b += 0x80ull << (8 * i);
#pragma unroll
  for (int i = 0; i < P; ++i) {
    const uint32_t byte = (uint32_t)(b >> (8 * (P - 1 - i))) & 0xffu;
    d[i] = __float_as_uint(__fsub_rn(__uint_as_float(0x4B000000u | byte), 8388736.0f)) >> 16;
  }
}

// c += |a| |b|: of leading digits, a measure of a product's terms (below).
__device__ __forceinline__ void mma_abs(float* c, const uint32_t* a, const uint32_t* b) {
  uint32_t x[4], y[2];
#pragma unroll
  for (int i = 0; i < 4; ++i) x[i] = a[i] & 0x7fff7fffu;
#pragma unroll
  for (int i = 0; i < 2; ++i) y[i] = b[i] & 0x7fff7fffu;
  mma(c, x, y);
}

// Whether a sum of digit products has to be formed in FP64 instead.  mag = sum |d0 d0'|
// of the leading digits, full scale 2^LEAD each; a digit that is not zero is at most twice its
// value, so the terms' magnitudes add up to at least mag 2^(-2 LEAD) / 4 of the two largest factors'
// product.  Below `part` of that they may be as small as what the digits drop; then the
// digits still serve if that, K 2^-57 of the factors' product for K terms, is no more than K
// FP64 additions may lose of the sum so far, K 2^-53 |sum|: |sum| >= 2^e, e four below the
// factors' exponents.
__device__ __forceinline__ bool weak(float mag, float part, int lead, double sum, int e) {
  return mag < part * (float)(1 << (2 * lead)) && exp_of(sum) <= e;
}
}  // namespace digit
}  // namespace tts
