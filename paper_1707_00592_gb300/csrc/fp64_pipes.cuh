// Correctly rounded binary64 division, square root and multiplication on the
// integer and FP32 pipes.
//
// GB300 issues one FP64-pipe instruction per warp and SM sub-partition every
// 76 cycles (measured; DADD, DMUL and DFMA alike) against 1 to 5 for an
// integer one, so the FP64 sweep is bound by the FP64 pipe while the other
// pipes idle.  A division or root compiled for that pipe holds it for 565 or
// 572 cycles; the digit-by-digit ones below take about 90 issue cycles of the
// other pipes, a product about 50, and leave the FP64 pipe to the additions.
// (An addition would take as many integer instructions as it saves: its
// alignment and normalisation shifts are the expensive part.)  Results are
// those of IEEE round-to-nearest-even, bit for bit.
#pragma once

#ifndef WS_FP64_PIPES_HOST  // the host test brings the few device functions used here
#include <cuda_runtime.h>
#endif
#include <stdint.h>

namespace ws {
namespace fp64 {

// y ~ 1/x and 1/sqrt(x) for 1 <= x < 4, to one FP32 ulp and two
#ifndef WS_FP64_PIPES_HOST
__device__ __forceinline__ float rcp_approx(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float rsqrt_approx(float x) {
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
#endif

__device__ __forceinline__ uint32_t hi_of(double x) { return (uint32_t)__double2hiint(x); }
__device__ __forceinline__ uint32_t lo_of(double x) { return (uint32_t)__double2loint(x); }
__device__ __forceinline__ bool is_zero(double x) { return ((hi_of(x) << 1) | lo_of(x)) == 0u; }
// x > 0 (false for NaN), decided on the bits
__device__ __forceinline__ bool positive(double x) {
  const long long b = __double_as_longlong(x);
  return b > 0 && b <= 0x7ff0000000000000LL;
}

// The functions below take operands of 2^-511 <= |x| < 2^513 (the two leading
// exponent bits differ) and, where they say so, zeros.  They do not branch on
// anything else (a branch per operation would keep the compiler from running
// independent ones side by side); instead `range` loses its bit 31, and the
// caller evaluates the whole expression again with the native operations.
// Quotients that are not normal numbers (or zeros) count as out of range.
constexpr uint32_t kInRange = 0xffffffffu;
__device__ __forceinline__ bool in_range(uint32_t range) { return (int)range < 0; }
__device__ __forceinline__ void check(uint32_t& range, uint32_t hi) { range &= (hi << 1) ^ (hi << 2); }
__device__ __forceinline__ void check_or_zero(uint32_t& range, uint32_t hi, bool zero) {
  range &= ((hi << 1) ^ (hi << 2)) | (zero ? 0x80000000u : 0u);
}

// a / b (a may be zero).  Long division with quotient digits of 19, 19 and 16
// bits, each from an FP32 product with y ~ 1/b, and exact remainders modulo 2^64:
//   A, B: the 53-bit significands;  y = (1/Bm)(1 + e), |e| < 2^-22, Bm = B/2^52
//   Q1 = round(A/B 2^19), off by < 0.75;    R1 = A 2^19 - Q1 B,  |R1| < 0.75 B
//   Q2 = round(R1/B 2^19), off by < 1.19;   R2 = R1 2^19 - Q2 B, |R2| < 1.19 B
//   Q3 = round(R2/B 2^16), off by < 0.61;   R3 = R2 2^16 - Q3 B, |R3| < 0.61 B
// so A/B = (Q1 2^35 + Q2 2^16 + Q3 + R3/B) 2^-54 exactly.  A quotient of two
// 53-bit numbers is never halfway between two others (B times an odd 54-bit
// number has more than the 53 + k significant bits of A 2^k), so the sign of
// R3 is all that rounding needs beside the digits: the digits are doubled and
// moved by one to the side of R3, and rounded by adding half a unit.
__device__ __forceinline__ double idiv(double a, double b, uint32_t& range) {
  const uint32_t ah = hi_of(a), al = lo_of(a), bh = hi_of(b), bl = lo_of(b);
  const bool za = ((ah << 1) | al) == 0u;
  check(range, bh);
  check_or_zero(range, ah, za);
  const uint32_t Ah = (ah & 0xfffffu) | 0x100000u, Bh = (bh & 0xfffffu) | 0x100000u;
  // leading 24 bits as floats in [1, 2)
  const float Af = __uint_as_float((__funnelshift_l(al, ah, 3) & 0x7fffffu) | 0x3f800000u);
  const float Bf = __uint_as_float((__funnelshift_l(bl, bh, 3) & 0x7fffffu) | 0x3f800000u);
  const float y = rcp_approx(Bf);
  const float magic = 12582912.0f;  // 1.5 2^23: adding it rounds to an integer kept in the low bits
  auto times_b = [&](int q) {       // q B modulo 2^64
    uint64_t p = (uint64_t)(uint32_t)q * bl;
    const uint32_t ph = (uint32_t)(p >> 32) + (uint32_t)q * Bh;
    return ((uint64_t)ph << 32) | (uint32_t)p;
  };
  // q is signed: (uint32_t)q = q + 2^32 [q < 0], so its product with bl is too large by bl 2^32
  auto times_b_signed = [&](int q) { return times_b(q) - ((uint64_t)((uint32_t)(q >> 31) & bl) << 32); };
  const uint32_t Q1 = __float_as_uint(__fmaf_rn(Af, y, 24.0f)) - 0x41c00000u;  // 24 = 1.5 2^4: 19 fraction bits
  const uint64_t A = ((uint64_t)Ah << 32) | al;
  const uint64_t R1 = (A << 19) - times_b((int)Q1);
  const float h1 = __uint_as_float((uint32_t)(R1 >> 32) + 0x4b400000u) - magic;
  const int Q2 = (int)(__float_as_uint(__fmaf_rn(h1, 0.5f * y, magic)) - 0x4b400000u);
  const uint64_t R2 = (R1 << 19) - times_b_signed(Q2);
  const float h2 = __uint_as_float((uint32_t)(R2 >> 32) + 0x4b400000u) - magic;
  const int Q3 = (int)(__float_as_uint(__fmaf_rn(h2, 0.0625f * y, magic)) - 0x4b400000u);
  const uint64_t R3 = (R2 << 16) - times_b_signed(Q3);
  // 2 (Q1 2^35 + Q2 2^16 + Q3) + sign(R3)
  const int c = 2 * Q3 + 1 + 2 * ((int)(uint32_t)(R3 >> 32) >> 31);
  uint64_t q = (uint64_t)((int64_t)Q2 * 131072 + c);
  q += (uint64_t)(Q1 << 4) << 32;
  const uint32_t g = (uint32_t)(q >> 55);  // 1: the quotient of the significands is >= 1
  q += 2u + 2u * g;
  const uint32_t qh = (uint32_t)(q >> 32), ql = (uint32_t)q, sh = 2u + g;
  const uint32_t ml = __funnelshift_r(ql, qh, sh), mh = qh >> sh;
  // mh carries the implicit bit
  const uint32_t e = (ah & 0x7ff00000u) - (bh & 0x7ff00000u);
  range &= ~(e + (1021u << 20)) | (za ? 0x80000000u : 0u);  // a quotient that may be below 2^-1022
  const uint32_t rh = mh + e + ((1021u + g) << 20);
  const uint32_t sign = (ah ^ bh) & 0x80000000u;
  return __hiloint2double((int)(za ? sign : rh | sign), (int)(za ? 0u : ml));
}

// Significands of the product of two normal numbers, rounded to nearest even:
// the 106-bit product from four 32 x 32 ones (sticky: the discarded low word).
// Returns the magnitude of the result.
__device__ __forceinline__ uint64_t product(uint32_t ah, uint32_t al, uint32_t bh, uint32_t bl) {
  const uint32_t Ah = (ah & 0xfffffu) | 0x100000u, Bh = (bh & 0xfffffu) | 0x100000u;
  const uint64_t p0 = (uint64_t)al * bl;
  uint64_t mid = (uint64_t)al * Bh + (uint32_t)(p0 >> 32);
  mid = (uint64_t)Ah * bl + mid;
  const uint64_t top = (uint64_t)Ah * Bh + (uint32_t)(mid >> 32);  // product bits 64 .. 105
  const uint32_t th = (uint32_t)(top >> 32), tl = (uint32_t)top, m0 = (uint32_t)mid, p0l = (uint32_t)p0;
  const uint32_t n = th >> 9;  // 1: the product of the significands is >= 2
  const uint32_t sh = 12u - n;
  const uint32_t mh = __funnelshift_l(tl, th, sh), ml = __funnelshift_l(m0, tl, sh);
  const uint32_t rest = (m0 << sh) | (p0l != 0u ? 1u : 0u);       // discarded bits, leading first
  const uint32_t up = rest > 0x80000000u - (ml & 1u) ? 1u : 0u;  // above half, or half and odd
  const uint64_t t = (((uint64_t)mh << 32) | ml) + up;
  return t + ((uint64_t)((ah & 0x7ff00000u) + (bh & 0x7ff00000u) - ((1024u - n) << 20)) << 32);
}

// a * b for |a b| < 2^1024 (either may be zero).  Not tested here, where it would
// cost the FP64 sweep 2.8 %: its callers keep within it.
__device__ __forceinline__ double imul(double a, double b, uint32_t& range) {
  const uint32_t ah = hi_of(a), al = lo_of(a), bh = hi_of(b), bl = lo_of(b);
  const bool za = is_zero(a), zb = is_zero(b);
  check_or_zero(range, ah, za);
  check_or_zero(range, bh, zb);
  const uint64_t r = product(ah, al, bh, bl);
  const uint32_t sign = (ah ^ bh) & 0x80000000u;
  const bool z = za || zb;
  return __hiloint2double((int)(z ? sign : (uint32_t)(r >> 32) | sign), (int)(z ? 0u : (uint32_t)r));
}

// a * b for a constant a of 2^-100 to 2^100
__device__ __forceinline__ double imul_const(double a, double b, uint32_t& range) {
  const uint32_t ah = hi_of(a), al = lo_of(a), bh = hi_of(b), bl = lo_of(b);
  const bool z = is_zero(b);
  check_or_zero(range, bh, z);
  const uint64_t r = product(ah, al, bh, bl);
  const uint32_t sign = (ah ^ bh) & 0x80000000u;
  return __hiloint2double((int)(z ? sign : (uint32_t)(r >> 32) | sign), (int)(z ? 0u : (uint32_t)r));
}

// a * a for |a| < 2^512, taken as zero where |a| < 2^-255
__device__ __forceinline__ double isquare(double a, uint32_t& range) {
  const uint32_t ah = hi_of(a) & 0x7fffffffu, al = lo_of(a);
  const bool z = ah < (768u << 20);
  check_or_zero(range, ah, z);
  const uint64_t r = product(ah, al, ah, al);
  return __hiloint2double((int)(z ? 0u : (uint32_t)(r >> 32)), (int)(z ? 0u : (uint32_t)r));
}

// sqrt(x) for x > 0 (or a zero, which it returns).  The digits of idiv:
//   x = m 4^k, 1 <= m < 4, M = m 2^52;  y ~ 1/sqrt(m) to 2^-22, s = sqrt(m)
//   S1 = round(s 2^19), off by < 0.9;  R1 = m 2^38 - S1^2 (kept times 2^14, an integer)
//   S2 = round(R1 2^19 / (2 S1)), off by < 1.9;    R2 = R1 2^38 - (2 S1 2^19 + S2) S2
//   S3 = round(R2 2^16 / (2 (S1 2^19 + S2))), off by < 0.7;  R3 likewise, modulo 2^64
// The root of a 53-bit number is never halfway between two others (the square
// of an odd 54-bit number is odd), so the sign of R3 decides the rounding.
__device__ __forceinline__ double isqrt(double x, uint32_t& range) {
  const uint32_t h = hi_of(x), l = lo_of(x);
  const bool z = ((h << 1) | l) == 0u;
  check_or_zero(range, h, z);
  range &= z ? 0xffffffffu : ~h;  // negative
  const uint32_t odd = ~(h >> 20) & 1u;  // exponent field even: an odd power of two, m in [2, 4)
  const uint32_t Mh = (((h & 0xfffffu) | 0x100000u) << odd) | (odd ? l >> 31 : 0u), Ml = l << odd;
  // leading 24 bits of m as a float in [1, 4)
  const float mf = __uint_as_float(((__funnelshift_l(l, h, 3) & 0x7fffffu) | 0x3f800000u) + (odd << 23));
  const float y = rsqrt_approx(mf);
  const float magic = 12582912.0f;
  const uint32_t S1 = __float_as_uint(__fmaf_rn(mf, y, 24.0f)) - 0x41c00000u;  // s 2^19, up to 2^20
  const int64_t R1 = (int64_t)(((uint64_t)Mh << 32) | Ml) - (int64_t)(((uint64_t)S1 * S1) << 14);  // |R1| < 2^36
  const float r1 = __uint_as_float((uint32_t)(R1 >> 15) + 0x4b400000u) - magic;                  // R1 2^-15
  const int S2 = (int)(__float_as_uint(__fmaf_rn(r1, y, magic)) - 0x4b400000u);
  const uint64_t R2 = ((uint64_t)R1 << 24) - (uint64_t)(int64_t)S2 * (((uint64_t)S1 << 20) + (uint64_t)(int64_t)S2);
  const float r2 = __uint_as_float((uint32_t)((int64_t)R2 >> 20) + 0x4b400000u) - magic;  // |R2| < 2^42
  const int S3 = (int)(__float_as_uint(__fmaf_rn(r2, 0.125f * y, magic)) - 0x4b400000u);
  const uint64_t S12 = ((uint64_t)S1 << 19) + (uint64_t)(int64_t)S2;
  const uint64_t R3 = (R2 << 32) - (uint64_t)(int64_t)S3 * ((S12 << 17) + (uint64_t)(int64_t)S3);
  const uint64_t S = (S12 << 16) + (uint64_t)(int64_t)S3;  // s 2^54
  const uint64_t q = 2u * S + 1u + 2u * (uint64_t)((int64_t)R3 >> 63) + 4u;
  const uint64_t m = q >> 3;  // s 2^52 rounded, implicit bit included
  // field 1023 + 2k + odd of x gives 1023 + k; m carries the implicit bit
  const uint32_t rh = (uint32_t)(m >> 32) + (((((h >> 20) + 1023u - odd) >> 1) - 1u) << 20);
  return __hiloint2double((int)(z ? h : rh), (int)(z ? 0u : (uint32_t)m));
}

static __device__ __noinline__ double native_div(double a, double b) { return a / b; }
static __device__ __noinline__ double native_sqrt(double x) { return sqrt(x); }
// a / b and sqrt(x) of any operands, subnormal results included
__device__ __forceinline__ double divide(double a, double b) {
  uint32_t rg = kInRange;
  const double q = idiv(a, b, rg);
  return in_range(rg) ? q : native_div(a, b);
}
__device__ __forceinline__ double root(double x) {
  uint32_t rg = kInRange;
  const double s = isqrt(x, rg);
  return in_range(rg) ? s : native_sqrt(x);
}
// The same out of line, where a kernel's code is long or runs once per thread:
// its warps then wait for less of it to be fetched.
static __device__ __noinline__ double divide_call(double a, double b) { return divide(a, b); }
static __device__ __noinline__ double root_call(double x) { return root(x); }

}  // namespace fp64
}  // namespace ws
