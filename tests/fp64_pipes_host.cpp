// Host build of csrc/fp64_pipes.cuh: random and hard operands of each operation
// against the host's own IEEE operations.  Arguments: samples per operation,
// seed.  Prints the number of results that differ and the number of samples
// whose operands were refused (out of range).
#include <math.h>
#include <stdint.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

#include <algorithm>
#include <random>

#define __device__
#define __forceinline__ inline
#define __noinline__
static uint64_t bits(double x) { uint64_t b; memcpy(&b, &x, 8); return b; }
static double dbl(uint64_t b) { double x; memcpy(&x, &b, 8); return x; }
static int __double2hiint(double x) { return (int)(bits(x) >> 32); }
static int __double2loint(double x) { return (int)bits(x); }
static long long __double_as_longlong(double x) { return (long long)bits(x); }
static double __hiloint2double(int h, int l) { return dbl(((uint64_t)(uint32_t)h << 32) | (uint32_t)l); }
static uint32_t __funnelshift_l(uint32_t lo, uint32_t hi, uint32_t s) { s &= 31; return s ? (hi << s) | (lo >> (32 - s)) : hi; }
static uint32_t __funnelshift_r(uint32_t lo, uint32_t hi, uint32_t s) { s &= 31; return s ? (lo >> s) | (hi << (32 - s)) : lo; }
static float __uint_as_float(uint32_t u) { float f; memcpy(&f, &u, 4); return f; }
static uint32_t __float_as_uint(float f) { uint32_t u; memcpy(&u, &f, 4); return u; }
static float __fmaf_rn(float a, float b, float c) { return fmaf(a, b, c); }

namespace ws {
namespace fp64 {
static int off = 0;  // error given to the approximations, in ulps
static float rcp_approx(float x) { return __uint_as_float(__float_as_uint(1.0f / x) + off); }
static float rsqrt_approx(float x) { return __uint_as_float(__float_as_uint((float)(1.0 / sqrt((double)x))) + 2 * off); }
}  // namespace fp64
}  // namespace ws
#define WS_FP64_PIPES_HOST
#include "../paper_1707_00592_gb300/csrc/fp64_pipes.cuh"

using namespace ws::fp64;

int main(int argc, char** argv) {
  const long n = atol(argv[1]);
  std::mt19937_64 r(atol(argv[2]));
  const uint64_t M = 0xfffffffffffffull;
  long differ = 0, refused = 0;
  auto verdict = [&](uint32_t rg, double got, double want) {
    if (!in_range(rg))
      ++refused;
    else if (bits(got) != bits(want))
      ++differ;
  };
  for (long i = 0; i < n; ++i) {
    off = (int)(r() % 3) - 1;
    uint64_t ma = r() & M, mb = r() & M;
    const int kind = (int)(r() % 8);
    if (kind == 0) ma &= ~0ull << (r() % 52);      // short significands
    if (kind == 1) mb &= ~0ull << (r() % 52);
    if (kind == 2) mb = (mb | ~(~0ull << (r() % 52))) & M;
    if (kind == 3) ma = (mb + (r() % 5) - 2) & M;  // quotients next to 1
    const int span = i % 16 == 0 ? 1000 : 100;
    double a = dbl(((1023 + r() % (2 * span) - span) << 52) | ma | (r() << 63));
    double b = dbl(((1023 + r() % (2 * span) - span) << 52) | mb | (r() << 63));
    if (kind == 4) a = (double)((long double)b * (long double)(double)((1ull << 53) | (r() & 0x1ffffffffffffeull) | 1));
    if (kind == 5) a = b * (double)((r() & M) | 0x10000000000000ull);
    if (i % 1000 == 0) a = 0.0;
    double x = fabs(b);
    if (kind == 6) {  // roots next to a double, and next to halfway
      const long double w = (long double)((r() & 0x1fffffffffffffull) | 0x20000000000000ull) + (i & 8 ? 0.5L : 0.0L);
      x = (double)(w * w);
    }
    uint32_t g = kInRange;
    double v = idiv(a, b, g);
    verdict(g, v, a / b);
    g = kInRange;
    v = imul(a, b, g);
    if (fabs(a) < 0x1p512) verdict(g, v, a * b);
    g = kInRange;
    v = imul_const(13.0 / 12.0, b, g);
    verdict(g, v, 13.0 / 12.0 * b);
    g = kInRange;
    v = isquare(a, g);
    if (fabs(a) < 0x1p512) verdict(g, v, fabs(a) < 0x1p-255 ? 0.0 : a * a);
    g = kInRange;
    v = isqrt(x, g);
    verdict(g, v, sqrt(x));
  }
  // refused: negative roots, infinities, NaN, subnormal numbers
  const double odd[] = {-1.0, INFINITY, -INFINITY, NAN, 5e-324, 1e300};
  for (double o : odd) {
    uint32_t g = kInRange;
    isqrt(o, g);
    differ += in_range(g);
    if (o == -1.0) continue;
    g = kInRange;
    idiv(1.0, o, g);
    differ += in_range(g);
    g = kInRange;
    imul(o, 1.0, g);
    differ += in_range(g);
  }
  uint32_t g = kInRange;  // a zero divisor
  idiv(1.0, 0.0, g);
  differ += in_range(g);
  printf("%ld %ld\n", differ, refused);
  return 0;
}
