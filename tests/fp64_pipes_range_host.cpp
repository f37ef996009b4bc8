// Host build of csrc/fp64_pipes.cuh at the ends of its range: operands next to
// 2^-511 and 2^512, whose quotients leave the normal numbers.
// Arguments: samples, seed.  Prints the number of results that differ from the
// host's IEEE operations, of those compared whose results are normal and of
// those refused.
#define main pipes_main
#include "fp64_pipes_host.cpp"
#undef main

int main(int argc, char** argv) {
  const long n = atol(argv[1]);
  std::mt19937_64 r(atol(argv[2]));
  const uint64_t M = 0xfffffffffffffull;
  const int ends[] = {-511, -510, -509, -1, 0, 1, 510, 511, 512};
  auto draw = [&] {
    const uint64_t e = 1023 + ends[r() % 9];
    const uint64_t m = r() % 4 == 0 ? 0 : (r() % 4 == 0 ? M : r() & M);
    return dbl((e << 52) | m | (r() << 63));
  };
  long differ = 0, normal = 0, refused = 0;
  auto verdict = [&](uint32_t rg, double got, double want) {
    const bool in = in_range(rg);
    if (in && bits(got) != bits(want)) ++differ;
    normal += std::isnormal(want);
    refused += !in;
  };
  for (long i = 0; i < n; ++i) {
    off = (int)(r() % 3) - 1;
    const double a = draw(), b = draw();
    uint32_t g = kInRange;
    double v = idiv(a, b, g);
    verdict(g, v, a / b);
    g = kInRange;
    v = imul(a, b, g);
    if (fabs(a * b) < INFINITY) verdict(g, v, a * b);
    g = kInRange;
    v = imul_const(13.0 / 12.0, a, g);
    verdict(g, v, 13.0 / 12.0 * a);
    g = kInRange;
    v = isqrt(fabs(a), g);
    verdict(g, v, sqrt(fabs(a)));
    // zeros stay in range
    g = kInRange;
    v = imul(0.0, a, g);
    if (!in_range(g) || bits(v) != bits(0.0 * a)) ++differ;
    g = kInRange;
    v = idiv(0.0, a, g);
    if (!in_range(g) || bits(v) != bits(0.0 / a)) ++differ;
  }
  printf("%ld %ld %ld\n", differ, normal, refused);
  return 0;
}
