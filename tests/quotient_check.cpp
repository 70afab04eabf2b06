// quotient.cuh's functions on the host, against the division: prints the number
// of operands tried and of results whose bits differ (NaN equals NaN).
#include <cstdio>
#include <cstdlib>
#include <limits>
#include <random>
#include <vector>

#include "quotient.cuh"

int main(int argc, char** argv) {
  std::mt19937_64 g(argc > 1 ? std::atoi(argv[1]) : 1);
  auto from_bits = [](uint64_t b) {
    double x;
    std::memcpy(&x, &b, 8);
    return x;
  };
  // sign, exponent field and mantissa: the edges of the range in which the fused steps serve, and mantissas at which
  // roundings go the other way
  const int edges[] = {0, 1, 2, 52, 199, 200, 201, 202, 1022, 1023, 1024, 1844, 1845, 1846, 1847, 2045, 2046, 2047};
  const uint64_t mants[] = {0, 1, 2, 3, (1ULL << 52) - 1, (1ULL << 52) - 2, 1ULL << 51, (1ULL << 51) - 1, (1ULL << 51) + 1};
  auto draw = [&](bool positive) {
    const uint64_t r = g();
    uint64_t e = (r >> 8) % 4 ? 600 + g() % 800 : (r >> 10) % 2 ? g() % 2048 : edges[(r >> 12) % (sizeof edges / sizeof *edges)];
    uint64_t m = (r >> 20) % 3 ? g() >> 12 : mants[(r >> 24) % (sizeof mants / sizeof *mants)];
    return from_bits((positive ? 0 : (r & 1) << 63) | e << 52 | m);
  };
  long n = 0, bad = 0;
  auto check = [&](double t, double c) {
    const double want = t / c, got = sharpy::quotient(t, c, 1.0 / c);
    uint64_t a, b;
    std::memcpy(&a, &want, 8);
    std::memcpy(&b, &got, 8);
    ++n;
    if (a != b && !(want != want && got != got)) {
      if (!bad++) std::fprintf(stderr, "%a / %a: %a, not %a\n", t, c, got, want);
    }
  };
  for (int i = 0; i < 4000000; ++i) check(draw(false), draw(true));
  const double inf = std::numeric_limits<double>::infinity(), nan = std::numeric_limits<double>::quiet_NaN(), tiny = 5e-324;
  const double special[] = {0.0, -0.0, 1.0, -1.0, 3.0, tiny, -tiny, 2.2250738585072014e-308, 1.7976931348623157e308, inf, -inf, nan};
  for (double t : special)
    for (double c : special) check(t, c);
  for (double t : special)
    for (int i = 0; i < 1000; ++i) check(t, draw(true)), check(draw(false), t);
  std::printf("%ld %ld\n", n, bad);
  return 0;
}
