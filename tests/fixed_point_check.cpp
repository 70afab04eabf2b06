// fixed.cuh's functions on the host against wider arithmetic. Prints one line per check: its name, the largest error
// and the bound, in the check's own units.
#include <cuda_runtime.h>

#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <random>
#include <vector>
#if defined(__x86_64__)
#include <quadmath.h>
using wide = __float128;
static void wide_sincos(wide x, wide* s, wide* c) { sincosq(x, s, c); }
static wide wide_abs(wide x) { return fabsq(x); }
static wide wide_floor(wide x) { return floorq(x); }
static wide wide_sqrt(wide x) { return sqrtq(x); }
#else  // long double has 113 bits
using wide = long double;
static void wide_sincos(wide x, wide* s, wide* c) { *s = sinl(x), *c = cosl(x); }
static wide wide_abs(wide x) { return fabsl(x); }
static wide wide_floor(wide x) { return floorl(x); }
static wide wide_sqrt(wide x) { return sqrtl(x); }
#endif
// common.cuh's device helpers, not called here
#define atomicCAS(p, a, b) (b)
#define __shfl_xor_sync(m, v, o) (v)
#include "fixed.cuh"

using namespace sharpy;

static wide pi2() {  // 2 pi to 113 bits: twice the root of cosine near the double
  wide x = 3.14159265358979323846 / 2, s, c;
  for (int i = 0; i < 4; ++i) {
    wide_sincos(x, &s, &c);
    x += c / s;
  }
  return 4 * x;
}
static const wide kTurn = pi2(), k64 = (wide)18446744073709551616.0;

static void report(const char* name, wide worst, double bound) { std::printf("%s %.6g %.6g\n", name, (double)worst, bound); }
static wide worst_of(wide a, wide b) { return a > b ? a : b; }
static int64_t value(Limbs l) { return (int64_t)((uint64_t)(int64_t)l.h << 32) + l.l; }

int main(int argc, char** argv) {
  std::mt19937_64 g(argc > 1 ? std::atoi(argv[1]) : 1);
  const int64_t top = 1LL << 61;

  {  // fix_limbs, fix_limbs_neg: the value, limbs whose negatives exist
    wide worst = 0;
    for (int i = 0; i < 200000; ++i) {
      int64_t v = (int64_t)g() >> (2 + g() % 60);
      if (i % 4 == 0) v = ((int64_t)(g() % 5) - 2) * (1LL << (28 + g() % 33)) + (int64_t)(g() % 5) - 2;
      worst = worst_of(worst, wide_abs((wide)value(fix_limbs(v)) - (wide)v));
      const Limbs n = fix_limbs_neg(v);
      wide d = wide_abs((wide)value(n) - (wide)v);
      if (n.l == INT32_MIN) d = 99;
      worst = worst_of(worst, d);
    }
    report("limbs", worst, 1.0);
  }
  {  // fix_frac: P mod 1 in 2^-64, what lies below cut off
    wide worst = 0;
    auto one = [&](double P) {
      wide q = (wide)P;
      q -= wide_floor(q);
      wide d = wide_abs((wide)fix_frac(P) - q * k64);
      if (d > k64 / 2) d = k64 - d;
      worst = worst_of(worst, d);
    };
    for (int i = 0; i < 400000; ++i) one(std::ldexp((double)(int64_t)g(), -(int)(g() % 150)));
    for (int e = -1074; e < 1024; ++e)
      for (double m : {1.0, 1.0 + 0x1p-52, 2.0 - 0x1p-52})
        for (double s : {1.0, -1.0}) one(s * std::ldexp(m, e));
    one(0.0);
    one(-0.0);
    report("frac", worst, 1.0);
  }
  // fractions at which the table's index wraps and the rest reaches its ends
  auto fraction = [&](int i) {
    uint64_t u = g();
    if (i % 8 == 1) u = (u & 0x3ff) << 54 | ((1ULL << 53) + (int64_t)(g() % 5) - 2);  // between two points
    if (i % 8 == 2) u = ((u & 0x3ff) << 54) + g() % 1000;                                // just after one
    if (i % 8 == 3) u = ((u & 0x3ff) << 54) - g() % 1000;                                // just before
    if (i % 8 == 4) u = ((u & 0x3ff) << 54) + ((g() % 3) << 22) - g() % 3;               // limb boundaries of the rest
    return u;
  };
  {  // index and rest put together again
    wide worst = 0;
    for (int i = 0; i < 400000; ++i) {
      const uint64_t u = fraction(i);
      const int64_t y = fix_rest(u);  // (pi / 1024) y 2^-62 = 2 pi y 2^-73 = y 2^-9 units of 2^-64 turns
      if (y > 1LL << 62 || y < -(1LL << 62)) worst = 99;
      wide d = wide_abs((wide)fix_index(u) * k64 / 1024 + (wide)y / 512 - (wide)u);
      if (d > k64 / 2) d = wide_abs(k64 - d);
      worst = worst_of(worst, d);
    }
    report("index_and_rest", worst, 0.0);
  }
  {  // sine and cosine - 1 of the rest, in 2^-64. Sine: t is cut off at three places, 1.65 units of 2^-48 of the angle
     // (at most pi / 1024) in all, 2^-57.28 = 105, and two roundings. Cosine: the term left out, kappa^3 / 720, is 21.4;
     // cut-offs in H0's units, a sixteenth each, and two roundings
    wide ws = 0, wc = 0;
    for (int i = 0; i < 400000; ++i) {
      int64_t y = fix_rest(fraction(i));
      if (i % 16 == 0) y = (1LL << 62) - (int64_t)(g() % 3);
      if (i % 16 == 1) y = -(1LL << 62) + (int64_t)(g() % 3);
      int64_t s, c;
      fix_small(y, &s, &c);
      wide ts, tc;
      wide_sincos(kTurn / 2048 * (wide)y / (wide)(1LL << 62), &ts, &tc);
      ws = worst_of(ws, wide_abs((wide)s - ts * k64));
      wc = worst_of(wc, wide_abs((wide)c - (tc - 1) * k64));
    }
    report("sine", ws, 107.0);
    report("cosine", wc, 25.0);
  }
  std::vector<int4> table(kFixTrig);
  for (int i = 0; i < kFixTrig; ++i) {
    wide s, c;
    wide_sincos(kTurn * i / kFixTrig, &s, &c);
    auto q = [](wide x) { return fix_limbs_neg((int64_t)wide_floor(x * (wide)(1LL << 62) + (wide)0.5)); };
    const Limbs C = q(c), S = q(s);
    table[i] = make_int4(C.h, C.l, S.h, S.l);
  }
  {  // E times the carrier, of |E|'s full scale (2^61 sqrt(2); 2^59 sqrt(2) in z's units): across it the sine's 5.8e-18,
     // along it the cosine's 1.4e-18, the table's 1.5e-19, and for each part and of the two products half a unit of 2^-59
     // of rounding and half of low limbs left out, 3.5e-18: 9.6e-18 < 2^-56.5
    wide worst = 0, ss = 0;
    const int N = 400000;
    for (int i = 0; i < N; ++i) {
      int64_t re = (int64_t)(g() >> 2) - top, im = (int64_t)(g() >> 2) - top;
      if (i % 5 == 0) re = g() & 1 ? top : -top;
      if (i % 7 == 0) im = g() & 1 ? top : -top;
      if (i % 11 == 0) re >>= g() % 50;
      const Limbs a = fix_limbs_neg(re), b = fix_limbs_neg(im);
      re = value(a), im = value(b);
      const uint64_t u = fraction(i);
      int64_t zr, zi;
      fix_carrier(u, make_int4(a.h, a.l, b.h, b.l), table[fix_index(u)], &zr, &zi);
      wide s, c;
      wide_sincos(kTurn * (wide)u / k64, &s, &c);
      const wide dr = (wide)zr - ((wide)re * c + (wide)im * s) / 4, di = (wide)zi - ((wide)im * c - (wide)re * s) / 4;
      worst = worst_of(worst, wide_sqrt(dr * dr + di * di));
      ss += (dr * dr + di * di) / 2;
    }
    const double full = 0x1p59 * std::sqrt(2.0);
    report("carrier", worst / full, 0x1p-57 * std::sqrt(2.0));
    report("carrier_rms_per_part", wide_sqrt(ss / N) / 0x1p59, 0x1p-58);
  }
  {  // moment sums of n products with the offset: each product's high word is within one unit
    wide worst = 0, worst1 = 0;
    for (int rep = 0; rep < 4000; ++rep) {
      const int n = 1 + (int)(g() % 256), sh = (int)(g() % 3);
      int64_t acc = fix_start(n), acc1 = fix_start(n);
      wide exact = 0, exact1 = 0;
      for (int k = 0; k < n; ++k) {
        // |z| <= 2^59 sqrt(2); |B| at most what the scale rule leaves a sum of 256 (2^58)
        int64_t z = (int64_t)(g() >> 4) - (1LL << 59), B = (int64_t)(g() >> 5) - (1LL << 58);
        if (sh == 1) z = g() & 1 ? (1LL << 59) : -(1LL << 59), B = g() & 1 ? (1LL << 58) : -(1LL << 58);
        if (sh == 2) z >>= g() % 58, B >>= g() % 57;
        const Limbs zl = fix_limbs(z), bl = fix_limbs_neg(B);
        acc = fix_moment(zl, bl.h, bl.l, acc);
        exact += (wide)z * (wide)value(bl) / k64;
        const int one = 1 << (24 + g() % 4);
        acc1 = fix_moment1(zl, one, acc1);
        exact1 += (wide)z * (wide)((int64_t)one << 32) / k64;
      }
      worst = worst_of(worst, wide_abs((wide)acc - exact) / n);
      worst1 = worst_of(worst1, wide_abs((wide)acc1 - exact1) / n);
    }
    report("moment_per_product", worst, 1.0);
    report("moment_of_one_per_product", worst1, 1.0);
  }
  return 0;
}
