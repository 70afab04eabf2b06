// The FP64 path's bins in 64-bit fixed point: carrier, data product and moment
// products on the integer pipe, the phase in FP64.
//
// An FP64 warp instruction holds a sub-partition's FP64 pipe for 60 cycles on
// this GPU, a 32 x 32 + 64 bit multiply-add its pipe for 2 to 4 (as the operands
// are reused); a bin and detector of the FP64 sweep takes about 50 of the former
// (a third in sincospi, two fifths in the moments), or 4 of them and about 170
// integer instructions as below. 1000 vectors near the injection (8033 bins,
// ~320 active), with the gradient: 166 to 70 us by this alone, a NUTS mutation
// of 1001 particles 22.0 to 11.6 ms (173 to 53 us and 21.3 to 9.1 ms with the
// prologue and epilogue on lanes, in another event); ln L and gradient as far
// from a 64-bit evaluation as before (1e-13 to 8e-13: the phase's rounding).
//
// Numbers are 64-bit integers v = h 2^32 + l with both limbs signed; the high
// word of a product is ah bh + (ah bl + al bh) / 2^32, rounded: 3 multiply-adds,
// error under one unit. Errors against the FP64 sweep's, per bin:
//   phase   the same FP64 sum, then its fraction of a turn exact to 2^-64;
//   carrier E times it within 2^-56.5 of the block's largest |E| (2^-59.5 rms a
//           part; a table of 1024 points to 2^-62, sine and cosine of the rest,
//           |d| <= pi / 1024, by their Taylor series: 2^-57.3 and 2^-59.5 at
//           its ends); FP64: 2^-53 of |E|;
//   data    E scaled to 2^61 by the block's largest;
//   moments sums of the products' high words: exact, in any order, up to the
//           block's final rounding to FP64 (FP64 sweep: one rounding per bin).
// Scales are powers of two per block of 256 bins (event_tables_kernel): over so
// few bins E and the basis change little, and their sums need few bits of
// headroom (with blocks of 2048 a sweep that ends early had up to 30 times the
// FP64 sweep's error).
// A bin far below its block's largest has a larger relative error than in FP64;
// the sum it joins has not if the sweep has met values as large before its end.
// That is what decides, per end of a sweep (fix_fails): the roundings up to the
// end tile of 32 bins, sqrt(n) units, against 16 roundings of FP64 to the root
// sum of squares of the products before that tile, for every moment. On random
// events (noise, signal, both; 10 or 20 Hz; one bin up to 2^12 times too large;
// host emulation against 128 bits, 12 000 sweeps) the moments' errors are then
// 0.5 times FP64's in the median and 2.7 times at most (mean of the ten); past
// the line the ratio grows with it, without bound. Sweeps that end before the bin fix_from of the event (the last
// failure, at least the first tile, whose bins nothing precedes) take the FP64
// sweep: noise from 20 Hz has no other failure, noise from 10 Hz, where the data
// rise by 2^5 within a block, some in the first block. Data that no scale fits
// keep the FP64 sweep throughout.
#pragma once
#include <cstdint>
#include <cstring>

#include "common.cuh"

namespace sharpy {

// Tile of 32 bins, lane = bin, 16 bytes a bin and quad:
//   0-8  {B_j in FP64, its limbs h, l}   9-11  E_a: {re h, re l, im h, im l}
constexpr int kFixDet = 3;                // detectors at most
constexpr int kFixQuads = kNBasis + kFixDet;
constexpr int kFixBins = 256;             // bins that share their scales: 8 lane iterations
constexpr int64_t kFixMaxBins = 1 << 24;  // 3.2 GB of tiles; more bins keep the FP64 sweep
constexpr int kFixNever = 0x7fffffff;     // fix_from of data that no scale fits
constexpr int kFixTrig = 1024;            // points of the carrier table, {cos h, l, sin h, l} to 2^-62

// A block's scales: moment (a, j) = scale[a * kNMom + j] x integer sum.
struct FixBlock {
  double scale[kFixDet * kNMom];
  int one;  // high limb of the basis value 1
};

// Whether a sweep that ends in tile t of a block fails: `unit` of the block's
// moment, `sq` the sum of squares of its products in all bins before the tile,
// which must reach fix_need.
__host__ __device__ __forceinline__ double fix_need(double unit, int t) {
  const double u = unit * 0x1p49;  // a unit in 16 roundings of FP64 to 1
  return u * u * (double)(kTileBins * (t + 1));
}
__host__ __device__ __forceinline__ bool fix_fails(double unit, int t, double sq) { return !(fix_need(unit, t) <= sq); }

struct Limbs {
  int h, l;
};
// c + a b, one instruction: from the plain expression the compiler makes a
// product and a 64-bit addition (4.3 against 6.7 cycles)
__host__ __device__ __forceinline__ int64_t fix_mad(int a, int b, int64_t c) {
#ifdef __CUDA_ARCH__
  int64_t r;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
  return r;
#else
  return c + (int64_t)a * b;
#endif
}
__host__ __device__ __forceinline__ int fix_hi(int64_t x) { return (int)((uint64_t)x >> 32); }
__host__ __device__ __forceinline__ Limbs fix_limbs(int64_t v) {
  const uint32_t l = (uint32_t)(uint64_t)v;
  return {(int)((uint32_t)((uint64_t)v >> 32) + (l >> 31)), (int)l};
}
// the same with l > -2^31 (the value may grow by one unit), so that both limbs can be negated
__host__ __device__ __forceinline__ Limbs fix_limbs_neg(int64_t v) {
  Limbs r = fix_limbs(v);
  r.l = r.l == INT32_MIN ? INT32_MIN + 1 : r.l;
  return r;
}
constexpr int64_t kFixHalf = 1LL << 31;
// c + (a b) / 2^64, rounded; |a b| < 2^125
__host__ __device__ __forceinline__ int64_t fix_mulhi(Limbs a, Limbs b) {
  const int64_t x = fix_mad(a.l, b.h, fix_mad(a.h, b.l, kFixHalf));
  return fix_mad(a.h, b.h, fix_hi(x));
}
__host__ __device__ __forceinline__ uint32_t fix_umulhi(uint32_t a, uint32_t b) {
  return (uint32_t)(((uint64_t)a * b) >> 32);
}
// shifts by any unsigned count (0 from 64 on)
__host__ __device__ __forceinline__ uint64_t fix_shl(uint64_t v, uint32_t n) {
#ifdef __CUDA_ARCH__
  uint64_t r;
  asm("shl.b64 %0, %1, %2;" : "=l"(r) : "l"(v), "r"(n));
  return r;
#else
  return n > 63 ? 0 : v << n;
#endif
}
__host__ __device__ __forceinline__ uint64_t fix_shr(uint64_t v, uint32_t n) {
#ifdef __CUDA_ARCH__
  uint64_t r;
  asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(v), "r"(n));
  return r;
#else
  return n > 63 ? 0 : v >> n;
#endif
}
__host__ __device__ __forceinline__ uint64_t fix_bits(double x) {
#ifdef __CUDA_ARCH__
  return (uint64_t)__double_as_longlong(x);
#else
  uint64_t b;
  std::memcpy(&b, &x, 8);
  return b;
#endif
}

// P mod 1 in units of 2^-64 (P finite; exact but for bits below 2^-64)
__host__ __device__ __forceinline__ uint64_t fix_frac(double P) {
  const uint64_t b = fix_bits(P);
  const int e = (int)(b >> 52) & 0x7ff;
  const uint64_t m = (b << 11) | (1ULL << 63);  // |P| = m 2^(e - 1086)
  const uint64_t u = fix_shl(m, (uint32_t)(e - 1022)) | fix_shr(m, (uint32_t)(1022 - e));  // one of the two is 0, or both are m
  return (int64_t)b < 0 ? 0 - u : u;
}

// Carrier table index of the fraction u, and the rest of the angle:
// d = (pi / 1024) y, |y| <= 1, returned as y 2^62.
__host__ __device__ __forceinline__ int fix_index(uint64_t u) {
  return (int)(((uint32_t)(u >> 32) + 0x200000u) >> 22);
}
__host__ __device__ __forceinline__ int64_t fix_rest(uint64_t u) { return (int64_t)(u << 10) >> 1; }

// kappa = (pi / 1024)^2
constexpr double kFixKappa = (kPi / 1024.0) * (kPi / 1024.0);
constexpr int64_t kFixG0 = 226375608064910089LL;  // 2^56 pi
constexpr uint32_t kFixA1 = (uint32_t)(562949953421312.0 * kPi * kFixKappa / 6.0 + 0.5);                 // 2^49 pi kappa / 6
constexpr uint32_t kFixA2 = (uint32_t)(1125899906842624.0 * kPi * kFixKappa * kFixKappa / 120.0 + 0.5);  // 2^50 pi kappa^2 / 120
constexpr int64_t kFixH0 = (int64_t)(147573952589676412928.0 * kFixKappa + 0.5);                         // 2^67 kappa
constexpr uint32_t kFixB1 = (uint32_t)(147573952589676412928.0 * kFixKappa * kFixKappa / 6.0 + 0.5);     // 2^68 kappa^2 / 12

// sin d and cos d - 1 in units of 2^-64:
//   sin d     = (pi / 1024) y (1 - kappa y^2 / 6 + kappa^2 y^4 / 120)   (next term 2^-70)
//   cos d - 1 = -(kappa y^2 / 2) (1 - kappa y^2 / 12)                   (next term 2^-59.6)
// The brackets' corrections, 2^-19 and below, need y^2 to 31 bits only.
__host__ __device__ __forceinline__ void fix_small(int64_t rest, int64_t* s, int64_t* c1) {
  const Limbs v = fix_limbs(rest);
  const int64_t x = fix_mad(v.h, v.l, kFixHalf);
  const int64_t y2 = fix_mad(v.h, v.h, 2 * (int64_t)fix_hi(x));  // y^2 2^60, never negative
  const uint32_t Y = (uint32_t)((uint64_t)y2 >> 29);               // y^2 2^31
  const uint32_t t = fix_umulhi(Y, kFixA1 - fix_umulhi(Y, kFixA2));
  *s = fix_mulhi(v, fix_limbs(kFixG0 - ((int64_t)t << 8)));
  *c1 = fix_mulhi(fix_limbs(y2), fix_limbs((int64_t)fix_umulhi(Y, kFixB1) - kFixH0));
}

// z = E e^{-i 2 pi u} / 4 (E's units): E's limbs (re, im), the table's point,
// then the small rotation.
__host__ __device__ __forceinline__ void fix_carrier(uint64_t u, int4 E, int4 T, int64_t* zr, int64_t* zi) {
  int64_t s64, c64;
  fix_small(fix_rest(u), &s64, &c64);
  const Limbs s = fix_limbs_neg(s64), c = fix_limbs(c64);
  // w = E (C - i S) / 4
  int64_t x = fix_mad(E.w, T.z, fix_mad(E.z, T.w, fix_mad(E.y, T.x, fix_mad(E.x, T.y, kFixHalf))));
  const int64_t wr = fix_mad(E.z, T.z, fix_mad(E.x, T.x, fix_hi(x)));
  x = fix_mad(-E.y, T.z, fix_mad(-E.x, T.w, fix_mad(E.w, T.x, fix_mad(E.z, T.y, kFixHalf))));
  const int64_t wi = fix_mad(-E.x, T.z, fix_mad(E.z, T.x, fix_hi(x)));
  // z = w (cos d - i sin d)
  const Limbs r = fix_limbs(wr), i = fix_limbs(wi);
  x = fix_mad(i.l, s.h, fix_mad(i.h, s.l, fix_mad(r.l, c.h, fix_mad(r.h, c.l, kFixHalf))));
  *zr = fix_mad(i.h, s.h, fix_mad(r.h, c.h, wr + fix_hi(x)));
  x = fix_mad(r.l, -s.h, fix_mad(r.h, -s.l, fix_mad(i.l, c.h, fix_mad(i.h, c.l, kFixHalf))));
  *zi = fix_mad(r.h, -s.h, fix_mad(i.h, c.h, wi + fix_hi(x)));
}

// acc + (z B) / 2^64, rounded, + 2^31: the offset makes the cross products' high
// word unsigned, which saves its sign extension (14 against 16.5 cycles a
// moment); a sum of n terms starts at fix_start(n).
constexpr uint64_t kFixBias = 1ULL << 63;
__host__ __device__ __forceinline__ int64_t fix_start(int n) { return -((int64_t)n << 31); }
__host__ __device__ __forceinline__ int64_t fix_moment(Limbs z, int bh, int bl, int64_t acc) {
  const int64_t x = fix_mad(z.l, bh, fix_mad(z.h, bl, (int64_t)(kFixBias + (uint64_t)kFixHalf)));
  return acc + fix_mad(z.h, bh, (int64_t)((uint64_t)x >> 32));
}
// the same for a basis value of a high limb alone
__host__ __device__ __forceinline__ int64_t fix_moment1(Limbs z, int bh, int64_t acc) {
  const int64_t x = fix_mad(z.l, bh, (int64_t)(kFixBias + (uint64_t)kFixHalf));
  return acc + fix_mad(z.h, bh, (int64_t)((uint64_t)x >> 32));
}

}  // namespace sharpy
