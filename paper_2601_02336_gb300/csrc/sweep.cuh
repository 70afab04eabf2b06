// The per-bin sweep: one warp accumulates the moments of one particle.
//
// Lane l visits bins k = l, l+32, ... <= k_ISCO, in tiles of 32 bins (common.cuh,
// fixed.cuh; the FP64 sweep reads SoA tables).
// Per bin the phase polynomial sum_j alpha_j B_j(f_k) + c0 is shared by all
// detectors; per detector it adds f_k tau_a, reduces mod 1 turn, forms the
// carrier e^{-i Psi}, multiplies the pre-whitened data E_ak and accumulates
// Z_a (and, for the gradient, Y_aj = sum z B_j).
//
//   SHARPY_FP64  : the phase in FP64; carrier, data product and moments in
//                  64-bit fixed point, or, for the data and ends where that
//                  would lose bits (fixed.cuh), FP64 throughout (reduction
//                  Psi - rint(Psi); sincospi).
//   SHARPY_MIXED_SPLIT : as SHARPY_MIXED, but the phase polynomial is built
//                  from hi/lo FP32 splits of alpha_j, tau_a and B_j(f_k):
//                  each product's integer turns are removed exactly (FMA error
//                  term kept), the fraction stays in [-1/2, 1/2]; no FP64 in
//                  the bin loop (worst-case phase error ~3e-7 turns).
//   SHARPY_MIXED : the post-Newtonian terms that carry the large phase
//                  (x^5, x^3, x^2, ln f) accumulated in FP64 on top of the
//                  offset 1.5 * 2^20 turns, whose low mantissa word is their
//                  fractional turn in 2^-32 units; the four terms below ~8
//                  turns (x, y, y ln f, y^2) in FP32 pairs as in the split
//                  path, added in 32-bit fixed point; the delay term f tau_a
//                  of each detector in FP32 from hi/lo splits (exact FMA error
//                  term, fraction added in 32-bit fixed point); FP32 sincos,
//                  carrier and moments. Per-lane FP32 partial sums are flushed
//                  every kFlush iterations through a fixed-order warp tree
//                  into compensated FP32 outer accumulators (blocked pairwise
//                  summation).
#pragma once
#include "fixed.cuh"
#include "physics.cuh"

namespace sharpy {

constexpr int kFlush = 64;  // lane iterations per block
// Long sweeps are cut into chunks of kFlush lane iterations (2048 bins) dealt
// to kStreams streams (chunk c to stream c mod kStreams); a stream's result
// does not depend on which warp computes it, and streams are merged in a fixed
// order, so any number of warps per particle gives the same moments.
constexpr int kChunkBins = kFlush * 32;
constexpr int kStreams = 8;
static_assert(kChunkBins % kFixBins == 0, "chunks are whole blocks of the fixed-point scales");

template <int NDET, bool GRAD>
struct MomCount {
  static constexpr int value = GRAD ? NDET * kNMom * 2 : NDET * 2;
};

// Index of moment (a, j, ri) in the full layout.
__device__ __forceinline__ int mom_index(int a, int j, int ri) { return (a * kNMom + j) * 2 + ri; }

template <int NDET, bool GRAD>
__device__ __forceinline__ int acc_to_mom(int i) {
  if (GRAD) return i;
  return mom_index(i / 2, 9, i & 1);
}

// Warp reduce-scatter of NP per-lane values (NP a power of two): at each
// butterfly level a lane keeps one half of its values and sends the other
// half to its partner, so the 32-lane sums of all NP values take
// NP/2 + NP/4 + ... shuffles instead of 5 NP. Fixed pairing: deterministic.
// Afterwards, for NP >= 32, lane l holds the sums of values
// l (NP/32) ... l (NP/32) + NP/32 - 1 in v[0 .. NP/32); for NP < 32 the lanes
// of each group of 32/NP consecutive lanes all hold the sum of value
// l / (32/NP) in v[0].
template <int N, int OFF, class T = float>
struct ReduceScatter {
  static __device__ __forceinline__ void run(T* v, int lane) {
    constexpr int H = N / 2;
    const bool up = (lane & OFF) != 0;
#pragma unroll
    for (int j = 0; j < H; ++j) {
      const T send = up ? v[j] : v[j + H];
      const T keep = up ? v[j + H] : v[j];
      v[j] = keep + __shfl_xor_sync(0xffffffffu, send, OFF);
    }
    ReduceScatter<H, OFF / 2, T>::run(v, lane);
  }
};
template <int OFF, class T>
struct ReduceScatter<1, OFF, T> {
  static __device__ __forceinline__ void run(T* v, int) {
#pragma unroll
    for (int o = OFF; o >= 1; o >>= 1) v[0] += __shfl_xor_sync(0xffffffffu, v[0], o);
  }
};
template <int N, class T>
struct ReduceScatter<N, 0, T> {
  static __device__ __forceinline__ void run(T*, int) {}
};
template <class T>
struct ReduceScatter<1, 0, T> {
  static __device__ __forceinline__ void run(T*, int) {}
};

template <int NACC>
struct FlushShape {
  static constexpr int NP = NACC <= 2 ? 2 : NACC <= 4 ? 4 : NACC <= 8 ? 8 : NACC <= 16 ? 16 : NACC <= 32 ? 32 : 64;
  static constexpr int KEEP = NP >= 32 ? NP / 32 : 1;  // sums held per lane
  static __device__ __forceinline__ int index(int lane, int t) { return NP >= 32 ? lane * KEEP + t : lane / (32 / NP); }
  static __device__ __forceinline__ bool owner(int lane) { return NP >= 32 || lane % (32 / NP) == 0; }
};

// Flush per-lane FP32 partials into the lane-distributed outer accumulators:
// each block sum (reduce-scatter above) is added with an error-free two-sum,
// so the outer sums carry ~48 bits without FP64 arithmetic.
template <int NACC>
__device__ __forceinline__ void flush(float* acc, float* hi, float* lo, int lane) {
  using F = FlushShape<NACC>;
  static_assert(NACC <= 64, "at most 64 moments per lane");
  float v[F::NP];
#pragma unroll
  for (int i = 0; i < F::NP; ++i) v[i] = i < NACC ? acc[i] : 0.0f;
  ReduceScatter<F::NP, 16>::run(v, lane);
#pragma unroll
  for (int t = 0; t < F::KEEP; ++t) {
    const float s = hi[t] + v[t];
    const float bp = s - hi[t];
    lo[t] += (hi[t] - (s - bp)) + (v[t] - bp);
    hi[t] = s;
  }
#pragma unroll
  for (int i = 0; i < NACC; ++i) acc[i] = 0.0f;
}

// Magic constant for exact round-to-nearest of |x| < 2^22 in FP32.
constexpr float kRound32 = 12582912.0f;  // 1.5 * 2^23

// x - rint(x) for |x| < 2^22, exact (explicit roundings: no contraction).
__device__ __forceinline__ float frac_turn(float x) {
  return __fsub_rn(x, __fsub_rn(__fadd_rn(x, kRound32), kRound32));
}

// Two FP32 values in one 64-bit register pair. The packed instructions round
// each half as the scalar ones do and issue once for both, at the same FP32
// rate per lane: they pay where issue binds.
using f32x2 = unsigned long long;
__device__ __forceinline__ f32x2 pack2(float a, float b) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ f32x2 dup2(float a) { return pack2(a, a); }
__device__ __forceinline__ float2 unpack2(f32x2 v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
// frac_turn of both halves (odd: frac2(-x) = -frac2(x))
__device__ __forceinline__ f32x2 frac2(f32x2 x) {
  const f32x2 r = add2(add2(x, dup2(kRound32)), dup2(-kRound32));
  return fma2(r, dup2(-1.0f), x);
}

// A bin's quads: from the tiles in global memory, or from a block of tiles in
// shared memory. Both sweeps walk tiles of 32 bins, lane = bin, so a quad is one
// coalesced 16-byte load at a constant offset from the lane's pointer.
struct GlobalTile {
  const float4* at;  // quad 0 of the lane's bin
  __device__ __forceinline__ float4 quad(int i) const { return __ldg(at + i * kTileBins); }
  __device__ __forceinline__ ulonglong2 pair(int i) const {
    return __ldg(reinterpret_cast<const ulonglong2*>(at + i * kTileBins));
  }
};
struct StagedTile {
  const float4* at;
  __device__ __forceinline__ float4 quad(int i) const { return at[i * kTileBins]; }
  __device__ __forceinline__ ulonglong2 pair(int i) const {
    return *reinterpret_cast<const ulonglong2*>(at + i * kTileBins);
  }
};

// Per-lane moment sums of NDET detectors. Mixed sweep with the gradient: pairs
// in the tile's order, one packed FMA for two moments (per bin and detector 10
// issues instead of 20; its FP64 terms leave the FP32 pipe slack that the
// packed form's longer latency needs: 12.8 against 14.4 ms on 8192 vectors of
// the 259585-bin segment). Otherwise single sums: the split sweep, whose FP32
// pipe is the busier one, is faster with scalar FMAs (3.50 against 3.73 ms on
// 1824 vectors).
template <bool GRAD, int NDET, bool SPLIT>
struct MomAcc {
  float v[MomCount<NDET, GRAD>::value];
  __device__ __forceinline__ void zero() {
#pragma unroll
    for (int i = 0; i < MomCount<NDET, GRAD>::value; ++i) v[i] = 0.0f;
  }
  // adds the products of z = (zr, zi) with the bin's basis values b (tile pairs) and f, and z itself
  __device__ __forceinline__ void add(int a, float zr, float zi, const f32x2* b, float f) {
    if (GRAD) {
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float2 x = unpack2(b[i]);
        const int j0 = mom_index(a, tile_basis(SPLIT, 2 * i), 0), j1 = mom_index(a, tile_basis(SPLIT, 2 * i + 1), 0);
        v[j0] = fmaf(zr, x.x, v[j0]);
        v[j0 + 1] = fmaf(zi, x.x, v[j0 + 1]);
        v[j1] = fmaf(zr, x.y, v[j1]);
        v[j1 + 1] = fmaf(zi, x.y, v[j1 + 1]);
      }
      const int jf = mom_index(a, 8, 0);
      v[jf] = fmaf(zr, f, v[jf]);
      v[jf + 1] = fmaf(zi, f, v[jf + 1]);
      v[jf + 2] += zr;
      v[jf + 3] += zi;
    } else {
      v[a * 2] += zr;
      v[a * 2 + 1] += zi;
    }
  }
  __device__ __forceinline__ void get(float* out) const {
#pragma unroll
    for (int i = 0; i < MomCount<NDET, GRAD>::value; ++i) out[i] = v[i];
  }
};
template <int NDET>
struct MomAcc<true, NDET, false> {
  f32x2 m[NDET][2][kNMom / 2];  // pair 4: (f, 1)
  __device__ __forceinline__ void zero() {
#pragma unroll
    for (int a = 0; a < NDET; ++a)
#pragma unroll
      for (int i = 0; i < kNMom / 2; ++i) m[a][0][i] = m[a][1][i] = 0ULL;
  }
  __device__ __forceinline__ void add(int a, float zr, float zi, const f32x2* b, float f) {
    const f32x2 z[2] = {dup2(zr), dup2(zi)};
    const f32x2 f1 = pack2(f, 1.0f);
#pragma unroll
    for (int r = 0; r < 2; ++r) {
#pragma unroll
      for (int i = 0; i < 4; ++i) m[a][r][i] = fma2(z[r], b[i], m[a][r][i]);
      m[a][r][4] = fma2(z[r], f1, m[a][r][4]);  // the second half adds z itself
    }
  }
  __device__ __forceinline__ void get(float* out) const {
#pragma unroll
    for (int a = 0; a < NDET; ++a)
#pragma unroll
      for (int r = 0; r < 2; ++r)
#pragma unroll
        for (int i = 0; i < kNMom / 2; ++i) {
          const float2 x = unpack2(m[a][r][i]);
          out[mom_index(a, i < 4 ? tile_basis(false, 2 * i) : 8, r)] = x.x;
          out[mom_index(a, i < 4 ? tile_basis(false, 2 * i + 1) : 9, r)] = x.y;
        }
  }
};

// Adds the lane sums to the outer accumulators and clears them.
template <bool SPLIT, bool GRAD, int NDET>
__device__ __forceinline__ void flush_acc(MomAcc<GRAD, NDET, SPLIT>& acc, float* hi, float* lo, int lane) {
  constexpr int NACC = MomCount<NDET, GRAD>::value;
  float v[NACC];
  acc.get(v);
  flush<NACC>(v, hi, lo, lane);
  acc.zero();
}

// Per-particle constants of the sweep, in registers. The pairs follow the
// tile's order; n*: negated (a product p = a b is formed as -p, so that its FMA
// error term needs no negation).
template <int NDET, bool SPLIT>
struct MixedCoef {
  static constexpr int NP = SPLIT ? 4 : 2;  // pairs of terms in FP32 pairs
  f32x2 ah[NP], nah[NP], al[NP];
  f32x2 th2, nth2, tl2;  // delays of detectors 0 and 1
  float th, tl;          // delay of the odd detector
  float c0f;             // split: c0 mod 1 turn
  double alpha[4], s0;   // mixed: the large terms, c0 on the turn offset

  __device__ __forceinline__ explicit MixedCoef(const SweepCoef& sc) {
#pragma unroll
    for (int i = 0; i < NP; ++i) {
      const int j0 = tile_basis(SPLIT, 2 * i), j1 = tile_basis(SPLIT, 2 * i + 1);
      ah[i] = pack2(sc.ahi[j0], sc.ahi[j1]);
      nah[i] = pack2(-sc.ahi[j0], -sc.ahi[j1]);
      al[i] = pack2(sc.alo[j0], sc.alo[j1]);
    }
    constexpr int d1 = NDET > 1 ? 1 : 0;
    th2 = pack2(sc.thi[0], sc.thi[d1]);
    nth2 = pack2(-sc.thi[0], -sc.thi[d1]);
    tl2 = pack2(sc.tlo[0], sc.tlo[d1]);
    th = sc.thi[NDET - 1];
    tl = sc.tlo[NDET - 1];
    if (SPLIT) {
      c0f = sc.c0f;
    } else {
#pragma unroll
      for (int i = 0; i < 4; ++i) alpha[i] = sc.alpha[large_pn(i)];
      s0 = sc.c0 + kTurnOffset;
    }
  }
};

// One bin of the mixed (or split) sweep: its phase, carrier and moment
// updates, with the bin's quads from the loader ld (global memory or a
// shared-memory stage: the same values, so the same sums).
template <bool GRAD, int NDET, bool SPLIT, class L>
__device__ __forceinline__ void mixed_bin(const MixedCoef<NDET, SPLIT>& P, const L& ld,
                                          MomAcc<GRAD, NDET, SPLIT>& acc) {
  const float4 qf = ld.quad(tile_quad_f(SPLIT));  // f hi, f lo, E of detector 0
  const float4 qe = NDET > 1 ? ld.quad(tile_quad_f(SPLIT) + 1) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
  const ulonglong2 h0 = ld.pair(0), h1 = GRAD || SPLIT ? ld.pair(1) : make_ulonglong2(0ULL, 0ULL);
  const f32x2 b[4] = {h0.x, h0.y, h1.x, h1.y};
  const float f = qf.x, fl = qf.y;
  // the terms in FP32 pairs: p = ahi bhi is exact up to its FMA error term, its
  // integer turns are removed exactly; nf: minus the fractions, er: the error
  // and cross terms, of the pairs' halves
  constexpr int NP = MixedCoef<NDET, SPLIT>::NP;
  f32x2 nf[NP], er[NP];
#pragma unroll
  for (int i = 0; i < NP; i += 2) {
    const ulonglong2 l = ld.pair(2 + i / 2);
#pragma unroll
    for (int u = i; u < i + 2; ++u) {
      const f32x2 np = mul2(P.nah[u], b[u]);
      nf[u] = frac2(np);
      er[u] = fma2(P.ah[u], u == i ? l.x : l.y, fma2(P.al[u], b[u], fma2(P.ah[u], b[u], np)));
    }
  }
  float ang[NDET];
  const f32x2 ff = dup2(f), fll = dup2(fl), m1 = dup2(-1.0f);
  if constexpr (!SPLIT) {
    // the four terms that carry the large phase (Newtonian, 1PN, 1.5PN and
    // the 2.5PN logarithm: up to ~2e3 turns on the long segment) accumulated
    // in FP64 on the offset, whose low word is their fractional turn
    const ulonglong2 q0 = ld.pair(5), q1 = ld.pair(6);
    const unsigned long long q[4] = {q0.x, q0.y, q1.x, q1.y};
    double S = P.s0;
#pragma unroll
    for (int i = 0; i < 4; ++i) S = fma(P.alpha[i], __longlong_as_double((long long)q[i]), S);
    int turn_s = __double2loint(S);  // 2^-32 units
    // the four terms below ~8 turns (2PN, 3PN, its logarithm, 3.5PN): the
    // fractions summed pairwise in [-1/2, 1/2], then added to the FP64 part in
    // 32-bit fixed point
    const float2 n2 = unpack2(frac2(add2(nf[0], nf[1]))), e2 = unpack2(add2(er[0], er[1]));
    const float n = frac_turn(__fadd_rn(n2.x, n2.y));
    const float qs = frac_turn(__fsub_rn(__fadd_rn(e2.x, e2.y), n));
    turn_s += __float2int_rn(qs * 4294967296.0f);  // wraps mod 1 turn
    // f tau_a mod 1 from (thi + tlo)(fhi + flo): p = thi fhi is exact up to e
    // (FMA), the other products are below 2^-20 turn
    float qa[NDET];
    if constexpr (NDET > 1) {
      const f32x2 np = mul2(P.nth2, ff);
      const f32x2 e = fma2(P.th2, fll, fma2(P.tl2, ff, fma2(P.th2, ff, np)));
      const float2 x = unpack2(mul2(frac2(fma2(frac2(np), m1, e)), dup2(4294967296.0f)));
      qa[0] = x.x;
      qa[1] = x.y;
    }
    if constexpr (NDET != 2) {
      const float p = __fmul_rn(P.th, f);
      const float e = fmaf(P.th, fl, fmaf(P.tl, f, fmaf(P.th, f, -p)));
      qa[NDET - 1] = frac_turn(__fadd_rn(frac_turn(p), e)) * 4294967296.0f;
    }
#pragma unroll
    for (int a = 0; a < NDET; ++a) {
      const int turn = turn_s + __float2int_rn(qa[a]);  // wraps mod 1 turn
      ang[a] = (float)turn * 1.46291807926715968e-9f;    // 2 pi / 2^32
    }
  } else {
    // sum_j alpha_j B_j mod 1: the fractions summed pairwise, reduced to
    // [-1/2, 1/2] at every level (three levels instead of an eight-step
    // chain), the error and cross terms likewise pairwise in Sm; the tile's
    // pairs are (0, 2) + (1, 3) and (4, 6) + (5, 7)
    static_assert(kNPn == 8, "the pairwise tree below is written for eight basis terms");
    const float2 n03 = unpack2(frac2(add2(nf[0], nf[1]))), n47 = unpack2(frac2(add2(nf[2], nf[3])));
    const float2 e03 = unpack2(add2(er[0], er[1])), e47 = unpack2(add2(er[2], er[3]));
    const float n = __fadd_rn(frac_turn(__fadd_rn(n03.x, n03.y)), frac_turn(__fadd_rn(n47.x, n47.y)));
    const float F = frac_turn(__fsub_rn(P.c0f, n));
    const float Sm = __fadd_rn(__fadd_rn(e03.x, e03.y), __fadd_rn(e47.x, e47.y));
    if constexpr (NDET > 1) {
      const f32x2 np = mul2(P.nth2, ff);
      const f32x2 Sa = fma2(P.th2, fll, fma2(P.tl2, ff, add2(dup2(Sm), fma2(P.th2, ff, np))));
      const f32x2 Fa = frac2(fma2(frac2(np), m1, dup2(F)));
      const float2 x = unpack2(mul2(add2(Fa, Sa), dup2(6.28318530717958648f)));
      ang[0] = x.x;
      ang[1] = x.y;
    }
    if constexpr (NDET != 2) {
      const float p = __fmul_rn(P.th, f);
      float Sa = __fadd_rn(Sm, fmaf(P.th, f, -p));
      Sa = fmaf(P.th, fl, fmaf(P.tl, f, Sa));
      const float Fa = frac_turn(__fadd_rn(F, frac_turn(p)));
      ang[NDET - 1] = (Fa + Sa) * 6.28318530717958648f;
    }
  }
#pragma unroll
  for (int a = 0; a < NDET; ++a) {
    float sn, cs;
    __sincosf(ang[a], &sn, &cs);
    const float2 E = a == 0 ? make_float2(qf.z, qf.w) : a == 1 ? make_float2(qe.x, qe.y) : make_float2(qe.z, qe.w);
    // E e^{-i ang}, the contraction fixed
    const float zr = __fmaf_rn(E.x, cs, __fmul_rn(E.y, sn));
    const float zi = __fmaf_rn(E.y, cs, -__fmul_rn(E.x, sn));
    acc.add(a, zr, zi, b, f);
  }
}

// One stream of a mixed sweep: the chunks c = s, s + kStreams, ... of 2048
// bins (64 lane iterations: one FP32 block each) below k_ISCO, accumulated
// into this lane's compensated outer sums hi, lo (kept lane-distributed as
// the flush leaves them). Returns whether the stream had any bin.
template <bool GRAD, int NDET, bool SPLIT>
__device__ bool mixed_stream(const DevEvent& ev, const SweepCoef& sc, int s, float* hi, float* lo) {
  constexpr int NACC = MomCount<NDET, GRAD>::value;
  constexpr int NOUT = FlushShape<NACC>::KEEP;
  constexpr int TQ = tile_quads(SPLIT) * kTileBins;  // float4 per tile
  const int lane = threadIdx.x & 31;
  MomAcc<GRAD, NDET, SPLIT> acc;
  acc.zero();
#pragma unroll
  for (int i = 0; i < NOUT; ++i) hi[i] = lo[i] = 0.0f;
  const MixedCoef<NDET, SPLIT> P(sc);
  const float4* tiles = (SPLIT ? ev.tile_split : ev.tile_mixed) + lane;
  const int kend = sc.kisco;
  bool any = false;
  // Warp-uniform trip counts: lanes past k_ISCO idle but still join the flushes.
  for (int c = s; c * kChunkBins <= kend; c += kStreams) {
    any = true;
    const float4* at = tiles + (int64_t)c * kFlush * TQ;
    const int its = min(kFlush, (kend - c * kChunkBins) / 32 + 1);
    int k = c * kChunkBins + lane;
#pragma unroll 1
    for (int it = 0; it < its; ++it, k += 32, at += TQ)
      if (k <= kend) mixed_bin<GRAD, NDET, SPLIT>(P, GlobalTile{at}, acc);
    flush_acc<SPLIT>(acc, hi, lo, lane);
  }
  return any;
}

// Moments of one particle on one warp (the NUTS kernel's sweep). A sweep of
// one chunk (k_ISCO < 2048: every BBH workload here) is its single stream:
// the moments are hi + lo. Longer sweeps take the kStreams streams in order
// and add each stream's hi + lo in FP64: the result the likelihood kernel
// gets from the same streams spread over several warps, bit for bit.
template <bool GRAD, int NDET, bool SPLIT>
__device__ void sweep_mixed(const DevEvent& ev, const SweepCoef& sc, float* mom) {
  constexpr int NACC = MomCount<NDET, GRAD>::value;
  constexpr int NOUT = FlushShape<NACC>::KEEP;
  const int lane = threadIdx.x & 31;
  float hi[NOUT], lo[NOUT];
  float out[NOUT];
  if (sc.kisco < kChunkBins) {
    mixed_stream<GRAD, NDET, SPLIT>(ev, sc, 0, hi, lo);
#pragma unroll
    for (int t = 0; t < NOUT; ++t) out[t] = hi[t] + lo[t];
  } else {
    double tot[NOUT];
#pragma unroll
    for (int t = 0; t < NOUT; ++t) tot[t] = 0.0;
    for (int st = 0; st < kStreams; ++st) {
      if (!mixed_stream<GRAD, NDET, SPLIT>(ev, sc, st, hi, lo)) break;
#pragma unroll
      for (int t = 0; t < NOUT; ++t) tot[t] += (double)hi[t] + (double)lo[t];
    }
#pragma unroll
    for (int t = 0; t < NOUT; ++t) out[t] = (float)tot[t];
  }
  if (FlushShape<NACC>::owner(lane)) {
#pragma unroll
    for (int t = 0; t < NOUT; ++t) {
      const int idx = FlushShape<NACC>::index(lane, t);
      if (idx < NACC) mom[acc_to_mom<NDET, GRAD>(idx)] = out[t];
    }
  }
}

// One stream of the FP64 path in fixed point (chunks c = s, s + kStreams, ...
// of 2048 bins below k_ISCO): the integer sums of each block of 256 bins go
// through the warp reduce-scatter exactly (~500 instructions against the
// block's ~4000), are rounded to FP64 once and added to the stream's; lane l
// holds its sums in v_out. Returns whether the stream had any bin.
// Per bin and detector 4 FP64 instructions and ~170 integer ones against ~50
// FP64 ones of fp64_stream (60 cycles each): see fixed.cuh.
template <bool GRAD, int NDET>
__device__ bool fixed_stream(const DevEvent& ev, const SweepCoef& sc, int s, double* v_out) {
  constexpr int NACC = MomCount<NDET, GRAD>::value;
  using F = FlushShape<NACC>;
  const int lane = threadIdx.x & 31;
  double al[kNPn];
#pragma unroll
  for (int j = 0; j < kNPn; ++j) al[j] = sc.alpha[j];
#pragma unroll
  for (int t = 0; t < F::KEEP; ++t) v_out[t] = 0.0;
  const int kend = sc.kisco;
  uint32_t top = 0;  // largest exponent of a phase: a non-finite one has no fraction
  bool any = false;
  // blocks of the chunks s, s + kStreams, ...
  constexpr int kPer = kChunkBins / kFixBins;
#pragma unroll 1
  for (int g = s * kPer; g * kFixBins <= kend; g += (g % kPer == kPer - 1 ? (kStreams - 1) * kPer : 0) + 1) {
    any = true;
    int64_t acc[NACC];
    const int kstop = min(kend, g * kFixBins + kFixBins - 1), k0 = g * kFixBins + lane;
    const int64_t start = fix_start(k0 <= kstop ? (kstop - k0) / 32 + 1 : 0);
#pragma unroll
    for (int i = 0; i < NACC; ++i) acc[i] = start;
    const FixBlock* fb = ev.fix_block + g;
    const int one = __ldg(&fb->one);
    const int4* at = ev.tile_fix + (int64_t)g * (kFixBins * kFixQuads) + lane;
#pragma unroll 1
    for (int k = k0; k <= kstop; k += 32, at += kFixQuads * kTileBins) {
      double S = sc.c0, f = 0.0;
      int bh[kNBasis], bl[kNBasis];
#pragma unroll
      for (int j = 0; j < kNBasis; ++j) {
        const int4 q = __ldg(at + j * kTileBins);
        const double b = __hiloint2double(q.y, q.x);
        bh[j] = q.z;
        bl[j] = q.w;
        if (j < kNPn)
          S = fma(al[j < kNPn ? j : 0], b, S);
        else
          f = b;
      }
#pragma unroll
      for (int a = 0; a < NDET; ++a) {
        const double P = fma(f, sc.tau[a], S);
        top = max(top, (uint32_t)__double2hiint(P) & 0x7ff00000u);
        const uint64_t u = fix_frac(P);
        int64_t zr, zi;
        fix_carrier(u, __ldg(at + (kNBasis + a) * kTileBins), __ldg(ev.fix_trig + fix_index(u)), &zr, &zi);
        const Limbs r = fix_limbs(zr), i = fix_limbs(zi);
        if (GRAD) {
#pragma unroll
          for (int j = 0; j < kNBasis; ++j) {
            int64_t* m = acc + (a * kNMom + j) * 2;
            m[0] = fix_moment(r, bh[j], bl[j], m[0]);
            m[1] = fix_moment(i, bh[j], bl[j], m[1]);
          }
        }
        int64_t* m = acc + (GRAD ? (a * kNMom + 9) * 2 : a * 2);
        m[0] = fix_moment1(r, one, m[0]);
        m[1] = fix_moment1(i, one, m[1]);
      }
    }
    int64_t v[F::NP];
#pragma unroll
    for (int i = 0; i < F::NP; ++i) v[i] = i < NACC ? acc[i] : 0;
    ReduceScatter<F::NP, 16, int64_t>::run(v, lane);
#pragma unroll
    for (int t = 0; t < F::KEEP; ++t) {
      const int i = F::index(lane, t);
      if (i < NACC) v_out[t] = fma((double)v[t], __ldg(fb->scale + (GRAD ? i / 2 : i / 2 * kNMom + 9)), v_out[t]);
    }
  }
  if (__any_sync(0xffffffffu, top >= 0x7ff00000u)) {
#pragma unroll
    for (int t = 0; t < F::KEEP; ++t) v_out[t] = NAN;
  }
  return any;
}

// One stream of the FP64 sweep (chunks c = s, s + kStreams, ... of 2048 bins
// below k_ISCO): per-lane FP64 sums, then the warp reduce-scatter (the same
// pairing as a butterfly sum per moment, with NP/2 + NP/4 + ... FP64 adds per
// lane instead of 5 NP); lane l holds its sums in v. Returns whether the
// stream had any bin.
template <bool GRAD, int NDET>
__device__ bool fp64_stream(const DevEvent& ev, const SweepCoef& sc, int s, double* v_out) {
  constexpr int NACC = MomCount<NDET, GRAD>::value;
  const int lane = threadIdx.x & 31;
  const int64_t K = ev.n_bins;
  double acc[NACC];
#pragma unroll
  for (int i = 0; i < NACC; ++i) acc[i] = 0.0;
  double al[kNPn];
#pragma unroll
  for (int j = 0; j < kNPn; ++j) al[j] = sc.alpha[j];
  const int kend = sc.kisco;
  bool any = false;
  for (int c = s; c * kChunkBins <= kend; c += kStreams) {
    any = true;
    const int kstop = min(kend, c * kChunkBins + kChunkBins - 1);
    for (int k = c * kChunkBins + lane; k <= kstop; k += 32) {
      double S = sc.c0;
#pragma unroll
      for (int j = 0; j < kNPn; ++j) S = fma(al[j], ev.b64[(int64_t)j * K + k], S);
      const double f = ev.b64[(int64_t)8 * K + k];
      double bf[kNBasis];
      if (GRAD) {
#pragma unroll
        for (int j = 0; j < kNBasis; ++j) bf[j] = ev.b64[(int64_t)j * K + k];
      }
#pragma unroll
      for (int a = 0; a < NDET; ++a) {
        const double P = fma(f, sc.tau[a], S);
        const double r = P - rint(P);
        double sn, cs;
        sincospi(2.0 * r, &sn, &cs);
        const double2 E = ev.e64[(int64_t)a * K + k];
        const double zr = E.x * cs + E.y * sn;
        const double zi = E.y * cs - E.x * sn;
        if (GRAD) {
#pragma unroll
          for (int j = 0; j < kNBasis; ++j) {
            acc[(a * kNMom + j) * 2] += zr * bf[j];
            acc[(a * kNMom + j) * 2 + 1] += zi * bf[j];
          }
          acc[(a * kNMom + 9) * 2] += zr;
          acc[(a * kNMom + 9) * 2 + 1] += zi;
        } else {
          acc[a * 2] += zr;
          acc[a * 2 + 1] += zi;
        }
      }
    }
  }
  using F = FlushShape<NACC>;
  double v[F::NP];
#pragma unroll
  for (int i = 0; i < F::NP; ++i) v[i] = i < NACC ? acc[i] : 0.0;
  ReduceScatter<F::NP, 16, double>::run(v, lane);
#pragma unroll
  for (int t = 0; t < F::KEEP; ++t) v_out[t] = v[t];
  return any;
}

// One stream of the FP64 path, in the arithmetic that the event's data allow
// for a sweep of this length (fixed.cuh).
template <bool GRAD, int NDET>
__device__ bool wide_stream(const DevEvent& ev, const SweepCoef& sc, int s, double* v_out) {
  return ev.tile_fix && sc.kisco >= *ev.fix_from ? fixed_stream<GRAD, NDET>(ev, sc, s, v_out) : fp64_stream<GRAD, NDET>(ev, sc, s, v_out);
}

// FP64 moments of one particle on one warp; streams as in sweep_mixed (a
// sweep below 2048 bins is its single stream).
template <bool GRAD, int NDET>
__device__ void sweep_fp64(const DevEvent& ev, const SweepCoef& sc, double* mom) {
  constexpr int NACC = MomCount<NDET, GRAD>::value;
  using F = FlushShape<NACC>;
  const int lane = threadIdx.x & 31;
  double v[F::KEEP], tot[F::KEEP];
  if (sc.kisco < kChunkBins) {
    wide_stream<GRAD, NDET>(ev, sc, 0, tot);
  } else {
#pragma unroll
    for (int t = 0; t < F::KEEP; ++t) tot[t] = 0.0;
    for (int st = 0; st < kStreams; ++st) {
      if (!wide_stream<GRAD, NDET>(ev, sc, st, v)) break;
#pragma unroll
      for (int t = 0; t < F::KEEP; ++t) tot[t] += v[t];
    }
  }
  if (F::owner(lane)) {
#pragma unroll
    for (int t = 0; t < F::KEEP; ++t) {
      const int idx = F::index(lane, t);
      if (idx < NACC) mom[acc_to_mom<NDET, GRAD>(idx)] = tot[t];
    }
  }
}

// Moment storage type of each path.
template <int PREC>
struct MomType {
  using type = float;
};
template <>
struct MomType<SHARPY_FP64> {
  using type = double;
};

template <int PREC, bool GRAD, int NDET>
__device__ __forceinline__ void sweep(const DevEvent& ev, const SweepCoef& sc, typename MomType<PREC>::type* mom) {
  if constexpr (PREC == SHARPY_FP64)
    sweep_fp64<GRAD, NDET>(ev, sc, mom);
  else
    sweep_mixed<GRAD, NDET, PREC == SHARPY_MIXED_SPLIT>(ev, sc, mom);
}

}  // namespace sharpy
