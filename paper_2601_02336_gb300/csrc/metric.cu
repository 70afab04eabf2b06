// Per-particle mass matrices (Sec. 5, "Exploitation of local geometry"): at
// the start of a stage every particle gets M = beta F(theta) + prior Hessian +
// 12 / width^2 on the diagonal, F the Fisher information of the Whittle
// likelihood (the Gauss-Newton part of -d^2 ln L, positive semi-definite), and
// keeps it through the stage's mutation.
//
// With the Newtonian amplitude every strain derivative is the strain times a
// function of frequency that is linear in the phase basis:
//   d_j h_a(f) = (d_j G_a - 2 pi i G_a phi_aj(f)) A(f) e^{-i Psi_a(f)},
//   phi_aj(f) = sum_m D_ajm B_m(f),  B = {x^5, x^3, x^2, x, ln f, y, y ln f, y^2, f, 1},
// so <d_j h_a | d_k h_a> needs only prefix sums over the bins below f_ISCO of
// W = w f^-7/3 times 1, B_m and B_m B_n (tables built once per event):
//   F_jk = sum_a Re(conj(dG_j) dG_k) P0 - 2 pi [Im(conj(G) dG_j) (D_k . P1)
//          + Im(conj(G) dG_k) (D_j . P1)] + 4 pi^2 |G|^2 D_j P2 D_k.
// FP64 throughout (the entries span many decades in physical units).
#include <cmath>
#include <vector>

#include "context.cuh"
#include "physics.cuh"
#include "quotient.cuh"

using namespace sharpy;

namespace sharpy {

constexpr int kNB = kNBasis + 1;  // basis incl. the constant
constexpr int kNPair = kNBasis * (kNBasis + 1) / 2;

__device__ __forceinline__ int pair_index(int m, int n) {  // m <= n < kNBasis
  return m * kNBasis - m * (m - 1) / 2 + (n - m);
}

// One CTA of kMetWarps warps forms the matrices of 32 particles, lane =
// particle in every warp: FP64 issues one warp instruction per 64 cycles and
// SM sub-partition here whatever its active lanes, so every instruction
// carries 32 particles and the independent parts of a particle's work go to
// the four sub-partitions at once (prologue halves and detectors, then the
// rows, columns and entries of the factorisations). The matrices live in
// shared memory, [entry][particle] in rows of kMetPad words: a warp's access
// to one entry and the coalesced copy-out of whole matrices are both free of
// bank conflicts. Bound by FP64 issue: 11-D, three detectors, 2048 particles
// (64 CTAs, each phase's chain on its own sub-partition) 141 us, 16384
// particles 271 us; one thread per particle with dense products, divisions and
// the matrices in local memory took 533 and 550 us.
constexpr int kMetWarps = 4;
constexpr int kMetPart = 32;      // particles per CTA
constexpr int kMetPad = kMetPart + 1;
constexpr int kTri = SHARPY_NPHYS * (SHARPY_NPHYS + 1) / 2;  // entries of a lower triangle

__host__ __device__ constexpr int tri(int i, int j) { return i * (i + 1) / 2 + j; }  // i >= j

struct MetricShared {
  double M[kTri][kMetPad];  // Fisher matrix, then M, then its Cholesky factor (lower)
  union {
    struct {
      SweepCoef sc[kMetPart];
      EpiCoef<double> ec[kMetPart];
    } pro;
    struct {
      double Ci[kTri][kMetPad];  // C^-1
      double Mi[kTri][kMetPad];  // M^-1, then its Cholesky factor
    } la;
  };
  double diag[SHARPY_NPHYS][kMetPad];  // M's diagonal (kept for the fallback)
  double rc[SHARPY_NPHYS][kMetPad];    // 1 / C_jj
  double piv[kMetPad], rpiv[kMetPad];
  unsigned ok[2];                      // per particle: the factorisation of M, of M^-1 went through
};

// The phase derivative's basis coefficients D_j: parameters 0..3 (masses and
// spins) have the eight post-Newtonian terms and the constant, phi_c the
// constant, t_c, ra and sin dec the term linear in f; the others none. dG_j is
// zero but for M_c, d_L and the response's parameters. The products below
// leave out the terms that are zero: a third of the FP64 operations of the
// dense form, with the same roundings in the rest.
__host__ __device__ constexpr bool has_pn(int j) { return j < 4; }
__host__ __device__ constexpr bool has_const(int j) { return j == SHARPY_PHIC; }
__host__ __device__ constexpr bool has_f(int j) { return j == SHARPY_RA || j == SHARPY_SINDEC || j == SHARPY_TC; }
__host__ __device__ constexpr bool has_phase(int j) { return has_pn(j) || has_const(j) || has_f(j); }
__host__ __device__ constexpr bool has_amp(int j) {
  return j == SHARPY_MC || j == SHARPY_DL || j == SHARPY_COSI || j == SHARPY_PSI || j == SHARPY_RA || j == SHARPY_SINDEC;
}

// F's lower triangle (physical parameters; v[tri(l, j)], l >= j) of detector a.
__device__ __forceinline__ void fisher_detector(const DevEvent& ev, const SweepCoef& sc, const EpiCoef<double>& ec,
                                                int a, double (&v)[kTri]) {
  const int64_t K = ev.n_bins;
  const int k = sc.kisco;
  const double P0 = ev.pref[(int64_t)a * K + k];
  const double A0 = ec.A0;
  const double Gr = A0 * ec.cre[a], Gi = A0 * ec.cim[a];
  double dGr[SHARPY_NPHYS], dGi[SHARPY_NPHYS], dp1[SHARPY_NPHYS], img[SHARPY_NPHYS];
  dGr[SHARPY_MC] = Gr * ec.rel_mc;
  dGi[SHARPY_MC] = Gi * ec.rel_mc;
  dGr[SHARPY_DL] = Gr * ec.rel_dl;
  dGi[SHARPY_DL] = Gi * ec.rel_dl;
  constexpr int resp[4] = {SHARPY_COSI, SHARPY_PSI, SHARPY_RA, SHARPY_SINDEC};
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    dGr[resp[r]] = A0 * ec.dcre[a][r];
    dGi[resp[r]] = A0 * ec.dcim[a][r];
  }
  // D_j: the PN parameters' rows d[p][0..8) with the constant's dc[p]; one
  // coefficient of f or of the constant for the others
  double d[4][kNPn], dc[4];
#pragma unroll
  for (int p = 0; p < 4; ++p) {
#pragma unroll
    for (int b = 0; b < kNPn; ++b) d[p][b] = ec.dalpha[b][p];
    dc[p] = ec.dc0[p];
  }
  auto single = [&](int j) {
    return j == SHARPY_PHIC ? -1.0 / kTwoPi : j == SHARPY_TC ? 1.0 : j == SHARPY_RA ? ec.dtau[a][0] : ec.dtau[a][1];
  };
  auto P1 = [&](int m) { return __ldg(ev.p1 + ((int64_t)a * kNBasis + m) * K + k); };
  auto P2 = [&](int m, int n) {
    return __ldg(ev.p2 + ((int64_t)a * kNPair + (m <= n ? pair_index(m, n) : pair_index(n, m))) * K + k);
  };
  // D_j . P1
  {
    double p1[kNBasis];
#pragma unroll
    for (int m = 0; m < kNBasis; ++m) p1[m] = P1(m);
#pragma unroll
    for (int j = 0; j < SHARPY_NPHYS; ++j) {
      double t = 0.0;
      if (has_pn(j)) {
#pragma unroll
        for (int b = 0; b < kNPn; ++b) t = __fma_rn(d[j & 3][b], p1[b], t);
        t = __fma_rn(dc[j & 3], P0, t);
      } else if (has_const(j)) {
        t = single(j) * P0;
      } else if (has_f(j)) {
        t = single(j) * p1[kNPn];
      }
      dp1[j] = t;
      img[j] = has_amp(j) ? __fma_rn(Gr, dGi[j], -__dmul_rn(Gi, dGr[j])) : 0.0;  // Im(conj(G) dG_j)
    }
  }
  const double g2 = __fma_rn(Gr, Gr, __dmul_rn(Gi, Gi));
  const double cg2 = __dmul_rn(kTwoPi * kTwoPi, g2);
  // q_jl = D_j P2 D_l by rows j: row_c = sum_b D_jb P2_bc
#pragma unroll
  for (int j = 0; j < SHARPY_NPHYS; ++j) {
    double row[kNB];
    if (has_phase(j)) {
#pragma unroll
      for (int c = 0; c < kNB; ++c) {
        auto p2 = [&](int b) {
          return b == kNBasis ? (c == kNBasis ? P0 : P1(c)) : c == kNBasis ? P1(b) : P2(b, c);
        };
        double t = 0.0;
        if (has_pn(j)) {
#pragma unroll
          for (int b = 0; b < kNPn; ++b) t = __fma_rn(d[j & 3][b], p2(b), t);
          t = __fma_rn(dc[j & 3], p2(kNBasis), t);
        } else {
          t = single(j) * p2(has_const(j) ? kNBasis : kNPn);
        }
        row[c] = t;
      }
    }
#pragma unroll
    for (int l = j; l < SHARPY_NPHYS; ++l) {
      // (Re(conj(dG_j) dG_l) P0 - 2 pi (img_j dp1_l + img_l dp1_j)) + 4 pi^2 |G|^2 q
      const bool t1 = has_amp(j) && has_amp(l);
      const bool t2a = has_amp(j) && has_phase(l), t2b = has_amp(l) && has_phase(j);
      double b2 = 0.0;
      if (t2b) b2 = __dmul_rn(img[l], dp1[j]);
      if (t2a) b2 = __fma_rn(img[j], dp1[l], b2);
      double x = 0.0;
      if (t2a || t2b) x = -__dmul_rn(kTwoPi, b2);
      if (t1) x = __fma_rn(__fma_rn(dGr[j], dGr[l], __dmul_rn(dGi[j], dGi[l])), P0, x);
      if (has_phase(j) && has_phase(l)) {
        double q = 0.0;
        if (has_pn(l)) {
#pragma unroll
          for (int c = 0; c < kNPn; ++c) q = __fma_rn(row[c], d[l & 3][c], q);
          q = __fma_rn(row[kNBasis], dc[l & 3], q);
        } else {
          q = row[has_const(l) ? kNBasis : kNPn] * single(l);
        }
        x = __fma_rn(cg2, q, x);
      }
      v[tri(l, j)] = x;
    }
  }
}

// Cholesky factor of the lower triangle T in place (T = C C^T), all warps:
// column by column, the pivot on warp j mod 4 while the others form their
// rows' sums; *ok gets the particles (lanes) whose pivots were all positive.
__device__ __forceinline__ void cholesky_cta(MetricShared& S, double (*T)[kMetPad], int D, bool keep_rc, int which,
                                             int warp, int lane) {
  for (int j = 0; j < D; ++j) {
    if (warp == (j & (kMetWarps - 1))) {
      double d = T[tri(j, j)][lane];
      for (int k = 0; k < j; ++k) d = __fma_rn(-T[tri(j, k)][lane], T[tri(j, k)][lane], d);
      const bool pos = d > 0.0 && isfinite(d);
      const double c = sqrt(d);
      const double r = 1.0 / c;
      S.piv[lane] = c;
      S.rpiv[lane] = r;
      if (keep_rc) S.rc[j][lane] = r;
      const unsigned m = __ballot_sync(0xffffffffu, pos);
      if (lane == 0) S.ok[which] &= m;
    }
    // rows i = j + 1 + w, + 4, ... (w counted from the pivot's next warp)
    const int w = (warp - j - 1) & (kMetWarps - 1);
    double t[3];
    int n = 0;
#pragma unroll
    for (int u = 0; u < 3; ++u) {
      const int i = j + 1 + w + u * kMetWarps;
      if (i >= D) break;
      double x = T[tri(i, j)][lane];
      for (int k = 0; k < j; ++k) x = __fma_rn(-T[tri(i, k)][lane], T[tri(j, k)][lane], x);
      t[u] = x;
      n = u + 1;
    }
    __syncthreads();
    const double c = S.piv[lane], r = S.rpiv[lane];
#pragma unroll
    for (int u = 0; u < 3; ++u)
      if (u < n) T[tri(j + 1 + w + u * kMetWarps, j)][lane] = quotient(t[u], c, r);
    if (warp == (j & (kMetWarps - 1))) T[tri(j, j)][lane] = c;
    __syncthreads();
  }
}

__global__ void __launch_bounds__(kMetWarps * 32)
    local_metric_kernel(DevModel m, DevEvent ev, int64_t n, const double* __restrict__ theta, const double* beta_ptr,
                        double beta_val, double* mass, double* minv, double* chol, int* status) {
  extern __shared__ __align__(16) unsigned char met_smem[];
  MetricShared& S = *reinterpret_cast<MetricShared*>(met_smem);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t base = (int64_t)blockIdx.x * kMetPart;
  // lanes past the end work on the last particle and store nothing
  const int64_t p = base + lane < n ? base + lane : n - 1;
  const int live = (int)(n - base < kMetPart ? n - base : kMetPart);
  const int D = m.n_dim;
  const double beta = beta_ptr ? *beta_ptr : beta_val;
  double x[kMaxDim];
  for (int i = 0; i < D; ++i) x[i] = theta[p * D + i];
  if (threadIdx.x == 0) S.ok[0] = S.ok[1] = 0xffffffffu;
  if (m.model == SHARPY_MODEL_TAYLORF2) {
    // prologue: the phase on warp 0, the amplitude and the detectors' sky on the others
    if (warp == 0) {
      prologue_phase<double, true>(m, ev, x, S.pro.sc[lane], S.pro.ec[lane]);
    } else {
      if (warp == 1) prologue_amp<double, true>(m, x, S.pro.ec[lane]);
      prologue_sky<double, true>(m, ev, x, min(warp - 1, ev.n_det), min(warp, ev.n_det), S.pro.sc[lane],
                                 S.pro.ec[lane]);
    }
    __syncthreads();
    // Fisher matrices of the detectors on warps 0.., added in detector order
    double v[kTri];
    const bool mine = warp < ev.n_det;
    const bool in = S.pro.sc[lane].ok && S.pro.sc[lane].kisco >= 0;
    if (mine) {
      if (in) {
        fisher_detector(ev, S.pro.sc[lane], S.pro.ec[lane], warp, v);
      } else {
#pragma unroll
        for (int e = 0; e < kTri; ++e) v[e] = 0.0;
      }
    }
    for (int a = 0; a < ev.n_det; ++a) {
      if (warp == a)
#pragma unroll
        for (int e = 0; e < kTri; ++e) S.M[e][lane] = a == 0 ? v[e] : S.M[e][lane] + v[e];
      __syncthreads();
    }
    // M = beta F on the free dimensions
    double f[(kTri + kMetWarps - 1) / kMetWarps];
    const int nt = D * (D + 1) / 2;
    int i = 0, j = 0, u = 0;
    for (int e = 0; e < nt; ++e) {
      if ((e & (kMetWarps - 1)) == warp) {
        const int a = m.phys[i], b = m.phys[j];
        f[u++] = beta * S.M[a >= b ? tri(a, b) : tri(b, a)][lane];
      }
      if (++j > i) {
        ++i;
        j = 0;
      }
    }
    __syncthreads();
    u = 0;
    for (int e = warp; e < nt; e += kMetWarps) S.M[e][lane] = f[u++];
  } else {
    // mixture: responsibility-weighted component precisions (diagonal)
    if (warp == 0) {
      double M[kMaxDim];
      for (int i = 0; i < D; ++i) M[i] = 0.0;
      double lc[SHARPY_MAX_COMP], best = -INFINITY;
      for (int c = 0; c < m.n_comp; ++c) {
        double t = m.mix_logw[c];
        for (int i = 0; i < D; ++i) {
          const double z = (x[i] - m.mix_mu[c][i]) / m.mix_sigma[c][i];
          t += -0.5 * z * z - log(m.mix_sigma[c][i]);
        }
        lc[c] = t;
        best = fmax(best, t);
      }
      double tot = 0.0;
      for (int c = 0; c < m.n_comp; ++c) tot += exp(lc[c] - best);
      for (int c = 0; c < m.n_comp; ++c) {
        const double r = exp(lc[c] - best) / tot;
        for (int i = 0; i < D; ++i) M[i] += beta * r / (m.mix_sigma[c][i] * m.mix_sigma[c][i]);
      }
      for (int i = 0; i < D; ++i)
        for (int j = 0; j <= i; ++j) S.M[tri(i, j)][lane] = i == j ? M[i] : 0.0;
    }
  }
  __syncthreads();
  for (int i = warp; i < D; i += kMetWarps) {
    const double w = m.hi[i] - m.lo[i];
    double t = S.M[tri(i, i)][lane] + 12.0 / (w * w);
    if (m.prior[i] == SHARPY_PRIOR_POWER2) t += 2.0 / (x[i] * x[i]);
    S.M[tri(i, i)][lane] = t;
    S.diag[i][lane] = t;
  }
  __syncthreads();
  // whole matrices to global memory, coalesced
  const int dd = D * D;
  auto copy_out = [&](double* out, const double (*T)[kMetPad], bool lower) {
    double* o = out + base * dd;
    for (int e = threadIdx.x; e < live * dd; e += blockDim.x) {
      const int q = e / dd, r = e - q * dd, i = r / D, j = r - i * D;
      o[e] = i >= j ? T[tri(i, j)][q] : lower ? 0.0 : T[tri(j, i)][q];
    }
  };
  if (mass) copy_out(mass, S.M, false);
  if (!minv && !chol) return;
  __syncthreads();
  // M^-1 = C^-T C^-1 with M = C C^T; then L L^T = M^-1 (lower L)
  cholesky_cta(S, S.M, D, true, 0, warp, lane);
  if (!((S.ok[0] >> lane) & 1u)) {
    // not positive definite in floating point: keep the diagonal (positive by construction)
    for (int i = warp; i < D; i += kMetWarps) {
      for (int j = 0; j < i; ++j) S.M[tri(i, j)][lane] = 0.0;
      const double c = sqrt(S.diag[i][lane]);
      S.M[tri(i, i)][lane] = c;
      S.rc[i][lane] = 1.0 / c;
    }
  }
  __syncthreads();
  // C^-1 (lower), a column per warp: j, then 7 - j, then the short ones
  for (int u = 0; u < 3; ++u) {
    const int j = u == 0 ? warp : u == 1 ? 2 * kMetWarps - 1 - warp : 2 * kMetWarps + warp;
    if (j >= D) continue;
    S.la.Ci[tri(j, j)][lane] = S.rc[j][lane];
    for (int i = j + 1; i < D; ++i) {
      double t = 0.0;
      for (int k = j; k < i; ++k) t = __fma_rn(-S.M[tri(i, k)][lane], S.la.Ci[tri(k, j)][lane], t);
      S.la.Ci[tri(i, j)][lane] = quotient(t, S.M[tri(i, i)][lane], S.rc[i][lane]);
    }
  }
  __syncthreads();
  {
    int i = 0, j = 0;
    for (int e = 0; e < D * (D + 1) / 2; ++e) {
      if ((e & (kMetWarps - 1)) == warp) {
        double t = 0.0;
        for (int k = i; k < D; ++k) t = __fma_rn(S.la.Ci[tri(k, i)][lane], S.la.Ci[tri(k, j)][lane], t);
        S.la.Mi[e][lane] = t;
      }
      if (++j > i) {
        ++i;
        j = 0;
      }
    }
  }
  __syncthreads();
  if (minv) copy_out(minv, S.la.Mi, false);
  if (!chol) return;
  __syncthreads();
  cholesky_cta(S, S.la.Mi, D, false, 1, warp, lane);
  if (!((S.ok[1] >> lane) & 1u))
    for (int i = warp; i < D; i += kMetWarps) {
      for (int j = 0; j < i; ++j) S.la.Mi[tri(i, j)][lane] = 0.0;
      S.la.Mi[tri(i, i)][lane] = S.rc[i][lane];
    }
  __syncthreads();
  copy_out(chol, S.la.Mi, true);
}

// Build the Fisher prefix tables of the staged event (host, compensated sums).
int ensure_fisher_tables(sharpy_ctx* c) {
  if (c->d_p1 && c->d_p2) return SHARPY_OK;
  const int nd = c->ev.n_det;
  const int64_t K = c->ev.n_bins;
  if ((int64_t)c->h_wamp2.size() != nd * K || (int64_t)c->h_basis.size() != kNBasis * K) return SHARPY_ESTATE;
  std::vector<double> p1((size_t)nd * kNBasis * K), p2((size_t)nd * kNPair * K);
  auto prefix = [&](double* out, auto term) {
    double s = 0.0, cmp = 0.0;
    for (int64_t k = 0; k < K; ++k) {
      const double t = term(k);
      const double u = s + t;
      cmp += std::fabs(s) >= std::fabs(t) ? (s - u) + t : (t - u) + s;
      s = u;
      out[k] = s + cmp;
    }
  };
  for (int a = 0; a < nd; ++a) {
    const double* W = c->h_wamp2.data() + (size_t)a * K;
    for (int m = 0; m < kNBasis; ++m) {
      const double* Bm = c->h_basis.data() + (size_t)m * K;
      prefix(p1.data() + ((size_t)a * kNBasis + m) * K, [&](int64_t k) { return W[k] * Bm[k]; });
      for (int n2 = m; n2 < kNBasis; ++n2) {
        const double* Bn = c->h_basis.data() + (size_t)n2 * K;
        const int pi = m * kNBasis - m * (m - 1) / 2 + (n2 - m);
        prefix(p2.data() + ((size_t)a * kNPair + pi) * K, [&](int64_t k) { return W[k] * Bm[k] * Bn[k]; });
      }
    }
  }
  if (cudaMalloc(&c->d_p1, p1.size() * sizeof(double)) != cudaSuccess ||
      cudaMalloc(&c->d_p2, p2.size() * sizeof(double)) != cudaSuccess) {
    cudaFree(c->d_p1);
    cudaFree(c->d_p2);
    c->d_p1 = c->d_p2 = nullptr;
    return SHARPY_ENOMEM;
  }
  if (cudaMemcpy(c->d_p1, p1.data(), p1.size() * sizeof(double), cudaMemcpyHostToDevice) != cudaSuccess ||
      cudaMemcpy(c->d_p2, p2.data(), p2.size() * sizeof(double), cudaMemcpyHostToDevice) != cudaSuccess)
    return SHARPY_ECUDA;
  c->ev.p1 = c->d_p1;
  c->ev.p2 = c->d_p2;
  return SHARPY_OK;
}

int enqueue_local_metric(sharpy_ctx* c, int64_t n, const double* theta, const double* beta_ptr, double beta,
                         double* mass, double* minv, double* chol, cudaStream_t s) {
  if (c->model.model == SHARPY_MODEL_TAYLORF2) {
    const int rc = ensure_fisher_tables(c);
    if (rc) return rc;
  }
  SHARPY_CUDA_TRY(cudaFuncSetAttribute(local_metric_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)sizeof(MetricShared)));
  local_metric_kernel<<<(unsigned)((n + kMetPart - 1) / kMetPart), kMetWarps * 32, sizeof(MetricShared), s>>>(
      c->model, c->ev, n, theta, beta_ptr, beta, mass, minv, chol, c->d_status);
  SHARPY_CUDA_TRY(cudaGetLastError());
  return SHARPY_OK;
}

}  // namespace sharpy

extern "C" int sharpy_local_metric(sharpy_ctx* c, int64_t n, const double* theta, double beta, double* mass,
                                   double* inv_mass, double* chol, sharpy_stream stream) {
  int rc = check_ctx(c, true);
  if (rc) return rc;
  if (n < 1 || n > ((int64_t)1 << 31) || !theta || !(beta >= 0.0 && beta <= 1.0) || (!mass && !inv_mass && !chol))
    return SHARPY_EINVAL;
  cudaStream_t s = (cudaStream_t)stream;
  c->last_stream = s;
  return enqueue_local_metric(c, n, theta, nullptr, beta, mass, inv_mass, chol, s);
}
