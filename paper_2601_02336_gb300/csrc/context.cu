// Context lifetime, event staging, status word and evidence accumulator.
#include <cmath>
#include <cstring>
#include <new>
#include <vector>

#include "context.cuh"
#include "fixed.cuh"

using namespace sharpy;

namespace sharpy {

int ensure_scratch(sharpy_ctx* ctx, size_t bytes) {
  if (bytes <= ctx->scratch_bytes) return SHARPY_OK;
  SHARPY_CUDA_TRY(cudaDeviceSynchronize());
  if (ctx->d_scratch) cudaFree(ctx->d_scratch);
  ctx->d_scratch = nullptr;
  ctx->scratch_bytes = 0;
  size_t want = bytes + bytes / 4;
  if (cudaMalloc(&ctx->d_scratch, want) != cudaSuccess) return SHARPY_ENOMEM;
  ctx->scratch_bytes = want;
  return SHARPY_OK;
}

int check_ctx(sharpy_ctx* ctx, bool need_data) {
  if (!ctx) return SHARPY_EINVAL;
  if (need_data && ctx->model.model == SHARPY_MODEL_TAYLORF2 && !ctx->has_data) return SHARPY_ESTATE;
  if (cudaSetDevice(ctx->device) != cudaSuccess) return SHARPY_ECUDA;
  return SHARPY_OK;
}

// Tables of one event, one CTA per block of kStageBins bins, one thread per bin,
// one warp per tile: the bin's quads of the mixed and of the split sweep's
// tiles and, if fix.tile is not null, of the FP64 path's in fixed point with the
// block's scales and what it brings to the rule on the sweeps' ends.
// Scales: E_a takes 2^e with 2^e |E| <= 2^61; basis function j the largest 2^b
// with 2^b |B| <= 2^61 for which no sum of the block's products can reach 2^62
// (the integer sums' high words; z is in E's units / 4); the basis value 1
// likewise. They come from the largest values' exponents, the products' sums in
// units of 2^-17 of the two powers of two, rounded up, and their squares in 2^-21,
// rounded down, so that a warp sums them with one integer instruction each. Bound
// by latency (32 CTAs for 8033 bins), which the host's own sums hide: a data set
// on the same grid takes 0.21 ms (433 bins: 0.05), without the fixed-point
// tables 0.23 (0.03); with a kernel of 30 warps a block, a moment each in FP64,
// before one for the limbs it took 0.33 (0.11).
struct FixTables {
  int4* tile;
  FixBlock* block;
  double *sq, *need;   // [kFixDet * kNMom][blocks]
  int* from;           // [blocks], then the event's fix_from
  unsigned int* done;  // blocks that have written these; zero between launches
};
__device__ __forceinline__ uint32_t fix_abs_hi(double x) {  // |x|'s high word, zero for zero only
  return ((uint32_t)__double2hiint(x) & 0x7fffffffu) | (__double2loint(x) != 0);
}
__device__ __forceinline__ double fix_pow2(int e) { return __hiloint2double((1023 + e) << 20, 0); }

// fix_from over all blocks, on the CTA that comes last: a warp a moment in turn,
// lanes over the blocks; an exclusive prefix sum of the blocks' squares against
// what each needs before it. Past the last block that fails, or what the blocks
// ask for themselves.
__device__ void fix_from_all(int n_det, int blocks, const FixTables& fix) {
  __shared__ int from_s;
  const int lane = threadIdx.x & 31;
  if (threadIdx.x == 0) from_s = 0;
  __syncthreads();
  int from = 0;
  for (int g = threadIdx.x; g < blocks; g += blockDim.x) from = max(from, __ldcg(fix.from + g));
  for (int n = threadIdx.x >> 5; n < n_det * kNMom; n += blockDim.x >> 5) {
    const double *sqs = fix.sq + (int64_t)n * blocks, *needs = fix.need + (int64_t)n * blocks;
    double before = 0.0;
    for (int g0 = 0; g0 < blocks; g0 += 32) {
      const int g = g0 + lane;
      double incl = g < blocks ? __ldcg(sqs + g) : 0.0;
      const double need = g < blocks ? __ldcg(needs + g) : 0.0;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const double x = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += x;
      }
      const double excl = __shfl_up_sync(0xffffffffu, incl, 1);
      if (!(need <= before + (lane ? excl : 0.0))) from = max(from, (g + 1) * kFixBins);
      before += __shfl_sync(0xffffffffu, incl, 31);
    }
  }
  atomicMax(&from_s, from);
  __syncthreads();
  if (threadIdx.x == 0) fix.from[blocks] = from_s;
}

static_assert(kFixBins == kStageBins, "one block size");
__global__ void __launch_bounds__(kStageBins)
    event_tables_kernel(DevEvent ev, float4* mixed, float4* split, FixTables fix) {
  constexpr int T = kFixBins / kTileBins, NV = kFixDet + kNBasis, NM = kFixDet * kNMom;
  const int64_t K = ev.n_bins, k = (int64_t)blockIdx.x * kStageBins + threadIdx.x;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const bool in = k < K;
  double b[kNBasis];
  double2 e[kFixDet];
#pragma unroll
  for (int j = 0; j < kNBasis; ++j) b[j] = in ? ev.b64[j * K + k] : 0.0;
#pragma unroll
  for (int a = 0; a < kFixDet; ++a) e[a] = in && a < ev.n_det ? ev.e64[a * K + k] : make_double2(0.0, 0.0);
  const int64_t tile = k / kTileBins;
  {
    float hi[kNBasis], lo[kNBasis];
    float2 E[kFixDet];
#pragma unroll
    for (int j = 0; j < kNBasis; ++j) {
      hi[j] = (float)b[j];
      lo[j] = (float)(b[j] - (double)hi[j]);
    }
#pragma unroll
    for (int a = 0; a < kFixDet; ++a) E[a] = make_float2((float)e[a].x, (float)e[a].y);
    auto words = [&](bool sp, const float* t, int i) {
      return make_float4(t[tile_basis(sp, i)], t[tile_basis(sp, i + 1)], t[tile_basis(sp, i + 2)], t[tile_basis(sp, i + 3)]);
    };
    float4* m = mixed + tile * tile_quads(false) * kTileBins + lane;
    m[0 * kTileBins] = words(false, hi, 0);
    m[1 * kTileBins] = words(false, hi, 4);
    m[2 * kTileBins] = words(false, lo, 0);
    m[3 * kTileBins] = make_float4(hi[8], lo[8], E[0].x, E[0].y);
    m[4 * kTileBins] = make_float4(E[1].x, E[1].y, E[2].x, E[2].y);
    for (int i = 0; i < 2; ++i)
      reinterpret_cast<double2*>(m)[(5 + i) * kTileBins] = make_double2(b[large_pn(2 * i)], b[large_pn(2 * i + 1)]);
    float4* s = split + tile * tile_quads(true) * kTileBins + lane;
    s[0 * kTileBins] = words(true, hi, 0);
    s[1 * kTileBins] = words(true, hi, 4);
    s[2 * kTileBins] = words(true, lo, 0);
    s[3 * kTileBins] = words(true, lo, 4);
    s[4 * kTileBins] = make_float4(hi[8], lo[8], E[0].x, E[0].y);
    s[5 * kTileBins] = make_float4(E[1].x, E[1].y, E[2].x, E[2].y);
  }
  if (!fix.tile) return;
  __shared__ uint32_t top[NV], sum_s[T][NM], sq_s[T][NM];
  __shared__ int be_s[kNBasis], last_s;
  // the largest values of E_a (either part) and of B_j, as high words
  if (threadIdx.x < NV) top[threadIdx.x] = 0;
  __syncthreads();
  {
    uint32_t own = 0;
#pragma unroll
    for (int i = 0; i < NV; ++i) {
      const uint32_t h = i < kFixDet ? max(fix_abs_hi(e[i < kFixDet ? i : 0].x), fix_abs_hi(e[i < kFixDet ? i : 0].y))
                                     : fix_abs_hi(b[i < kFixDet ? 0 : i - kFixDet]);
      const uint32_t m = __reduce_max_sync(0xffffffffu, h);
      if (lane == i) own = m;
    }
    if (lane < NV) atomicMax(&top[lane], own);
  }
  __syncthreads();
  // exponents (zeros: 0); a block with values outside 2^-200 .. 2^200 (past
  // which FP64 may not hold the squares), infinities or NaN has no scales
  bool fits = true;
  auto expo = [&](int i) {
    const int x = (int)(top[i] >> 20) - 1023;
    if (top[i] == 0) return 0;
    fits = fits && x >= -200 && x < 200;
    return x;
  };
  int ea[kFixDet], eb[kNMom];
#pragma unroll
  for (int a = 0; a < kFixDet; ++a) ea[a] = expo(a);
#pragma unroll
  for (int j = 0; j < kNBasis; ++j) eb[j] = expo(kFixDet + j);
  eb[kNBasis] = -1;
  if (!fits) {
    if (threadIdx.x == 0) fix.from[blockIdx.x] = kFixNever;
  } else {
    // products p < 4 sqrt(2) of this tile, rounded outwards by the factor
    {
      uint32_t sum = 0, sq = 0;
      float bs[kNMom];
#pragma unroll
      for (int j = 0; j < kNBasis; ++j) bs[j] = (float)(fabs(b[j]) * fix_pow2(-eb[j]));
      bs[kNBasis] = 2.0f;
#pragma unroll
      for (int a = 0; a < kFixDet; ++a) {
        if (a >= ev.n_det) break;
        const float x = (float)(e[a].x * fix_pow2(-ea[a])), y = (float)(e[a].y * fix_pow2(-ea[a]));
        const float l = sqrtf(fmaf(x, x, y * y));
#pragma unroll
        for (int j = 0; j < kNMom; ++j) {
          const float p = l * bs[j];
          const uint32_t u = __reduce_add_sync(0xffffffffu, __float2uint_ru(p * (131072.0f * (1.0f + 0x1p-20f))));
          const uint32_t v = __reduce_add_sync(0xffffffffu, __float2uint_rd(p * p * (2097152.0f * (1.0f - 0x1p-20f))));
          if (lane == a * kNMom + j) sum = u, sq = v;
        }
      }
      if (lane < NM) sum_s[warp][lane] = sum, sq_s[warp][lane] = sq;
    }
    __syncthreads();
    if (warp == 0) {
      // lane = moment (a, j): sum in 2^-17, squares before tile t in 2^-21
      const int n = lane < NM ? lane : NM - 1, a = n / kNMom, j = n % kNMom;
      uint32_t sum = 0;
#pragma unroll
      for (int t = 0; t < T; ++t) sum += sum_s[t][n];
      int shift = max(0, 31 - __clz(sum | 1) - 24);  // sum < 2^(shift + 25)
      shift = max(shift, max(__shfl_sync(0xffffffffu, shift, (lane + kNMom) % NM),
                             __shfl_sync(0xffffffffu, shift, (lane + 2 * kNMom) % NM)));
      int xa = 0, xb = -1;
      uint32_t ha = 0, hb = 1;
#pragma unroll
      for (int i = 0; i < kFixDet; ++i)
        if (a == i) xa = ea[i], ha = top[i];
#pragma unroll
      for (int i = 0; i < kNBasis; ++i)
        if (j == i) xb = eb[i], hb = top[kFixDet + i];
      const bool any = ha != 0 && hb != 0;  // else the products are zero, and exact
      const int ee = ha ? 60 - xa : 0, be = hb ? 60 - xb - shift : 0;
      const int ends = (int)((min(K - (int64_t)blockIdx.x * kFixBins, (int64_t)kFixBins) + kTileBins - 1) / kTileBins);
      int last = 0;  // the last tile in which an end fails with nothing before the block
      FixBlock& fc = fix.block[blockIdx.x];
      if (lane < NM && a < ev.n_det) {
        fc.scale[n] = fix_pow2(66 - ee - be);
        double sq = 0.0, need = 0.0;  // in 2^(2 (xa + xb))
#pragma unroll
        for (int t = 0; t < T; ++t) {
          if (any && t < ends && fix_fails(fix_pow2(shift - 54), t, sq)) {
            need = fmax(need, fix_need(fix_pow2(shift - 54), t) - sq);
            last = t;
          }
          sq += (double)sq_s[t][n] * 0x1p-21;
        }
        const double u = fix_pow2(2 * (xa + xb));
        const int64_t at = (int64_t)n * gridDim.x + blockIdx.x;
        fix.sq[at] = sq * u;
        fix.need[at] = blockIdx.x == 0 ? 0.0 : need * u;
        if (a == 0 && j < kNBasis) be_s[j] = be;
        if (n == kNBasis) fc.one = 1 << (be - 32);
      }
      __syncwarp();
      last = __reduce_max_sync(0xffffffffu, last);
      if (lane == 0) fix.from[blockIdx.x] = blockIdx.x == 0 ? kTileBins * (last + 1) : 0;
    }
    __syncthreads();
    int4* t = fix.tile + tile * (kFixQuads * kTileBins) + lane;
#pragma unroll
    for (int j = 0; j < kNBasis; ++j) {
      const Limbs l = fix_limbs_neg(__double2ll_rn(b[j] * fix_pow2(be_s[j])));
      t[j * kTileBins] = make_int4(__double2loint(b[j]), __double2hiint(b[j]), l.h, l.l);
    }
#pragma unroll
    for (int a = 0; a < kFixDet; ++a) {
      const double u = top[a] ? fix_pow2(60 - ea[a]) : 1.0;
      const Limbs x = fix_limbs_neg(__double2ll_rn(e[a].x * u)), y = fix_limbs_neg(__double2ll_rn(e[a].y * u));
      t[(kNBasis + a) * kTileBins] = make_int4(x.h, x.l, y.h, y.l);
    }
  }
  // (the last block's reads of the others' writes go past L1)
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) last_s = atomicInc(fix.done, gridDim.x - 1) == gridDim.x - 1;
  __syncthreads();
  if (!last_s) return;
  __threadfence();
  fix_from_all(ev.n_det, (int)gridDim.x, fix);
}

}  // namespace sharpy

// The carrier's table, cos and sin of 2 pi i / 1024 to 2^-62 (from the first
// octant, where long double has the bits for it on every host).
static const int4* fix_trig_host() {
  static const std::vector<int4> t = [] {
    std::vector<int4> v(kFixTrig + 1, int4{0, 0, 0, 0});  // the count after it (FixTables::done) starts at zero
    constexpr int O = kFixTrig / 8;
    int64_t co[O + 1], si[O + 1];
    for (int i = 0; i <= O; ++i) {
      const long double x = 6.283185307179586476925286766559L / kFixTrig * i;
      co[i] = (int64_t)std::rint(std::ldexp(std::cos(x), 62));
      si[i] = (int64_t)std::rint(std::ldexp(std::sin(x), 62));
    }
    for (int i = 0; i < kFixTrig; ++i) {
      const int q = i / (2 * O), r = i % (2 * O);  // quadrant, place in it
      const int64_t a = r > O ? si[2 * O - r] : co[r], b = r > O ? co[2 * O - r] : si[r];
      const Limbs c = fix_limbs_neg(q == 0 ? a : q == 1 ? -b : q == 2 ? -a : b);
      const Limbs s = fix_limbs_neg(q == 0 ? b : q == 1 ? a : q == 2 ? -b : -a);
      v[i] = make_int4(c.h, c.l, s.h, s.l);
    }
    return v;
  }();
  return t.data();
}

// The sweeps' tables, built with every data set (they hold E). Without the
// fixed-point ones (memory, too many bins, data that no scale fits) the FP64
// sweep runs.
static cudaError_t build_tables(sharpy_ctx* c, int64_t blocks) {
  DevEvent& ev = c->ev;
  ev.tile_fix = nullptr;
  ev.fix_from = nullptr;
  ev.fix_block = nullptr;
  ev.fix_trig = nullptr;
  float4* split = c->d_tile + blocks * (stage_bytes(false) / 16);
  const size_t tiles = (size_t)blocks * kStageBins * kFixQuads, rule = (size_t)blocks * kFixDet * kNMom;
  if (!c->d_fix && ev.n_bins <= kFixMaxBins && ev.n_det <= kFixDet) {
    if (cudaMalloc(&c->d_fix, (tiles + kFixTrig + 1) * sizeof(int4) + (size_t)blocks * (sizeof(FixBlock) + sizeof(int)) +
                                  2 * rule * sizeof(double) + sizeof(int)) != cudaSuccess) {
      c->d_fix = nullptr;
      (void)cudaGetLastError();
    } else {
      const cudaError_t e = cudaMemcpy(c->d_fix + tiles, fix_trig_host(), (kFixTrig + 1) * sizeof(int4), cudaMemcpyHostToDevice);
      if (e != cudaSuccess) return e;
    }
  }
  FixTables fix{};
  if (c->d_fix) {
    fix.tile = c->d_fix;
    fix.done = reinterpret_cast<unsigned int*>(c->d_fix + tiles + kFixTrig);
    fix.block = reinterpret_cast<FixBlock*>(c->d_fix + tiles + kFixTrig + 1);
    fix.sq = reinterpret_cast<double*>(fix.block + blocks);
    fix.need = fix.sq + rule;
    fix.from = reinterpret_cast<int*>(fix.need + rule);
  }
  event_tables_kernel<<<(unsigned)blocks, kStageBins>>>(ev, c->d_tile, split, fix);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  ev.tile_mixed = c->d_tile;
  ev.tile_split = split;
  if (c->d_fix) {
    ev.tile_fix = fix.tile;
    ev.fix_from = fix.from + blocks;
    ev.fix_block = fix.block;
    ev.fix_trig = c->d_fix + tiles;
  }
  return cudaSuccess;
}

static void free_event(sharpy_ctx* c) {
  cudaFree(c->d_f);
  cudaFree(c->d_b64);
  cudaFree(c->d_e64);
  cudaFree(c->d_pref);
  cudaFree(c->d_p1);
  cudaFree(c->d_p2);
  cudaFree(c->d_tile);
  cudaFree(c->d_fix);
  c->d_tile = nullptr;
  c->d_fix = nullptr;
  c->d_p1 = c->d_p2 = nullptr;
  c->ev.p1 = c->ev.p2 = nullptr;
  c->d_f = c->d_b64 = c->d_pref = nullptr;
  c->d_e64 = nullptr;
  c->has_data = false;
}

// Detector tensor and position of an L-shaped detector on a spherical Earth.
static void detector_geometry(const sharpy_detector& in, DevDetector& out) {
  out.fixed_response = in.fixed_response;
  out.fplus = in.fplus;
  out.fcross = in.fcross;
  out.delay = in.delay;
  double sl = std::sin(in.lat), cl = std::cos(in.lat), so = std::sin(in.lon), co = std::cos(in.lon);
  double east[3] = {-so, co, 0.0};
  double north[3] = {-sl * co, -sl * so, cl};
  double ca = std::cos(in.azimuth), sa = std::sin(in.azimuth);
  double x[3], y[3];
  for (int i = 0; i < 3; ++i) {
    x[i] = ca * north[i] + sa * east[i];
    y[i] = -sa * north[i] + ca * east[i];
  }
  for (int i = 0; i < 3; ++i)
    for (int j = 0; j < 3; ++j) {
      out.D[i][j] = 0.5 * (x[i] * x[j] - y[i] * y[j]);
      out.Df[i][j] = (float)out.D[i][j];
    }
  out.r[0] = kEarthR * cl * co;
  out.r[1] = kEarthR * cl * so;
  out.r[2] = kEarthR * sl;
  for (int i = 0; i < 3; ++i) {
    out.rcd[i] = out.r[i] / kClight;
    out.rcf[i] = (float)out.rcd[i];
  }
}

extern "C" {

int sharpy_create(sharpy_ctx** out, const sharpy_config* cfg, int device) {
  if (!out || !cfg) return SHARPY_EINVAL;
  *out = nullptr;
  if (cfg->n_dim < 1 || cfg->n_dim > SHARPY_MAX_DIM) return SHARPY_EINVAL;
  if (cfg->model != SHARPY_MODEL_TAYLORF2 && cfg->model != SHARPY_MODEL_GAUSSMIX) return SHARPY_EINVAL;
  for (int i = 0; i < cfg->n_dim; ++i) {
    if (!(cfg->lo[i] < cfg->hi[i]) || !std::isfinite(cfg->lo[i]) || !std::isfinite(cfg->hi[i])) return SHARPY_EINVAL;
    if (cfg->model == SHARPY_MODEL_TAYLORF2 && (cfg->phys[i] < 0 || cfg->phys[i] >= SHARPY_NPHYS)) return SHARPY_EINVAL;
    if (cfg->prior[i] == SHARPY_PRIOR_POWER2 && !(cfg->lo[i] > 0.0)) return SHARPY_EINVAL;
    if (cfg->prior[i] != SHARPY_PRIOR_UNIFORM && cfg->prior[i] != SHARPY_PRIOR_POWER2) return SHARPY_EINVAL;
    if (cfg->boundary[i] != SHARPY_BOUND_REFLECT && cfg->boundary[i] != SHARPY_BOUND_PERIODIC) return SHARPY_EINVAL;
  }
  if (cfg->model == SHARPY_MODEL_GAUSSMIX) {
    if (cfg->n_comp < 1 || cfg->n_comp > SHARPY_MAX_COMP) return SHARPY_EINVAL;
    for (int c = 0; c < cfg->n_comp; ++c)
      for (int i = 0; i < cfg->n_dim; ++i)
        if (!(cfg->mix_sigma[c][i] > 0.0)) return SHARPY_EINVAL;
  }
  int ndev = 0;
  if (cudaGetDeviceCount(&ndev) != cudaSuccess || device < 0 || device >= ndev) return SHARPY_ECUDA;
  if (cudaSetDevice(device) != cudaSuccess) return SHARPY_ECUDA;
  sharpy_ctx* c = new (std::nothrow) sharpy_ctx();
  if (!c) return SHARPY_ENOMEM;
  c->device = device;
  DevModel& m = c->model;
  m.model = cfg->model;
  m.n_dim = cfg->n_dim;
  for (int i = 0; i < SHARPY_MAX_DIM; ++i) {
    m.phys[i] = cfg->phys[i];
    m.lo[i] = cfg->lo[i];
    m.hi[i] = cfg->hi[i];
    m.prior[i] = cfg->prior[i];
    m.boundary[i] = cfg->boundary[i];
  }
  for (int i = 0; i < SHARPY_NPHYS; ++i) m.fixed[i] = cfg->fixed[i];
  m.n_comp = cfg->n_comp;
  for (int k = 0; k < SHARPY_MAX_COMP; ++k) {
    m.mix_logw[k] = cfg->mix_logw[k];
    for (int i = 0; i < SHARPY_MAX_DIM; ++i) {
      m.mix_mu[k][i] = cfg->mix_mu[k][i];
      m.mix_sigma[k][i] = cfg->mix_sigma[k][i];
    }
  }
  bool ok = cudaMalloc(&c->d_status, sizeof(int)) == cudaSuccess &&
            cudaMalloc(&c->d_lnz, 2 * sizeof(double)) == cudaSuccess &&
            cudaMallocHost(&c->h_pinned, 64 * sizeof(double)) == cudaSuccess &&
            cudaMemset(c->d_status, 0, sizeof(int)) == cudaSuccess &&
            cudaMemset(c->d_lnz, 0, 2 * sizeof(double)) == cudaSuccess &&
            cudaDeviceSynchronize() == cudaSuccess;
  if (!ok) {
    sharpy_destroy(c);
    return SHARPY_ENOMEM;
  }
  *out = c;
  return SHARPY_OK;
}

void sharpy_destroy(sharpy_ctx* c) {
  if (!c) return;
  cudaSetDevice(c->device);
  cudaDeviceSynchronize();
  free_event(c);
  cudaFree(c->d_status);
  cudaFree(c->d_lnz);
  cudaFree(c->d_scratch);
  cudaFreeHost(c->h_pinned);
  delete c;
}

int sharpy_set_data(sharpy_ctx* c, int n_det, int64_t n_bins, double f_min, double df, const double* d,
                    const double* psd, const sharpy_detector* det) {
  if (!c || !d || !psd || !det) return SHARPY_EINVAL;
  if (c->model.model != SHARPY_MODEL_TAYLORF2) return SHARPY_EINVAL;
  if (n_det < 1 || n_det > SHARPY_MAX_DET || n_bins < 1 || n_bins > (int64_t)1 << 30) return SHARPY_EINVAL;
  if (!(f_min > 0.0) || !(df > 0.0) || !std::isfinite(f_min) || !std::isfinite(df)) return SHARPY_EINVAL;
  if (n_det != 1 && n_det != 2 && n_det != 3) return SHARPY_EINVAL;  // kernels are instantiated for 1-3
  int64_t K = n_bins;
  for (int64_t i = 0; i < (int64_t)n_det * K; ++i) {
    if (!std::isfinite(psd[i]) || !(psd[i] > 0.0)) return SHARPY_ENONFINITE;
    if (!std::isfinite(d[2 * i]) || !std::isfinite(d[2 * i + 1])) return SHARPY_ENONFINITE;
  }
  int rc = check_ctx(c, false);
  if (rc) return rc;

  // The frequency-grid tables (f, basis functions, f^-7/6) depend only on
  // (K, f_min, df): a new event on the same grid and detector count keeps
  // them and the device buffers, and only the data-dependent tables are
  // rebuilt and copied.
  const int64_t blocks = (K + kStageBins - 1) / kStageBins;
  const bool same_grid = c->has_data && c->ev.n_det == n_det && c->ev.n_bins == K && c->ev.f_min == f_min &&
                         c->ev.df == df && (int64_t)c->h_amp.size() == K;
  if (!same_grid) {
    std::vector<double> f(K), b64(kNBasis * K), amp(K);
    for (int64_t k = 0; k < K; ++k) {
      double fk = f_min + (double)k * df;
      f[k] = fk;
      double x = std::cbrt(1.0 / fk), y = std::cbrt(fk), l = std::log(fk);
      double x2 = x * x;
      double B[kNBasis] = {x2 * x2 * x, x2 * x, x2, x, l, y, y * l, y * y, fk};
      for (int j = 0; j < kNBasis; ++j) b64[j * K + k] = B[j];
      amp[k] = std::pow(fk, -7.0 / 6.0);
    }
    free_event(c);
    bool ok = cudaMalloc(&c->d_f, K * sizeof(double)) == cudaSuccess &&
              cudaMalloc(&c->d_b64, kNBasis * K * sizeof(double)) == cudaSuccess &&
              cudaMalloc(&c->d_e64, n_det * K * sizeof(double2)) == cudaSuccess &&
              cudaMalloc(&c->d_tile, (size_t)blocks * (stage_bytes(false) + stage_bytes(true))) == cudaSuccess &&
              cudaMalloc(&c->d_pref, n_det * K * sizeof(double)) == cudaSuccess;
    if (!ok) {
      free_event(c);
      return SHARPY_ENOMEM;
    }
    ok = cudaMemcpy(c->d_f, f.data(), K * sizeof(double), cudaMemcpyHostToDevice) == cudaSuccess &&
         cudaMemcpy(c->d_b64, b64.data(), b64.size() * sizeof(double), cudaMemcpyHostToDevice) == cudaSuccess;
    if (!ok) {
      free_event(c);
      return SHARPY_ECUDA;
    }
    c->h_basis.swap(b64);
    c->h_amp.swap(amp);
    c->h_wamp2.clear();
  } else if (cudaDeviceSynchronize() != cudaSuccess) {
    // the previous event's tables may still be read by queued work
    return SHARPY_ECUDA;
  }
  const std::vector<double>& amp = c->h_amp;
  std::vector<double> e64(2 * n_det * K), pref(n_det * K), wamp2(n_det * K);
  // E = w conj(d) f^-7/6, from which the device makes the sweeps' tables while
  // the host goes on
  for (int a = 0; a < n_det; ++a)
    for (int64_t k = 0; k < K; ++k) {
      const int64_t i = a * K + k;
      const double w = 4.0 * df / psd[i];
      wamp2[i] = w;
      e64[2 * i] = w * d[2 * i] * amp[k];
      e64[2 * i + 1] = -w * d[2 * i + 1] * amp[k];
    }
  DevEvent& ev = c->ev;
  ev.n_det = n_det;
  ev.n_bins = K;
  ev.f_min = f_min;
  ev.df = df;
  ev.inv_df = 1.0 / df;
  ev.f = c->d_f;
  ev.b64 = c->d_b64;
  ev.e64 = c->d_e64;
  ev.pref = c->d_pref;
  if (cudaMemcpy(c->d_e64, e64.data(), e64.size() * sizeof(double), cudaMemcpyHostToDevice) != cudaSuccess ||
      build_tables(c, blocks) != cudaSuccess) {
    free_event(c);
    return SHARPY_ECUDA;
  }
  // <d|d> with a compensated sum; P_a prefix sums of w f^-7/3 (compensated).
  double dd = 0.0, ddc = 0.0;
  for (int a = 0; a < n_det; ++a) {
    double s = 0.0, cmp = 0.0;
    for (int64_t k = 0; k < K; ++k) {
      int64_t i = a * K + k;
      double w = wamp2[i];
      double dr = d[2 * i], di = d[2 * i + 1];
      double term = w * amp[k] * amp[k];
      wamp2[i] = term;
      double t = s + term;
      cmp += std::fabs(s) >= std::fabs(term) ? (s - t) + term : (term - t) + s;
      s = t;
      pref[i] = s + cmp;
      double dt = w * (dr * dr + di * di);
      double u = dd + dt;
      ddc += std::fabs(dd) >= std::fabs(dt) ? (dd - u) + dt : (dt - u) + dd;
      dd = u;
    }
  }
  // the Fisher prefix tables depend on w f^-7/3 only: kept while it is unchanged
  if (wamp2 != c->h_wamp2) {
    cudaFree(c->d_p1);
    cudaFree(c->d_p2);
    c->d_p1 = c->d_p2 = nullptr;
    c->h_wamp2.swap(wamp2);
  }
  ev.dd = dd + ddc;
  {
    const double h = -0.5 * ev.dd;  // the epilogue's starting sum, as a double-float
    ev.ddh_hi = (float)h;
    ev.ddh_lo = (float)(h - (double)ev.ddh_hi);
  }
  ev.p1 = c->d_p1;
  ev.p2 = c->d_p2;
  for (int a = 0; a < n_det; ++a) detector_geometry(det[a], ev.det[a]);
  if (cudaMemcpy(c->d_pref, pref.data(), pref.size() * sizeof(double), cudaMemcpyHostToDevice) != cudaSuccess ||
      cudaDeviceSynchronize() != cudaSuccess) {
    free_event(c);
    return SHARPY_ECUDA;
  }
  c->has_data = true;
  return SHARPY_OK;
}

int sharpy_fixed_point_from(sharpy_ctx* c, int64_t* bin) {
  int rc = check_ctx(c, true);
  if (rc) return rc;
  if (!bin) return SHARPY_EINVAL;
  if (c->model.model != SHARPY_MODEL_TAYLORF2) return SHARPY_EINVAL;
  int from = kFixNever;
  if (c->ev.tile_fix) SHARPY_CUDA_TRY(cudaMemcpy(&from, c->ev.fix_from, sizeof(int), cudaMemcpyDeviceToHost));
  *bin = from < c->ev.n_bins ? from : c->ev.n_bins;
  return SHARPY_OK;
}

int sharpy_reset_evidence(sharpy_ctx* c, sharpy_stream stream) {
  int rc = check_ctx(c, false);
  if (rc) return rc;
  SHARPY_CUDA_TRY(cudaMemsetAsync(c->d_lnz, 0, 2 * sizeof(double), (cudaStream_t)stream));
  c->last_stream = (cudaStream_t)stream;
  return SHARPY_OK;
}

int sharpy_set_evidence(sharpy_ctx* c, double lnz, int n_stages, sharpy_stream stream) {
  int rc = check_ctx(c, false);
  if (rc) return rc;
  if (!std::isfinite(lnz) || n_stages < 0) return SHARPY_EINVAL;
  cudaStream_t s = (cudaStream_t)stream;
  // through the pinned staging buffer, after the stream's earlier work has read it
  SHARPY_CUDA_TRY(cudaStreamSynchronize(s));
  c->h_pinned[0] = lnz;
  c->h_pinned[1] = (double)n_stages;
  SHARPY_CUDA_TRY(cudaMemcpyAsync(c->d_lnz, c->h_pinned, 2 * sizeof(double), cudaMemcpyHostToDevice, s));
  SHARPY_CUDA_TRY(cudaStreamSynchronize(s));
  c->last_stream = s;
  return SHARPY_OK;
}

int sharpy_log_evidence(sharpy_ctx* c, double* lnz, int* n_stages) {
  int rc = check_ctx(c, false);
  if (rc) return rc;
  if (!lnz) return SHARPY_EINVAL;
  SHARPY_CUDA_TRY(cudaMemcpyAsync(c->h_pinned, c->d_lnz, 2 * sizeof(double), cudaMemcpyDeviceToHost,
                                  c->last_stream));
  SHARPY_CUDA_TRY(cudaStreamSynchronize(c->last_stream));
  *lnz = c->h_pinned[0];
  if (n_stages) *n_stages = (int)c->h_pinned[1];
  return SHARPY_OK;
}

int sharpy_get_status(sharpy_ctx* c) {
  int rc = check_ctx(c, false);
  if (rc) return rc;
  int s = 0;
  SHARPY_CUDA_TRY(cudaDeviceSynchronize());
  SHARPY_CUDA_TRY(cudaMemcpy(&s, c->d_status, sizeof(int), cudaMemcpyDeviceToHost));
  return s;
}

int sharpy_clear_status(sharpy_ctx* c) {
  int rc = check_ctx(c, false);
  if (rc) return rc;
  SHARPY_CUDA_TRY(cudaDeviceSynchronize());
  SHARPY_CUDA_TRY(cudaMemset(c->d_status, 0, sizeof(int)));
  SHARPY_CUDA_TRY(cudaDeviceSynchronize());
  return SHARPY_OK;
}

const char* sharpy_error_string(int code) {
  switch (code) {
    case SHARPY_OK: return "ok";
    case SHARPY_EINVAL: return "invalid argument";
    case SHARPY_ECUDA: return "CUDA runtime error";
    case SHARPY_ENOMEM: return "out of memory";
    case SHARPY_ENONFINITE: return "non-finite value";
    case SHARPY_ETIMEOUT: return "device loop bound reached";
    case SHARPY_EBOUNDS: return "index out of bounds";
    case SHARPY_ESTATE: return "call out of order";
    default: return "unknown error";
  }
}

}  // extern "C"

extern "C" void sharpy_uniform2(uint64_t key, uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3, double* u) {
  if (u) sharpy::uniform2(key, c0, c1, c2, c3, u, u + 1);
}
