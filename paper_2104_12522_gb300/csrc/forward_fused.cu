// Host side of the persistent fused emission launch (the kernels are in
// emission_fused.cuh, instantiated per species count in fused_s1.cu ..
// fused_s4.cu so the translation units compile in parallel): constant tables,
// scratch (work counters, published layer states, band partials), the tile
// autotuner and the launch.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <vector>

#include "emission_fused.cuh"

using namespace bartem;

namespace {

FusedLauncher pick_fused(int S, int na, FusedForm form, int nt, int mode) {
  switch (S) {
    case 1: return fused_launcher<1>(na, form, nt, mode);
    case 2: return fused_launcher<2>(na, form, nt, mode);
    case 3: return fused_launcher<3>(na, form, nt, mode);
    case 4: return fused_launcher<4>(na, form, nt, mode);
    default: return nullptr;
  }
}

// The form of a call of n proposals: the bulk-copy variant on request, where
// its 16-byte row starts hold (n_nu a multiple of 4 and an aligned grid), else two
// pairs per thread where the rows allow it and the call has enough wavenumbers
// to fill the SMs twice with such threads (354 proposals on 1,600, a fill and a
// half: 80 us in pairs, 84 with two), from 24 proposals on or where columns may
// end early.  Without early ends, on the 100-layer grid of 4 species: 16
// proposals 410 us in pairs and 417 with two (few share a row: DRAM), 32 716 and
// 688, 512 9.30 and 8.65 ms; with them 512 7.60 ms, 16 of a checked grid 328 us.
FusedForm fused_form(const bart_ctx* ctx, const bart_grid_desc* g, int n, bool ends) {
  const int64_t N = g->nu.n_nu;
  const bool rows16 = (N % 4 == 0) && (reinterpret_cast<uintptr_t>(g->grid) % 16 == 0);
  return !rows16 ? FUSED_PAIR
         : ctx->em_launch == BART_LAUNCH_FUSED_TMA ? FUSED_BULK
         : (n >= 24 || ends) && (double)n * (double)N >= 8.0 * FUSED_OCC_THREADS2 * ctx->sm_count ? FUSED_TWO_PAIRS
                                                                                                  : FUSED_PAIR;
}

// Sets *bad where a value of the grid is negative (or -0), infinite or not a
// number: its bits are above those of the largest float.  Bound by the reads of
// the grid from DRAM.
constexpr int CHECK_THREADS = 512;
__global__ void __launch_bounds__(CHECK_THREADS)
grid_check_kernel(const float* __restrict__ grid, size_t n, int* __restrict__ bad) {
  const size_t step = (size_t)gridDim.x * CHECK_THREADS, first = (size_t)blockIdx.x * CHECK_THREADS + threadIdx.x;
  unsigned int m = 0;
  if ((reinterpret_cast<uintptr_t>(grid) & 15) == 0) {
    const uint4* g4 = reinterpret_cast<const uint4*>(grid);
#pragma unroll 8
    for (size_t i = first; i < n / 4; i += step) {
      const uint4 v = __ldg(g4 + i);
      m = max(max(max(m, v.x), max(v.y, v.z)), v.w);
    }
    for (size_t i = n / 4 * 4 + first; i < n; i += step) m = max(m, __float_as_uint(__ldg(grid + i)));
  } else {
    for (size_t i = first; i < n; i += step) m = max(m, __float_as_uint(__ldg(grid + i)));
  }
  if (m > 0x7f7fffffu) *bad = 1;
}

// Proposals per grid temperature from which a call checks the grid so that
// columns may end early.  The check reads S L M n_nu values from DRAM (3.2 GB:
// 0.48 ms); the layers that n proposals leave out save 0.40 ms of 128 proposals
// on a grid of 20 temperatures, 0.78 ms of 256, 1.5 ms of 512.  Of the smallest
// grids its two launches are the cost, 6 us (200 x 60 x 4,096, 2 species: 102 us
// without, 110 with; 100 x 100 x 8,000, 4 species: 172 and 165): n S L n_nu of at
// least CHECK_VALUES.
constexpr int CHECK_FROM = 10;
constexpr double CHECK_VALUES = 1e8;

}  // namespace

bool bartem::columns_may_end(const bart_ctx* ctx, const bart_grid_desc* g, const bart_fwd_cfg* c, const bart_batch* b) {
  bool ends = ctx->em_launch != BART_LAUNCH_SPLIT && fused_offsets_fit(g) &&
              fused_form(ctx, g, b->n, true) == FUSED_TWO_PAIRS && !b->nu_lo;
  for (int s = 0; s < g->n_species; ++s) ends = ends && c->x0[s] >= 0.0;
  return ends;
}

bart_status bartem::check_grid_values(bart_ctx* ctx, const bart_grid_desc* g, const int** bad) {
  void* p = nullptr;
  bart_status st;
  if ((st = bart_scratch(ctx, "ff_bad", sizeof(int), &p)) != BART_OK) return st;
  BART_CUDA(ctx, cudaMemsetAsync(p, 0, sizeof(int), ctx->stream));
  const size_t n = (size_t)g->n_species * g->n_layers * g->n_temps * (size_t)g->nu.n_nu;
  const size_t want = n / (32 * CHECK_THREADS) + 1;      // 8 16-byte loads a thread
  grid_check_kernel<<<(unsigned)std::min<size_t>(want, 4 * (size_t)ctx->sm_count), CHECK_THREADS, 0, ctx->stream>>>(
      g->grid, n, (int*)p);
  *bad = (const int*)p;
  return bart_check_launch(ctx, "grid_check_kernel");
}

bart_status bartem::fused_emission(bart_ctx* ctx, const bart_grid_desc* g, const bart_fwd_cfg* c,
                                   const bart_batch* b, float* spectra, const bart_filters* f, float* bands, int nb) {
  const int S = g->n_species, L = g->n_layers, M = g->n_temps, n = b->n, NA = c->n_angles;
  const int64_t N = g->nu.n_nu;
  const int mode = emission_mode(g, c);
  // columns may end early where the grid was checked (by the retrieval loop) or
  // the check pays for the call (of which every proposal is active)
  const bool pays = n >= (int64_t)CHECK_FROM * M && (double)n * S * L * (double)N >= CHECK_VALUES && !b->active;
  const bool ends = (ctx->grid_bad || pays) && columns_may_end(ctx, g, c, b);
  const FusedForm form = fused_form(ctx, g, n, ends);
  if (S > FUSED_MAX_SPECIES || !pick_fused(S, NA, form, FUSED_THREADS[1], mode))
    return bart_fail(ctx, BART_EUNSUPPORTED, "emission with %d species and %d angles is not instantiated "
                     "(species 1-4; angles 1, 2, 4, 8, 16)", S, NA);
  bart_status st;
  // device table: level pressures, temperature axis, (P_{k+1} - P_k) / 2g
  std::vector<float> hconst;
  for (int k = 0; k < L; ++k) hconst.push_back((float)(g->p_bar[k] * bartc::BAR));
  for (int m = 0; m < M; ++m) hconst.push_back((float)g->t_K[m]);
  for (int k = 0; k + 1 < L; ++k)
    hconst.push_back((float)((g->p_bar[k + 1] - g->p_bar[k]) * bartc::BAR / (2.0 * c->g_cgs)));
  void *p_const, *p_work, *p_done = nullptr, *p_part = nullptr;
  if ((st = bart_upload_const(ctx, "ff_const", hconst.data(), hconst.size() * sizeof(float), &p_const)) != BART_OK)
    return st;
  void *p_twc, *p_flag, *p_bad;
  if ((st = bart_scratch(ctx, "ff_work", 3 * sizeof(unsigned long long), &p_work)) != BART_OK) return st;
  if ((st = bart_scratch(ctx, "ff_twc", (size_t)n * L * sizeof(LayerTW), &p_twc)) != BART_OK) return st;
  if ((st = bart_scratch(ctx, "ff_flag", (size_t)n * sizeof(unsigned int), &p_flag)) != BART_OK) return st;
  // (of every call, so that a capture may follow an eager call that did not check)
  if ((st = bart_scratch(ctx, "ff_bad", sizeof(int), &p_bad)) != BART_OK) return st;
  const int max_tiles = (int)((N + 3 + 2 * FUSED_THREADS[0] - 1) / (2 * FUSED_THREADS[0]));   // smallest tile, aligned start
  if (nb > 0) {
    if ((st = bart_scratch(ctx, "ff_done", (size_t)n * sizeof(unsigned int), &p_done)) != BART_OK) return st;
    if ((st = bart_scratch(ctx, "fw_part", (size_t)n * max_tiles * nb * sizeof(float2), &p_part)) != BART_OK)
      return st;
  }
  FusedArgs a{};
  a.grid = g->grid;
  a.L = L;
  a.M = M;
  a.N = N;
  a.theta = b->theta;
  a.n_theta = 5 + S;
  a.t_profile = b->t_profile;
  a.n = n;
  a.nu_lo = b->nu_lo;
  a.nu_hi = b->nu_hi;
  a.offs = b->spec_offsets;
  a.active = b->active;
  const float* dc = (const float*)p_const;
  a.p_cgs = dc;
  a.t_axis = dc + L;
  a.dpg = dc + L + M;
  for (int s = 0; s < S; ++s) a.x0mu[s] = (float)(c->x0[s] / (c->mu_amu * bartc::AMU));
  std::vector<double> mu, w;
  gauss_legendre01(NA, mu, w);
  float tw_top = 0.0f;
  for (int i = 0; i < NA; ++i) {
    a.ang[i] = (float)(-1.4426950408889634 / mu[i]);
    a.ang[NA + i] = (float)(2.0 * bartc::PI * w[i] * mu[i] * 0.5);   // the 1/2 of the layer-mean source
    tw_top += a.ang[NA + i];
  }
  a.tw_top = tw_top;
  a.inv_g = (float)(1.0 / c->g_cgs);
  a.tint4 = (float)std::pow(c->t_int_K, 4.0);
  const double rs = c->r_star_tp_cm, ao = c->a_orbit_cm;
  a.tirr0 = (rs > 0 && ao > 0) ? (float)(std::sqrt(rs / (2.0 * ao)) * c->t_star_K) : 0.0f;
  a.t_min = (float)c->t_min_K;
  a.t_max = (float)std::min(c->t_max_K, 1e30);
  a.nu_start = g->nu.nu_start_cm;
  a.dnu = g->nu.dnu_cm;
  a.spectra = spectra;
  a.filt = nb ? f->weights : nullptr;
  a.n_bands = nb;
  a.partial = (float2*)p_part;
  a.bands = bands;
  a.work = (unsigned long long*)p_work;
  a.p_done = (unsigned int*)p_done;
  a.tw_cache = (LayerTW*)p_twc;
  a.tw_flag = (unsigned int*)p_flag;
  a.status = ctx->d_status;
  a.ex = emission_extra(g, c);
  if (ends && ctx->grid_bad) a.grid_bad = ctx->grid_bad;
  else if (ends && (st = check_grid_values(ctx, g, &a.grid_bad)) != BART_OK) return st;
  a.wide_x = (mode & 1) != 0;
  a.tau_lim = (mode & 2) != 0;

  // The CTAs in flight work on the same wavenumber span for neighbouring
  // proposals, which between them read the rows of every layer and
  // temperature bracket of that span: a unit spans at most as many
  // wavenumbers as keep those rows (S L M x span x 4 B) within half of L2.
  int l2_bytes = 0;
  if (cudaDeviceGetAttribute(&l2_bytes, cudaDevAttrL2CacheSize, ctx->device) != cudaSuccess) {
    cudaGetLastError();
    l2_bytes = 0;
  }
  const long long span_cap =
      (l2_bytes > 0 ? (long long)l2_bytes / 2 : (64LL << 20)) / ((long long)S * L * M * (long long)sizeof(float));
  auto run = [&](int nt, bool load_only = false) -> bart_status {
    const int tw = fused_width(form, nt);
    // several consecutive tiles per unit amortise the unit's fixed work (layer
    // states, band partials and counts), as long as there are enough units to
    // balance the CTAs (about 8 per CTA of a full grid)
    const int n_tiles = (int)((N + 3 + tw - 1) / tw);                // tiles start on an aligned index
    const long long target = 8LL * ctx->sm_count * (fused_occ_threads(form == FUSED_TWO_PAIRS ? 2 : 1) / nt);
    const long long tpu_cap = std::max(1LL, std::min<long long>(MAX_TILES_PER_UNIT, span_cap / tw));
    a.tpu = (int)std::max(1LL, std::min<long long>(tpu_cap, (long long)n * n_tiles / target));
    a.n_groups = (n_tiles + a.tpu - 1) / a.tpu;
    a.n_units = load_only ? 0 : (unsigned long long)a.n_groups * (unsigned long long)n;
    cudaError_t e = pick_fused(S, NA, form, nt, mode)(a, ctx->sm_count, ctx->stream);
    if (e != cudaSuccess) return bart_fail(ctx, BART_ECUDA, "launch of emission_fused_kernel failed: %s",
                                           cudaGetErrorString(e));
    return BART_OK;
  };
  // threads per CTA: fixed by the caller, cached per shape, or measured once
  // (each candidate timed with CUDA events on the stream) outside a capture
  char key[160];
  snprintf(key, sizeof(key), "fused%s S%d A%d L%d/%d M%d N%lld n%d b%d span%d m%d", form == FUSED_BULK ? " tma" : ends ? " x4 ends" : form == FUSED_TWO_PAIRS ? " x4" : "",
           S, NA, L, a.ex.L_run, M, (long long)N, n, nb, b->nu_lo ? 1 : 0, mode);
  // (the caller's width is that of the one-wavenumber-per-thread kernels)
  int nt = ctx->em_tile > 0 ? ctx->em_tile : FUSED_THREADS[1];
  auto it = ctx->tiles.find(key);
  if (ctx->em_tile > 0) {
    // fixed by the caller
  } else if (it != ctx->tiles.end()) {
    nt = it->second / fused_width(form, 1);
  } else if (ctx->autotune && (long long)n * max_tiles <= 2LL * ctx->sm_count) {
    // At most about a unit per SM: the widths run alike (31.8, 31.7 and 31.9 us
    // for one spectrum of 2,000 points at 64, 128 and 256 threads), below what
    // one run of each can tell.
    ctx->tiles[key] = fused_width(form, nt);
  } else if (ctx->autotune) {
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    BART_CUDA(ctx, cudaStreamIsCapturing(ctx->stream, &cs));
    if (cs == cudaStreamCaptureStatusNone) {
      cudaEvent_t e0, e1;
      BART_CUDA(ctx, cudaEventCreate(&e0));
      BART_CUDA(ctx, cudaEventCreate(&e1));
      float best = 1e30f;
      // Each candidate is another kernel, which the driver loads at its first
      // use: here, before the timing, where it decided the choice by chance (301
      // ragged spectra took 256 threads in one of six programs, 674 us for 648 at
      // 128).
      for (int cand : FUSED_THREADS)
        if ((st = run(cand, true)) != BART_OK) return st;
      for (int cand : FUSED_THREADS) {
        BART_CUDA(ctx, cudaEventRecord(e0, ctx->stream));
        if ((st = run(cand)) != BART_OK) return st;
        BART_CUDA(ctx, cudaEventRecord(e1, ctx->stream));
        BART_CUDA(ctx, cudaEventSynchronize(e1));
        float ms = 0.f;
        BART_CUDA(ctx, cudaEventElapsedTime(&ms, e0, e1));
        if (ms < best) {
          best = ms;
          nt = cand;
        }
      }
      cudaEventDestroy(e0);
      cudaEventDestroy(e1);
      ctx->tiles[key] = fused_width(form, nt);
    }
  }
  return run(nt);
}
