// Contribution functions of emission spectra (post-processing of Sec. 3) and
// their band means.
//
//   contrib_kernel       the layer loop of the emission kernels with each
//                        layer's term stored instead of accumulated,
//                        C_k = 2 pi sum_i w_i mu_i (B_k + B_{k+1})/2 (t_k - t_{k+1})
//                        for the layer between levels k and k+1, then at the last
//                        level integrated (kb: the deck, the optical-depth limit or
//                        L-1) its blackbody seen through the column, and zeros
//                        below.  sum_k C_k is the flux of the emission kernels.
//                        Its CTAs also find the first and last wavenumber at which
//                        each filter is not zero, a proposal's CTAs taking every
//                        n-th filter (a launch of their own for this and a memset
//                        of its result were 5 of 53 us of one small spectrum).
//   contrib_band_kernel  band means of the rows over those wavenumbers only.
//
// The pass reads 2 S grid rows per (proposal, layer) once and is bound by that
// (a few proposals share few rows): two neighbouring wavenumbers per thread on
// 8-byte loads with the next layer's rows in flight.  The band means were the
// larger part: FP64 sums (GB300 gives 2 FP64 results per clock and SM) of every
// row over the whole grid for every band.  They are now taken over each
// filter's extent only, in pairs of FP32 (two-sum and two-product: the sums
// carry about 48 bits, the band value is FP32), with a band's weights read
// once for 8 rows.  The terms of deep rows go down to FP32's smallest numbers, so
// they are scaled for the products (CB_SCALE).
// Measured, 4 proposals x 100 layers x 100,000 wavenumbers, 4 species, 10
// bands: 3.47 ms before, 0.39 ms now (0.59 ms with every sum in FP64); the rows'
// reads alone need 0.19 ms of the DRAM copy rate.
#include <algorithm>
#include <cmath>

#include "emission_fused.cuh"

using namespace bartem;

namespace {

constexpr int CF_THREADS = 128;
constexpr int CF_TILE = 2 * CF_THREADS;          // wavenumbers per CTA
constexpr int CB_THREADS = 256;
constexpr int CB_ROWS = 8;                       // rows of one proposal per CTA of the band means

// Sum of FP32 values as an unevaluated pair hi + lo.
struct Pair {
  float hi = 0.0f, lo = 0.0f;
};
__device__ __forceinline__ void pair_add(Pair& a, float p, float e) {   // a += p + e, |e| <= ulp(p)
  const float s = a.hi + p, b = s - a.hi;
  a.lo += ((a.hi - (s - b)) + (p - b)) + e;
  a.hi = s;
}
__device__ __forceinline__ void pair_fma(Pair& a, float x, float y) {   // a += x y
  const float p = x * y;
  pair_add(a, p, fmaf(x, y, -p));
}

struct Angles {
  float v[2 * MAX_ANGLES];      // -log2(e) / mu_i, then 2 pi w_i mu_i / 2
};

// Two wavenumbers per thread.  flag[p L + k] is set where a term is not
// finite: its band means then take every wavenumber, so that a NaN reaches
// every band as 0 x NaN does.
template <int S, int NA>
__global__ void __launch_bounds__(CF_THREADS)
contrib_kernel(const float* __restrict__ grid, int L, int M, int64_t N, const LayerTW* __restrict__ tw,
               const float* __restrict__ coef, const float* __restrict__ dpg, const __grid_constant__ Angles ang,
               double nu_start, double dnu, const int64_t* __restrict__ nu_lo, const int64_t* __restrict__ nu_hi,
               float* __restrict__ contrib, const int32_t* __restrict__ act_mask, int* __restrict__ status,
               EmExtra ex, int wide_x, int tau_lim, int* __restrict__ flag, const float* __restrict__ filt,
               int n_bands, int* __restrict__ ext) {
  const int p = blockIdx.x;
  const int tid = threadIdx.x;
  // ext[2 b] = N - first, ext[2 b + 1] = last + 1 over the wavenumbers where
  // filter b is not zero (0, 0: none); ext starts at 0.  The CTAs along y
  // cover the whole grid, whatever the spans are.
  for (int b = p; b < n_bands; b += gridDim.x) {
    const int64_t j = (int64_t)blockIdx.y * CF_TILE + 2 * tid;
    const float* w = filt + (int64_t)b * N + j;
    const bool on_a = j < N && __ldg(w) != 0.0f, on_b = j + 1 < N && __ldg(w + 1) != 0.0f;   // true for NaN
    const int first = __reduce_max_sync(0xffffffffu, on_a ? (int)(N - j) : on_b ? (int)(N - j - 1) : 0);
    const int last = __reduce_max_sync(0xffffffffu, on_b ? (int)(j + 2) : on_a ? (int)(j + 1) : 0);
    if ((tid & 31) == 0 && last > 0) {
      atomicMax(ext + 2 * b, first);
      atomicMax(ext + 2 * b + 1, last);
    }
  }
  if (act_mask && !act_mask[p]) return;
  const int64_t lo = nu_lo ? nu_lo[p] : 0;
  const int64_t hi = nu_hi ? nu_hi[p] : N;
  if (lo < 0 || hi > N || lo >= hi) {
    if (tid == 0 && blockIdx.y == 0) atomicOr(status, BART_DEV_RANGE);
    return;
  }
  const int64_t t0 = (lo & ~(int64_t)1) + (int64_t)blockIdx.y * CF_TILE;   // pairs start on even indices
  if (t0 >= hi) return;
  __shared__ LayerTW s_tw[MAX_LAYERS];
  __shared__ float s_dpg[MAX_LAYERS];
  for (int k = tid; k < L; k += CF_THREADS) {
    s_tw[k] = tw[(int64_t)p * L + k];
    s_dpg[k] = k > 0 ? dpg[k - 1] : 0.0f;
  }
  __syncthreads();
  const int64_t ja = t0 + 2 * tid, jb = ja + 1;
  const bool act_a = ja >= lo && ja < hi, act_b = jb < hi;
  const int64_t ka = ja < hi ? ja : t0, kb_ = jb < hi ? jb : ka;   // idle lanes compute on valid indices
  float xs[S];
#pragma unroll
  for (int s = 0; s < S; ++s) xs[s] = coef[(int64_t)p * S + s];
  const double nua = nu_start + (double)ka * dnu, nub = nu_start + (double)kb_ * dnu;
  const float2 nuf = make_float2((float)nua, (float)nub);
  const float2 c1nu3 = make_float2((float)(2.0 * bartc::H * bartc::C * bartc::C * nua * nua * nua),
                                   (float)(2.0 * bartc::H * bartc::C * bartc::C * nub * nub * nub));
  const float2 chi_r = make_float2((float)(ex.ray * (nua * nua) * (nua * nua)), (float)(ex.ray * (nub * nub) * (nub * nub)));
  // per angle lt = -log2(e) tau / mu and the transmittance t = 2^lt at the current level
  float2 lt[NA], t[NA];
#pragma unroll
  for (int i = 0; i < NA; ++i) {
    lt[i] = f2(0.0f);
    t[i] = f2(1.0f);
  }
  const int64_t sstride = (int64_t)L * M * N;
  const int64_t dm = (M > 1) ? N : 0;
  const float* gj = grid + ka;
  const int64_t dkb = kb_ - ka;
  // 8-byte reads and stores need an even row length and aligned bases
  const bool pair_loads = ((N & 1) == 0) && ((reinterpret_cast<uintptr_t>(grid) & 7) == 0);
  const bool pair_stores = ((N & 1) == 0) && ((reinterpret_cast<uintptr_t>(contrib) & 7) == 0) && act_a && act_b;

  auto fetch = [&](int k, float2* x, float2* y) {
    const float* g = gj + s_tw[k].row;
#pragma unroll
    for (int s = 0; s < S; ++s) {
      const float* b = g + s * sstride;
      if (pair_loads) {
        x[s] = __ldg(reinterpret_cast<const float2*>(b));
        y[s] = __ldg(reinterpret_cast<const float2*>(b + dm));
      } else {
        x[s] = make_float2(__ldg(b), __ldg(b + dkb));
        y[s] = make_float2(__ldg(b + dm), __ldg(b + dm + dkb));
      }
    }
  };
  auto chi_of = [&](int k, const float2* x, const float2* y) {
    const float2 w = f2(s_tw[k].w);
    float2 chi = chi_r;
#pragma unroll
    for (int s = 0; s < S; ++s) chi = fma2(f2(xs[s]), fma2(w, sub2(y[s], x[s]), x[s]), chi);
    return chi;
  };
  // (one rounding of c2 nu / T, which is up to 100 and enters B as an exponent)
  auto planck_k = [&](int k) {
    const float2 x = mul2(nuf, f2(s_tw[k].c2_t));
    return wide_x ? make_float2(planck<true>(c1nu3.x, x.x), planck<true>(c1nu3.y, x.y))
                  : make_float2(planck<false>(c1nu3.x, x.x), planck<false>(c1nu3.y, x.y));
  };
  float* out = contrib + (int64_t)p * L * N + ja;
  bool bad = false;
  auto store = [&](int row, float2 v) {
    bad = (act_a && !(fabsf(v.x) <= 3.402823466e38f)) || (act_b && !(fabsf(v.y) <= 3.402823466e38f));
    float* o = out + (int64_t)row * N;
    if (pair_stores) {
      *reinterpret_cast<float2*>(o) = v;
    } else {
      if (act_a) o[0] = v.x;
      if (act_b) o[1] = v.y;
    }
    if (bad && flag) flag[(int64_t)p * L + row] = 1;
  };
  auto bottom = [&](float2 B) {                // the level's blackbody through the column
    float2 c = f2(0.0f);
#pragma unroll
    for (int i = 0; i < NA; ++i) c = fma2(f2(ang.v[NA + i]), mul2(mul2(f2(2.0f), B), t[i]), c);
    return c;
  };

  float2 cx[S], cy[S], nx[S], ny[S];
  fetch(0, cx, cy);
  fetch(min(1, ex.L_run - 1), nx, ny);
  float2 chi_prev = chi_of(0, cx, cy), B_prev = planck_k(0), tau = f2(0.0f);
  float2 low = f2(0.0f);                       // the bottom term of a wavenumber that stopped
  int end_a = L, end_b = L;                    // the level where it stopped
  int k = 1;
  for (; k < ex.L_run; ++k) {
    const float2 chi = chi_of(k, nx, ny), B = planck_k(k);   // one set of rows in registers
    fetch(min(k + 1, ex.L_run - 1), nx, ny);
    const float2 dtau = mul2(add2(chi_prev, chi), f2(s_dpg[k]));
    const float2 Bsum = add2(B_prev, B);
    tau = add2(tau, dtau);
    float2 C = f2(0.0f);
#pragma unroll
    for (int i = 0; i < NA; ++i) {
      lt[i] = fma2(dtau, f2(ang.v[i]), lt[i]);
      const float2 te = ex2_2(lt[i]);
      C = fma2(f2(ang.v[NA + i]), mul2(Bsum, sub2(t[i], te)), C);
      t[i] = te;
    }
    chi_prev = chi;
    B_prev = B;
    if (tau_lim) {
      // a wavenumber that stopped at level end: its bottom term there, zeros after
      if (k > end_a) C.x = (k - 1 == end_a) ? low.x : 0.0f;
      if (k > end_b) C.y = (k - 1 == end_b) ? low.y : 0.0f;
    }
    store(k - 1, C);
    if (tau_lim) {
      const bool sa = end_a == L && tau.x > ex.tau_cut, sb = end_b == L && tau.y > ex.tau_cut;
      if (sa || sb) {
        const float2 v = bottom(B);
        if (sa) { end_a = k; low.x = v.x; }
        if (sb) { end_b = k; low.y = v.y; }
      }
      if (end_a < L && end_b < L) {
        ++k;
        break;
      }
    }
  }
  // k - 1 is now the last level integrated by either wavenumber
  float2 Cb = bottom(B_prev);
  if (end_a < L) Cb.x = (end_a == k - 1) ? low.x : 0.0f;
  if (end_b < L) Cb.y = (end_b == k - 1) ? low.y : 0.0f;
  store(k - 1, Cb);
  for (int q = k; q < L; ++q) store(q, f2(0.0f));
}

// The terms are multiplied by CB_SCALE (exactly) before their products with the
// weights, so that no product's low part that matters lies below the FP32 range:
// what 2^17 products lose there, 2^-149 each, is 2^-188 of a band's sum, for
// weights that sum to CB_LEAST 2^-175 of its value, below 2^-26 of the smallest
// FP32 number.  Sums that are larger than CB_MOST or not finite, and smaller weights, are
// taken again in FP64.
constexpr float CB_SCALE = 7.205759403792794e16f;                                   // 2^56
constexpr double CB_LEAST = 1.220703125e-4, CB_MOST = 1.329227995784916e36;         // 2^-13, 2^120

// Band means of CB_ROWS contribution rows of one proposal: trapezoid weights
// over the proposal's span, the sums as FP32 pairs per thread and across the
// warp, FP64 across the warps.
__global__ void __launch_bounds__(CB_THREADS)
contrib_band_kernel(const float* __restrict__ contrib, int L, int64_t N, const int64_t* __restrict__ nu_lo,
                    const int64_t* __restrict__ nu_hi, const float* __restrict__ filt, int n_bands,
                    const int32_t* __restrict__ act_mask, const int* __restrict__ ext, const int* __restrict__ flag,
                    float* __restrict__ out) {
  const int groups = (L + CB_ROWS - 1) / CB_ROWS;
  const int p = blockIdx.x / groups, b = blockIdx.y;
  if (act_mask && !act_mask[p]) return;
  const int64_t lo = nu_lo ? nu_lo[p] : 0, hi = nu_hi ? nu_hi[p] : N;
  if (lo < 0 || hi > N || lo >= hi) return;   // reported by contrib_kernel
  const int k0 = (blockIdx.x % groups) * CB_ROWS, nr = min(CB_ROWS, L - k0);
  bool any = false;                            // a row with a term that is not finite
  for (int r = 0; r < nr; ++r) any |= flag[(int64_t)p * L + k0 + r] != 0;
  const int64_t j0 = any ? lo : max(lo, N - ext[2 * b]), j1 = any ? hi : min(hi, (int64_t)ext[2 * b + 1]);
  const float* w = filt + (int64_t)b * N;
  const float* c[CB_ROWS];
#pragma unroll
  for (int r = 0; r < CB_ROWS; ++r) c[r] = contrib + ((int64_t)p * L + k0 + min(r, nr - 1)) * N;
  Pair num[CB_ROWS], den;
  for (int64_t j = j0 + threadIdx.x; j < j1; j += CB_THREADS) {
    const float dw = (hi - lo == 1) ? 1.0f : ((j == lo || j == hi - 1) ? 0.5f : 1.0f);
    const float W = __ldg(w + j) * dw;         // exact: dw is 1 or 1/2
    pair_add(den, W, 0.0f);
#pragma unroll
    for (int r = 0; r < CB_ROWS; ++r) pair_fma(num[r], W, __ldg(c[r] + j) * CB_SCALE);
  }
  __shared__ double sh[CB_THREADS / 32][CB_ROWS + 1];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  auto reduce = [&](Pair v, int slot) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const float h = __shfl_xor_sync(0xffffffffu, v.hi, o), l = __shfl_xor_sync(0xffffffffu, v.lo, o);
      pair_add(v, h, 0.0f);
      v.lo += l;
    }
    if (lane == 0) sh[warp][slot] = (double)v.hi + (double)v.lo;
  };
#pragma unroll
  for (int r = 0; r < CB_ROWS; ++r) reduce(num[r], r);
  reduce(den, CB_ROWS);
  __syncthreads();
  double a = 0.0, d = 0.0;
  auto add = [&]() {
    a = d = 0.0;
    for (int q = 0; q < CB_THREADS / 32; ++q) {
      a += sh[q][min((int)threadIdx.x, CB_ROWS)];
      d += sh[q][CB_ROWS];
    }
  };
  add();
  if (__syncthreads_or((int)threadIdx.x < nr && !(fabs(a) <= CB_MOST && d >= CB_LEAST && d <= CB_MOST))) {
    double sum[CB_ROWS] = {}, weight = 0.0;    // the products of FP32 values are exact
    for (int64_t j = j0 + threadIdx.x; j < j1; j += CB_THREADS) {
      const float dw = (hi - lo == 1) ? 1.0f : ((j == lo || j == hi - 1) ? 0.5f : 1.0f);
      const double W = (double)(__ldg(w + j) * dw);
      weight += W;
#pragma unroll
      for (int r = 0; r < CB_ROWS; ++r) sum[r] = fma(W, (double)__ldg(c[r] + j), sum[r]);
    }
    auto put = [&](double v, int slot) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
      if (lane == 0) sh[warp][slot] = v;
    };
#pragma unroll
    for (int r = 0; r < CB_ROWS; ++r) put(sum[r], r);
    put(weight, CB_ROWS);
    __syncthreads();
    add();
  } else {
    a *= 1.0 / (double)CB_SCALE;
  }
  if ((int)threadIdx.x < nr)
    out[((int64_t)p * L + k0 + threadIdx.x) * n_bands + b] = d > 0.0 ? (float)(a / d) : 0.0f;
}

using CfLauncher = void (*)(dim3, cudaStream_t, const float*, int, int, int64_t, const LayerTW*, const float*,
                            const float*, const Angles&, double, double, const int64_t*, const int64_t*, float*,
                            const int32_t*, int*, EmExtra, int, int, int*, const float*, int, int*);

template <int S, int NA>
void launch_contrib(dim3 g, cudaStream_t st, const float* grid, int L, int M, int64_t N, const LayerTW* tw,
                    const float* coef, const float* dpg, const Angles& ang, double nu_start, double dnu,
                    const int64_t* lo, const int64_t* hi, float* contrib, const int32_t* active, int* status,
                    EmExtra ex, int wide_x, int tau_lim, int* flag, const float* filt, int n_bands, int* ext) {
  contrib_kernel<S, NA><<<g, CF_THREADS, 0, st>>>(grid, L, M, N, tw, coef, dpg, ang, nu_start, dnu, lo, hi, contrib,
                                                  active, status, ex, wide_x, tau_lim, flag, filt, n_bands, ext);
}

template <int S>
CfLauncher pick_angles(int na) {
  switch (na) {
    case 1: return launch_contrib<S, 1>;
    case 2: return launch_contrib<S, 2>;
    case 4: return launch_contrib<S, 4>;
    case 8: return launch_contrib<S, 8>;
    case 16: return launch_contrib<S, 16>;
    default: return nullptr;
  }
}

CfLauncher pick_contrib(int S, int na) {
  switch (S) {
    case 1: return pick_angles<1>(na);
    case 2: return pick_angles<2>(na);
    case 3: return pick_angles<3>(na);
    default: return pick_angles<4>(na);
  }
}

}  // namespace

extern "C" bart_status bart_contribution_functions(bart_ctx* ctx, const bart_grid_desc* g, const bart_fwd_cfg* c,
                                                   const bart_batch* b, float* contrib, const bart_filters* f,
                                                   float* bands) {
  if (!ctx) return BART_EINVAL;
  bart_status st;
  if ((st = check_forward_request(ctx, g, c, b)) != BART_OK) return st;
  BART_REQUIRE(ctx, c->geometry == BART_EMISSION, "contribution functions are defined for emission only");
  BART_REQUIRE(ctx, contrib || bands, "nothing requested: contrib and bands are both NULL");
  int nb = 0;
  if (bands) {
    BART_REQUIRE(ctx, f && f->weights, "bands requested without filters");
    nb = f->n_bands;
    BART_REQUIRE(ctx, nb >= 1 && nb <= 65535, "n_bands must be in [1, 65535]");
  }
  CfLauncher launch = pick_contrib(g->n_species, c->n_angles);
  BART_REQUIRE(ctx, launch != nullptr, "n_angles must be 1, 2, 4, 8 or 16");
  BART_REQUIRE(ctx, g->n_species <= 4, "contribution functions support 1-4 species");
  const int L = g->n_layers, M = g->n_temps, n = b->n;
  const int64_t N = g->nu.n_nu;
  BART_REQUIRE(ctx, (int64_t)n * L <= 2147483647LL, "n x n_layers too large");
  BART_CUDA(ctx, cudaSetDevice(ctx->device));
  float* out = contrib;
  if (!out) {
    void* p = nullptr;
    if ((st = bart_scratch(ctx, "cf_rows", (size_t)n * L * N * sizeof(float), &p)) != BART_OK) return st;
    out = (float*)p;
  }
  // band extents and the rows' flags, both cleared by the prologue's launch
  int *ext = nullptr, *flag = nullptr;
  size_t words = 0;
  std::vector<void*> held;
  if (nb > 0) {
    words = 2 * (size_t)nb + (size_t)n * L;
    if ((st = bart_scratch_any(ctx, "cf_ext", words * sizeof(int), (void**)&ext, &held)) != BART_OK) return st;
    flag = ext + 2 * nb;
  }
  EmPrep pr;
  if ((st = emission_prologue(ctx, g, c, b, &pr, ext, words)) != BART_OK) {
    bart_scratch_give_back(ctx, &held);
    return st;
  }
  const int mode = emission_mode(g, c);
  std::vector<double> mu, w;
  gauss_legendre01(c->n_angles, mu, w);
  Angles ang{};
  for (int i = 0; i < c->n_angles; ++i) {
    ang.v[i] = (float)(-1.4426950408889634 / mu[i]);
    ang.v[c->n_angles + i] = (float)(2.0 * bartc::PI * w[i] * mu[i] * 0.5);
  }
  const int64_t n_tiles = (N + 1 + CF_TILE - 1) / CF_TILE;     // an odd span start takes one pair more
  launch(dim3((unsigned)n, (unsigned)n_tiles), ctx->stream, g->grid, L, M, N, pr.tw, pr.coef, pr.dc + pr.off_dpg,
         ang, g->nu.nu_start_cm, g->nu.dnu_cm, b->nu_lo, b->nu_hi, out, b->active, ctx->d_status,
         emission_extra(g, c), mode & 1, (mode >> 1) & 1, flag, nb > 0 ? f->weights : nullptr, nb, ext);
  st = bart_check_launch(ctx, "contrib_kernel");
  if (st == BART_OK && nb > 0) {
    const int64_t groups = (L + CB_ROWS - 1) / CB_ROWS;
    contrib_band_kernel<<<dim3((unsigned)(n * groups), (unsigned)nb), CB_THREADS, 0, ctx->stream>>>(
        out, L, N, b->nu_lo, b->nu_hi, f->weights, nb, b->active, ext, flag, bands);
    st = bart_check_launch(ctx, "contrib_band_kernel");
  }
  bart_scratch_give_back(ctx, &held);
  return st;
}
