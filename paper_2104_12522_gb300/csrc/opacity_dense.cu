// Opacity of dense line lists: the same sum over lines as opacity_kernel,
// arranged by distance so that the cost of a line far from a point is shared
// with its neighbours.
//
// The 5e6-line grid holds 17 lines per wavenumber point and each line reaches
// 2,500 points, so most of the work of a line-by-line sum is far wings of lines
// that lie within a fraction of a point of one another.  Lines are taken in
// source blocks of 8 grid points (by their nearest point jc).  For a point j
//   near   source blocks closer than m1 blocks: every line evaluated on its own
//          (dense_near_kernel);
//   mid    source blocks from m1 blocks on, by their moments;
//   far    blocks of 32 points from m2 such blocks on, by theirs;
//   edges  the block that a cutoff edge of j divides, by the moments of its
//          groups of lines with one and the same cutoff window [jlo, jhi]: a
//          line is counted at exactly the points of its window.
//
// Moments.  With lengths in grid points, V(d) = (S / pi) Im sum_n E[z^n] /
// d^(n+1) far from the line, z = delta + g + i gamma, delta the line's offset
// from the block's centre and g Gaussian with the Doppler width (the asymptotic
// series of the Voigt profile and the expansion about the centre in one).  The
// E[z^n] follow K_0 = 1, K_1 = w, K_(n+1) = w K_n + n sigma^2 K_(n-1),
// w = delta + i gamma; a block keeps I_n = sum_lines (S / pi) Im K_n, n = 1 ..
// DN_P.  m1 and m2 keep sqrt(half^2 + gamma^2) <= DN_RHO x the distance: the
// first term left out is then below 9 DN_RHO^8 = 1.3e-6 of a line's own at the
// nearest point for the line farthest from the centre, far below that in a sum.
//
// Lorentz widths beyond about 3 points need moments about a complex centre:
// with the lines of a block in bins of gamma_ref (ratio <= sqrt 2 within a bin),
// u = delta + g + i (gamma - gamma_c) about the bin's middle gamma_c and
// Z = d - i gamma_c, V = (S / pi) Im sum_n E[u^n] / Z^(n+1): |Z| >= gamma_c, so a
// wide profile is smooth on the scale of a block and needs no near lines at
// all.  DN_PC terms hold where |u| <= DN_RHOC |Z| (15 DN_RHOC^14 = 9e-7).
// Distances where the moments about the real centre hold take those (one set
// per block, half the operations).
//
// Near lines.  A warp takes one source block, a lane one line: constants,
// moments and all the block's near points (8 (2 m1 - 1), the same for all lanes)
// without a line's constants leaving its registers, so lanes agree on how far
// they are from a point and the profile's form is chosen once per point for the
// warp: shifted Lorentz where its error is below EPS_L, the 4-point
// Gauss-Hermite form (a positive sum of Lorentzians: no cancellation; <= 3.6e-7
// for |z| >= 9) from |x| = 9 on, the full profile closer in.  Per-lane sums
// stay in shared memory over the block's lines and are folded into a TwoSum
// pair every 8 chunks; dense_sum_kernel adds the near windows of the 2 m1 - 1
// blocks around a point, then the moments.  No atomics: every sum has a fixed
// order.
//
// Used (dense_applies, dense_plan_kernel) for lists of at least DN_DENSITY lines
// per point, where blocks pay for their fixed cost, and for cells whose widths
// fit: Doppler widths that keep |x| >= 9 from the first mid block on; Lorentz
// widths up to about 3 grid points, or gamma_ref within a factor 4 over the
// list (4 bins) and widths below a sixth of the cutoff (the moments of the
// divided blocks are about the real centre), or a cutoff so short that the near
// window holds all of it.  Other cells go line by line.
// Measured: one species of the 5e6-line grid (1.67e6 lines, 100,000 points), 10
// layers over 1e-8 .. 100 bar x 20 temperatures: 169 ms line by line, 58 ms with
// the 160 cells of widths up to 3 points here, 44 ms with the wider ones too;
// 2 species x 10,000 lines, 60 cells, 2,000 points 1 cm^-1 apart: 2.59 ms and
// 0.33 ms.
#include <algorithm>
#include <cmath>

#include "opacity.cuh"

using namespace bartop;

namespace {

constexpr int DN_B = 8;                     // points of a source block
constexpr int DN_P = 8;                     // moments
constexpr int DN_M1 = 4, DN_M1_MAX = 5;     // near radius in blocks
constexpr int DN_WIN = (2 * DN_M1_MAX - 1) * DN_B;   // near points of a block, at most
constexpr int DN_GROUPS = 20;               // groups of a block: jlo and jhi each step at most 9 times
constexpr float DN_RHO = 0.14f;
constexpr int DN_BINS = 4;                  // bins of gamma_ref
constexpr int DN_PC = 14;                   // moments about a complex centre
constexpr float DN_RHOC = 0.305f;
constexpr float DN_RHO_EDGE = 0.175f;       // divided blocks: 9 x 0.175^8 = 8e-6 of a line at its cutoff
constexpr double DN_DENSITY = 0.5;          // lines per point
constexpr int DN_WARPS = 4;
constexpr int DN_FOLD = 8;                  // chunks of 32 lines between two folds
constexpr float DN_EPS_L = 2e-6f;           // bound of the shifted Lorentz form
constexpr size_t DN_SCRATCH = (size_t)256 << 20;     // moments and windows of a batch of cells (a third of it is
                                                     // touched for a cell: within L2)

struct DensePoint {           // per grid point (indexes of groups and blocks)
  int gl, gr;                 // groups whose window holds the point: [gl, gr)
  int bl, br;                 // blocks all of whose lines do: [bl, br)
};

// Lines whose window is not empty: [r[0], r[1]).
__global__ void dense_range_kernel(const int* __restrict__ jlo, const int* __restrict__ jhi, int n_lines, int n_nu,
                                   int* __restrict__ r) {
  r[0] = (int)lower_bound_i(jhi, 0, n_lines, 0);
  r[1] = (int)lower_bound_i(jlo, r[0], n_lines, n_nu);
}

__device__ __forceinline__ int block_of(int jc, int boff) { return (jc >> 3) + boff; }

// First line of each block.
__global__ void dense_block_kernel(const LineWin* __restrict__ win, const int* __restrict__ range, int boff, int nb,
                                   int* __restrict__ lstart) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b > nb) return;
  int lo = range[0], hi = range[1];
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    if (block_of(win[mid].jc, boff) < b) lo = mid + 1; else hi = mid;
  }
  lstart[b] = lo;
}

constexpr int GR_TILE = 1024;
// 1 where line i is the first of a group: lines of one block and one window.
__device__ __forceinline__ int group_first(const LineWin* __restrict__ win, const int* __restrict__ range, int64_t i) {
  if (i < range[0] || i >= range[1]) return 0;
  if (i == range[0]) return 1;
  const LineWin a = win[i - 1], b = win[i];
  return a.jlo != b.jlo || a.jhi != b.jhi || (a.jc >> 3) != (b.jc >> 3);
}

__global__ void __launch_bounds__(GR_TILE)
dense_group_count_kernel(const LineWin* __restrict__ win, const int* __restrict__ range, int* __restrict__ count) {
  const int n = __syncthreads_count(group_first(win, range, (int64_t)blockIdx.x * GR_TILE + threadIdx.x));
  if (threadIdx.x == 0) count[blockIdx.x] = n;
}

// Inclusive sum over the CTA's GR_TILE threads.
__device__ int cta_scan(int v, int* sh) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int t = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= o) v += t;
  }
  __syncthreads();
  if (lane == 31) sh[warp] = v;
  __syncthreads();
  if (warp == 0) {
    int t = sh[lane];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int u = __shfl_up_sync(0xffffffffu, t, o);
      if (lane >= o) t += u;
    }
    sh[lane] = t;
  }
  __syncthreads();
  return v + (warp > 0 ? sh[warp - 1] : 0);
}

// Exclusive sums of the tiles' counts, in place; the total behind them.
__global__ void __launch_bounds__(GR_TILE) dense_group_scan_kernel(int* __restrict__ count, int tiles) {
  __shared__ int sh[32];
  int base = 0;
  for (int t0 = 0; t0 < tiles; t0 += GR_TILE) {
    const int t = t0 + threadIdx.x, v = t < tiles ? count[t] : 0;
    const int s = cta_scan(v, sh);
    if (t < tiles) count[t] = base + s - v;
    base += sh[31];
  }
  if (threadIdx.x == 0) count[tiles] = base;
}

__global__ void __launch_bounds__(GR_TILE)
dense_group_kernel(const LineWin* __restrict__ win, const int* __restrict__ range, const int* __restrict__ count,
                   int64_t n_lines, int* __restrict__ gid) {
  __shared__ int sh[32];
  const int64_t i = (int64_t)blockIdx.x * GR_TILE + threadIdx.x;
  const int s = cta_scan(group_first(win, range, i), sh);
  if (i < n_lines) gid[i] = count[blockIdx.x] + s - 1;
}

__global__ void dense_first_group_kernel(const int* __restrict__ lstart, const int* __restrict__ range,
                                         const int* __restrict__ gid, const int* __restrict__ total, int nb,
                                         int* __restrict__ gfirst) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b <= nb) gfirst[b] = lstart[b] < range[1] ? gid[lstart[b]] : *total;
}

__global__ void dense_point_kernel(const LineWin* __restrict__ win, const int* __restrict__ jlo,
                                   const int* __restrict__ jhi, const int* __restrict__ range,
                                   const int* __restrict__ gid, const int* __restrict__ total,
                                   const int* __restrict__ lstart, int boff, int nb, int n_nu,
                                   DensePoint* __restrict__ pts) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= n_nu) return;
  const int i0 = range[0], i1 = range[1];
  const int il = (int)lower_bound_i(jhi, i0, i1, j), ir = (int)lower_bound_i(jlo, il, i1, j + 1);
  DensePoint p;
  p.gl = il < i1 ? gid[il] : *total;
  p.gr = ir < i1 ? gid[ir] : *total;
  p.bl = nb;
  if (il < i1) {
    const int b = block_of(win[il].jc, boff);
    p.bl = lstart[b] == il ? b : b + 1;
  }
  p.br = ir < i1 ? block_of(win[ir].jc, boff) : nb;
  p.bl = min(max(p.bl, 0), nb);             // in range for a list that is not sorted, too
  p.br = min(max(p.br, 0), nb);
  pts[j] = p;
}

// stat[0]: largest gamma_ref (bits of a non-negative float), stat[1]: a value
// that is negative or not a number, stat[2]: 0x7fffffff - bits of the smallest.
__global__ void __launch_bounds__(256)
dense_gamma_kernel(const float* __restrict__ gref, int64_t n, int* __restrict__ stat) {
  unsigned m = 0, mi = 0;
  bool bad = false;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const float g = gref[i];
    bad |= !(g >= 0.0f);
    const unsigned bits = __float_as_uint(fmaxf(g, 0.0f)) & 0x7fffffffu;
    m = max(m, bits);
    mi = max(mi, 0x7fffffffu - bits);
  }
  m = __reduce_max_sync(0xffffffffu, m);
  mi = __reduce_max_sync(0xffffffffu, mi);
  bad = __any_sync(0xffffffffu, bad);
  if ((threadIdx.x & 31) == 0) {
    if (m) atomicMax(stat, (int)m);
    if (mi) atomicMax(stat + 2, (int)mi);
    if (bad) atomicOr(stat + 1, 1);
  }
}

// Bins of gamma_ref: n of equal ratio over the list's range, 0 if it does not
// fit; middle and reach of the bins, at 1 bar and 296 K.
struct DenseBins {
  int n;
  float inv_g0, inv_lr;       // bin of g: floor(log2(g inv_g0) inv_lr)
  float eta;                  // half width of a bin over its middle
  float c[DN_BINS];
};

__device__ DenseBins dense_bins(const int* __restrict__ stat) {
  DenseBins r{};
  const float g1 = __int_as_float(stat[0]), g0 = __int_as_float(0x7fffffff - stat[2]);
  if (!(g0 > 1e-30f) || !(g1 < 1e30f)) return r;
  const float lr = log2f(g1 / g0);
  const int n = max(1, (int)ceilf(2.0f * lr - 1e-3f));
  if (n > DN_BINS) return r;
  r.n = n;
  r.inv_g0 = 1.0f / g0;
  r.inv_lr = lr > 0.0f ? (float)n / lr : 0.0f;
  const float rb = exp2f(lr / n);
  r.eta = (rb - 1.0f) / (rb + 1.0f);
  for (int q = 0; q < n; ++q) r.c[q] = g0 * exp2f(lr * q / n) * 0.5f * (1.0f + rb);
  return r;
}

__global__ void dense_plan_kernel(const CellConst* __restrict__ cells, int n_cells, const int* __restrict__ stat,
                                  float inv_dnu, int reach, DensePlan* __restrict__ plan,
                                  DenseBins* __restrict__ bins) {
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  const DenseBins bn = dense_bins(stat);
  if (c == 0) *bins = bn;
  if (c >= n_cells) return;
  DensePlan p{DN_NONE, 0, 0, 0};
  const float scale = cells[c].gfac * inv_dnu, g = __int_as_float(stat[0]) * scale;   // widest line, in points
  if (cells[c].dense && !stat[1] && g < 1e6f) {
    // a point of block t is at least 8 m - 3.5 points from the centre of block t +- m
    const int m1 = max(DN_M1, (int)ceilf((sqrtf(16.0f + g * g) / DN_RHO + 3.5f) / 8.0f));
    const int m2 = max(4, (int)ceilf((sqrtf(256.0f + g * g) / DN_RHO + 15.5f) / 32.0f));
    if (m1 <= DN_M1_MAX) {
      p = {DN_REAL, m1, 0, m2};
    } else if (8 * (DN_M1_MAX - 1) > reach) {    // the near window holds every line's points
      p = {DN_REAL, DN_M1_MAX, 0, m2};
    } else if (bn.n > 0 && sqrtf(16.0f + g * g) <= DN_RHO_EDGE * (float)(reach - 8)) {
      float d8 = 0.0f, d32 = 0.0f;               // squared distances from which the complex moments hold
      for (int q = 0; q < bn.n; ++q) {
        const float gc = bn.c[q] * scale, e2 = bn.eta * bn.eta * gc * gc;
        d8 = fmaxf(d8, (16.0f + e2) / (DN_RHOC * DN_RHOC) - gc * gc);
        d32 = fmaxf(d32, (256.0f + e2) / (DN_RHOC * DN_RHOC) - gc * gc);
      }
      p.kind = DN_COMPLEX;
      p.m1 = d8 > 0.0f ? (int)ceilf((sqrtf(d8) + 3.5f) / 8.0f) : 0;
      p.mh = d32 > 0.0f ? (int)ceilf((sqrtf(d32) + 15.5f) / 32.0f) : 0;
      p.m2 = max(m2, p.mh);
    }
  }
  plan[c] = p;
}

// G(x) = -Im w'(x) = (2 / sqrt(pi)) (2 x F(x) - 1), F Dawson's integral, x >= 0:
// up to 9.3 a rational function of x^2 fitted (least squares, reweighted
// towards the largest error) to |dG| <= 1e-6 (50 e^(-x^2) + |G|) in FP32 -- near
// its zero at 0.92 the Gaussian term of the profile is far larger -- and its
// asymptotic series beyond.
__device__ __forceinline__ float dawson_g(float x, float u) {
  float n = 4.43394788e-06f, d = 7.85838861e-06f;
  n = fmaf(n, u, -3.46022744e-05f);
  n = fmaf(n, u, 4.63677612e-04f);
  n = fmaf(n, u, -2.12909611e-04f);
  n = fmaf(n, u, 2.23139278e-02f);
  n = fmaf(n, u, -9.76259707e-02f);
  n = fmaf(n, u, 1.38819137f);
  n = fmaf(n, u, -1.12835006f);
  d = fmaf(d, u, -7.29758443e-05f);
  d = fmaf(d, u, 8.88062378e-04f);
  d = fmaf(d, u, -8.60452054e-04f);
  d = fmaf(d, u, 1.95862562e-02f);
  d = fmaf(d, u, 6.41052559e-02f);
  d = fmaf(d, u, 2.97722797e-01f);
  d = fmaf(d, u, 7.68709942e-01f);
  d = fmaf(d, u, 1.0f);
  const bool far = x > 9.3f;
  const float t = bartw::rcp_approx(far ? u : d);
  float s = fmaf(t, 29.53125f, 6.5625f);       // (2k-1)!! / 2^k, k = 5 .. 1
  s = fmaf(s, t, 1.875f);
  s = fmaf(s, t, 0.75f);
  s = fmaf(s, t, 0.5f);
  return t * (far ? 1.1283791670955126f * s : n);
}

// Re w(x + i y) for 0 <= y <= SMALL_Y: the expansion in y of small_y_re
// (faddeeva.cuh) without a branch or a table.
__device__ __forceinline__ float core_small(float x, float y) {
  constexpr float L2E_LO = (float)(1.4426950408889634 - (double)LOG2EF);
  const float u = x * x, lo = fmaf(x, x, -u);          // x^2 = u + lo
  const float ah = -u * LOG2EF;
  const float al = -fmaf(u, LOG2EF, ah) - fmaf(lo, LOG2EF, u * L2E_LO);
  const float e = ex2f_approx(ah) * fmaf(al, LN2F_, 1.0f);
  const float g = dawson_g(x, u);
  const float y2 = y * y;
  const float cub = x < 40.0f ? fmaf(g, fmaf(-4.0f, u, 6.0f), 2.2567583341910252f) : 0.0f;
  return fmaf(e, fmaf(y2, fmaf(-2.0f, u, 1.0f), 1.0f), y * fmaf(y2 * (1.0f / 6.0f), cub, g));
}

// (sqrt(pi) / y) Re w by Gauss-Hermite quadrature of w = (i / pi) int e^(-t^2) /
// (z - t) dt: Re w = (y / pi) sum_k w_k / ((x - t_k)^2 + y^2), the two nodes +-t
// as 2 w s / (s^2 - 4 x^2 t^2) with s = x^2 + y^2 + t^2.  Weights divided by
// sqrt(pi) here.  4 nodes: <= 3.6e-7 for |z| >= 9.
__device__ __forceinline__ float gh4_ratio(float x, float y2) {
  constexpr float T1 = 0.27525512860841095f, T2 = 2.7247448713915889f;      // t^2
  constexpr float W1 = 0.90824829046386302f, W2 = 0.091751709536136983f;    // 2 w / sqrt(pi)
  const float u = x * x, s1 = u + (y2 + T1), s2 = u + (y2 + T2);
  const float d1 = fmaf(s1, s1, -4.0f * T1 * u), d2 = fmaf(s2, s2, -4.0f * T2 * u);
  const float n = fmaf(W2 * s2, d1, W1 * s1 * d2);
  return n * bartw::rcp_approx(d1 * d2);
}
// 8 nodes: <= 1.5e-7 for |z| >= 5, plus the residue e^(y^2 - x^2) cos 2xy that
// the quadrature misses near the real axis.
__device__ __forceinline__ float gh8_re(float x, float y) {
  constexpr float T[4] = {0.14530352150331707f, 1.3390972881263614f, 3.9269635013582872f, 8.5886356890120343f};
  constexpr float Wt[4] = {0.746024515358155f, 0.234479815323518f, 0.0192704402415765f, 0.00022522907675073f};
  const float u = x * x, y2 = y * y;
  float r = 0.0f;
#pragma unroll
  for (int k = 0; k < 4; k += 2) {
    const float s1 = u + (y2 + T[k]), s2 = u + (y2 + T[k + 1]);
    const float d1 = fmaf(s1, s1, -4.0f * T[k] * u), d2 = fmaf(s2, s2, -4.0f * T[k + 1] * u);
    r = fmaf(fmaf(Wt[k + 1] * s2, d1, Wt[k] * s1 * d2), bartw::rcp_approx(d1 * d2), r);
  }
  const float g = fmaf(y, y, -u);
  const float e = (y < 1.0f && g > -87.0f) ? __expf(g) * __cosf(2.0f * x * y) : 0.0f;
  return fmaf(bartw::INV_SQRTPI * y, r, e);
}
__device__ __forceinline__ float core_any(float x, float y, const float2* __restrict__ wtab) {
  return fmaf(x, x, y * y) < 25.0f ? bartw::taylor_re<1>(x, y, wtab) : gh8_re(x, y);
}

struct DenseArgs {
  const LineWin* win;
  const float* gref;
  const int* lstart;
  const int* gid;
  const int* gfirst;
  const CellConst* cells;
  const DensePlan* plan;
  const DensePoint* pts;
  const DenseBins* bins;
  const int* smax;
  const int* tmap;
  const float2* wtab;
  float ln_rel, dnu, inv_dnu, w_scale;       // w_scale: 1 / (pi dnu)
  int boff, nb, n_nu, reach, c0;             // reach: points within the cutoff on each side; c0: first cell
  int64_t g_stride;
  float* window;                             // [cell][nb][DN_WIN]
  float* m8;                                 // [cell][nb][DN_P]
  float* m32;                                // [cell][nb / 4][DN_P]
  float* mg;                                 // [cell][g_stride][DN_P]
  float2* mc8;                               // [cell][nb][DN_BINS][DN_PC], complex centres
  float2* mc32;                              // [cell][nb / 4][DN_BINS][DN_PC]
  float* out;
};

struct NearShared {
  float4 acc[DN_WARPS][DN_WIN / 4][32];      // per lane, four neighbouring points
  float group[DN_WARPS][DN_GROUPS][DN_P];
};

__global__ void __launch_bounds__(32 * DN_WARPS)
dense_near_kernel(const __grid_constant__ DenseArgs a) {
  extern __shared__ __align__(16) unsigned char dn_smem[];
  NearShared& sh = *reinterpret_cast<NearShared*>(dn_smem);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int b = blockIdx.x * DN_WARPS + warp;
  const int cell = a.c0 + blockIdx.y;
  const DensePlan plan = a.plan[cell];
  if (plan.kind == DN_NONE || b >= a.nb) return;   // warps are independent: no CTA barrier below
  const int l0 = a.lstart[b], l1 = a.lstart[b + 1];
  // (the bounds hold for any list; a sorted one has no block with more groups)
  const int g0 = a.gfirst[b], ng = max(0, min(min(a.gfirst[b + 1] - g0, DN_GROUPS), (int)a.g_stride - g0));
  const CellConst cc = a.cells[cell];
  const float ln_thr = a.smax ? ordered_float(a.smax[a.tmap[cell]]) + a.ln_rel : -3.0e38f;
  const int m1 = max(plan.m1, 1);
  const int n_pts = plan.m1 > 0 ? (2 * m1 - 1) * DN_B : 0, steps = n_pts / 4;
  const int w0 = (b - a.boff - (m1 - 1)) * DN_B;              // grid index of the window's first point
  const float centre = (float)((m1 - 1) * DN_B) + 3.5f;       // the block's centre in the window
  const bool check = 8 * m1 >= a.reach;                       // the window passes the cutoff
  float4 (*acc)[32] = sh.acc[warp];
  float (*grp)[DN_P] = sh.group[warp];
  for (int s = 0; s < steps; ++s) acc[s][lane] = make_float4(0.f, 0.f, 0.f, 0.f);
  for (int q = lane; q < DN_GROUPS * DN_P; q += 32) grp[q / DN_P][q % DN_P] = 0.0f;
  __syncwarp();
  float hi[3] = {0.f, 0.f, 0.f}, lo[3] = {0.f, 0.f, 0.f};     // points lane, lane + 32, lane + 64 of the window
  // adds the lanes' sums of every point (32 different banks at a time) into the
  // compensated pairs and clears them
  auto fold = [&]() {
    __syncwarp();
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      const int k = lane + 32 * q, s = k >> 2;
      float v = 0.0f;
      if (k < n_pts) {
        const float* p = reinterpret_cast<const float*>(acc[s]) + (k & 3);
#pragma unroll 8
        for (int i = 0; i < 32; ++i) v += p[((i + s) & 31) * 4];
      }
      const float t = hi[q] + v, bp = t - hi[q];
      lo[q] += (hi[q] - (t - bp)) + (v - bp);
      hi[q] = t;
    }
    __syncwarp();
  };

  int chunks = 0;
  for (int base = l0; base < l1; base += 32) {
    const int i = min(base + lane, l1 - 1);
    const bool act = base + lane < l1;
    const LineWin w = a.win[i];
    const float inv = bartw::rcp_approx(w.nu0f * cc.dfac);    // 1 / (sigma sqrt 2)
    const float gam = a.gref[i] * cc.gfac;
    const float y = gam * inv, q = y * y;
    const float ln_s = line_ln_s(w, cc);
    const float S = (act && ln_s >= ln_thr) ? ex2f_approx((ln_s + LN_SCALE) * LOG2EF) : 0.0f;
    const float B = S * inv * bartw::INV_SQRTPI;              // V = B Re w
    const float A = B * y * bartw::INV_SQRTPI;                // far: V = A x (sqrt(pi) / y) Re w
    const float dx = a.dnu * inv, xc = w.delta * inv;
    const float off = (float)(w.jc - w0);                     // the line's nearest point in the window (exact)

    // ---- moments about the block's centre, in points
    {
      const float de = (off - centre) - w.delta * a.inv_dnu, ga = gam * a.inv_dnu;
      const float rdx = bartw::rcp_approx(dx), s2 = 0.5f * rdx * rdx;
      const float wt = S * a.w_scale;
      float M[DN_P];
      float r0 = 1.0f, i0 = 0.0f, r1 = de, i1 = ga;
#pragma unroll
      for (int n = 1; n <= DN_P; ++n) {
        M[n - 1] = wt * i1;
        const float ns = (float)n * s2;
        const float r2 = fmaf(de, r1, fmaf(-ga, i1, ns * r0)), i2 = fmaf(de, i1, fmaf(ga, r1, ns * i0));
        r0 = r1;
        i0 = i1;
        r1 = r2;
        i1 = i2;
      }
      // sums over the lanes of a group (segments of equal group index), added
      // by the group's last lane
      const int g = act ? a.gid[i] - g0 : -1;
      const int gn = __shfl_down_sync(0xffffffffu, g, 1);
      const bool tail = act && (lane == 31 || gn != g);
      const int gp = __shfl_up_sync(0xffffffffu, g, 1);
      const unsigned heads = __ballot_sync(0xffffffffu, lane == 0 || gp != g);
      const int first = 31 - __clz(heads & (0xffffffffu >> (31 - lane)));   // first lane of my segment
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const bool in = lane - o >= first;
        if (!__any_sync(0xffffffffu, in)) break;              // every segment is shorter
#pragma unroll
        for (int n = 0; n < DN_P; ++n) {
          const float t = __shfl_up_sync(0xffffffffu, M[n], o);
          if (in) M[n] += t;
        }
      }
      if (tail && g < DN_GROUPS) {
#pragma unroll
        for (int n = 0; n < DN_P; ++n) grp[g][n] += M[n];
      }
      __syncwarp();
    }

    // ---- near points.  The warp's lines lie in [cmin, cmax] (window
    // coordinates); a point's smallest |x| over them decides the form.
    const float pos = off - w.delta * a.inv_dnu;
    const float cmin = __uint_as_float(__reduce_min_sync(0xffffffffu, __float_as_uint(pos)));
    const float cmax = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(pos)));
    const float dxm = __uint_as_float(__reduce_min_sync(0xffffffffu, __float_as_uint(dx)));
    const float ymax = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(y)));
    const float ymin = __uint_as_float(__reduce_min_sync(0xffffffffu, __float_as_uint(y)));
    const bool small = ymax <= bartw::SMALL_Y;
    // |x| from which the shifted Lorentz form holds for every lane
    const float xl = sqrtf(sqrtf(fmaf(2.0f * ymax, ymax, 1.5f) * (1.0f / DN_EPS_L)) * 1.001f);
    const float x_core = ymin >= 9.0f ? -1.0f : 9.0f;         // |z| >= 9 everywhere: no core
    const float rdm = bartw::rcp_approx(dxm);
    const float p_far = xl * rdm, p_core = x_core * rdm;      // the same distances in points
    const float qL = q - 1.5f;
    const int jl = w.jlo - w0, jh = w.jhi - w0;
    for (int s = 0; s < steps; ++s) {
      const float p0 = (float)(4 * s);
      const float gap = fmaxf(cmin - (p0 + 3.0f), p0 - cmax);   // distance of the four points from the lines
      const float k0 = p0 - off;
      float v[4];
      if (gap >= p_far) {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const float x = fmaf(k0 + (float)k, dx, xc);
          v[k] = A * bartw::rcp_approx(fmaf(x, x, qL));
        }
      } else if (gap >= p_core) {
#pragma unroll
        for (int k = 0; k < 4; ++k) v[k] = A * gh4_ratio(fmaf(k0 + (float)k, dx, xc), q);
      } else {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const float p = p0 + (float)k;
          const float x = fabsf(fmaf(k0 + (float)k, dx, xc));
          if (fmaxf(cmin - p, p - cmax) >= p_core) v[k] = A * gh4_ratio(x, q);
          else if (small) v[k] = B * core_small(x, y);
          else v[k] = B * core_any(x, y, a.wtab);
        }
      }
      if (check) {
#pragma unroll
        for (int k = 0; k < 4; ++k)
          if (4 * s + k < jl || 4 * s + k > jh) v[k] = 0.0f;
      }
      float4 t = acc[s][lane];
      t.x += v[0];
      t.y += v[1];
      t.z += v[2];
      t.w += v[3];
      acc[s][lane] = t;
    }
    if (++chunks % DN_FOLD == 0 && base + 32 < l1) {
      fold();
      for (int s = 0; s < steps; ++s) acc[s][lane] = make_float4(0.f, 0.f, 0.f, 0.f);
      __syncwarp();
    }
  }
  if (l1 > l0) fold();
  const int64_t at = (int64_t)blockIdx.y * a.nb + b;
#pragma unroll
  for (int q = 0; q < 3; ++q)
    if (lane + 32 * q < n_pts) a.window[at * DN_WIN + lane + 32 * q] = hi[q] + lo[q];
  // the groups' moments, and the block's from them
  for (int e = lane; e < ng * DN_P; e += 32) a.mg[((int64_t)blockIdx.y * a.g_stride + g0) * DN_P + e] = grp[e / DN_P][e % DN_P];
  if (lane < DN_P) {
    float t = 0.0f;
    for (int g = 0; g < ng; ++g) t += grp[g][lane];
    a.m8[at * DN_P + lane] = t;
  }
  if (plan.kind != DN_COMPLEX) return;
  // ---- moments about the complex centres, a pass over the lines per bin
  const DenseBins bn = *a.bins;
  for (int bin = 0; bin < bn.n; ++bin) {
    float2 M[DN_PC];
#pragma unroll
    for (int n = 0; n < DN_PC; ++n) M[n] = make_float2(0.f, 0.f);
    const float gc = bn.c[bin] * cc.gfac;
    for (int base = l0; base < l1; base += 32) {
      const int i = min(base + lane, l1 - 1);
      const LineWin w = a.win[i];
      const float gr = a.gref[i];
      const int mine = min(max((int)floorf(log2f(gr * bn.inv_g0) * bn.inv_lr), 0), bn.n - 1);
      const float ln_s = line_ln_s(w, cc);
      const bool take = base + lane < l1 && mine == bin && ln_s >= ln_thr;
      const float wt = take ? ex2f_approx((ln_s + LN_SCALE) * LOG2EF) * a.w_scale : 0.0f;
      const float inv = bartw::rcp_approx(w.nu0f * cc.dfac), rdx = bartw::rcp_approx(a.dnu * inv), s2 = 0.5f * rdx * rdx;
      const float de = ((float)(w.jc - w0) - centre) - w.delta * a.inv_dnu, ga = (gr * cc.gfac - gc) * a.inv_dnu;
      // K_0 = 1, K_1 = u, K_(n+1) = u K_n + n sigma^2 K_(n-1), weighted
      float r0 = wt, i0 = 0.0f, r1 = de * wt, i1 = ga * wt;
#pragma unroll
      for (int n = 0; n < DN_PC; ++n) {
        M[n].x += r0;
        M[n].y += i0;
        const float ns = (float)(n + 1) * s2;
        const float r2 = fmaf(de, r1, fmaf(-ga, i1, ns * r0)), i2 = fmaf(de, i1, fmaf(ga, r1, ns * i0));
        r0 = r1;
        i0 = i1;
        r1 = r2;
        i1 = i2;
      }
    }
    float2 mine = make_float2(0.f, 0.f);
#pragma unroll
    for (int n = 0; n < DN_PC; ++n) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        M[n].x += __shfl_xor_sync(0xffffffffu, M[n].x, o);
        M[n].y += __shfl_xor_sync(0xffffffffu, M[n].y, o);
      }
      if (lane == n) mine = M[n];
    }
    if (lane < DN_PC) a.mc8[(at * DN_BINS + bin) * DN_PC + lane] = mine;
  }
}

// Moments of the blocks of 32 points from their four blocks of 8: with t the
// offset of a block's centre, I'_n = sum_k C(n, k) t^(n-k) I_k (k >= 1).
__global__ void __launch_bounds__(128)
dense_up_kernel(const __grid_constant__ DenseArgs a) {
  const int P = blockIdx.x * blockDim.x + threadIdx.x;
  const int kind = a.plan[a.c0 + blockIdx.y].kind;
  if (P >= a.nb / 4 || kind == DN_NONE) return;
  const float* m = a.m8 + ((int64_t)blockIdx.y * a.nb + 4 * P) * DN_P;
  float o[DN_P] = {};
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    const float t = (float)(8 * c - 12);
    float v[DN_P];
#pragma unroll
    for (int n = 0; n < DN_P; ++n) v[n] = m[c * DN_P + n];
    // the binomial sums as DN_P passes of I_n += t I_(n-1), pass r for n > r
    // (v[n] = I_(n+1); I_0 = 0)
#pragma unroll
    for (int r = 0; r < DN_P; ++r)
#pragma unroll
      for (int n = DN_P - 1; n >= (r > 0 ? r : 1); --n) v[n] = fmaf(t, v[n - 1], v[n]);
#pragma unroll
    for (int n = 0; n < DN_P; ++n) o[n] += v[n];
  }
  float* d = a.m32 + ((int64_t)blockIdx.y * (a.nb / 4) + P) * DN_P;
#pragma unroll
  for (int n = 0; n < DN_P; ++n) d[n] = o[n];
  if (kind != DN_COMPLEX) return;
  for (int bin = 0; bin < a.bins->n; ++bin) {
    float2 u[DN_PC] = {};
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const float t = (float)(8 * c - 12);
      const float2* src = a.mc8 + (((int64_t)blockIdx.y * a.nb + 4 * P + c) * DN_BINS + bin) * DN_PC;
      float2 v[DN_PC];
#pragma unroll
      for (int n = 0; n < DN_PC; ++n) v[n] = src[n];
#pragma unroll
      for (int r = 1; r < DN_PC; ++r)
#pragma unroll
        for (int n = DN_PC - 1; n >= r; --n) v[n] = make_float2(fmaf(t, v[n - 1].x, v[n].x), fmaf(t, v[n - 1].y, v[n].y));
#pragma unroll
      for (int n = 0; n < DN_PC; ++n) u[n] = make_float2(u[n].x + v[n].x, u[n].y + v[n].y);
    }
    float2* dst = a.mc32 + (((int64_t)blockIdx.y * (a.nb / 4) + P) * DN_BINS + bin) * DN_PC;
#pragma unroll
    for (int n = 0; n < DN_PC; ++n) dst[n] = u[n];
  }
}

// sum_n I_n / D^(n+1)
__device__ __forceinline__ float moment_sum(const float* __restrict__ m, float D) {
  const float4 a = *reinterpret_cast<const float4*>(m), b = *reinterpret_cast<const float4*>(m + 4);
  const float r = bartw::rcp_approx(D);
  float v = b.w;
  v = fmaf(v, r, b.z);
  v = fmaf(v, r, b.y);
  v = fmaf(v, r, b.x);
  v = fmaf(v, r, a.w);
  v = fmaf(v, r, a.z);
  v = fmaf(v, r, a.y);
  v = fmaf(v, r, a.x);
  return v * (r * r);
}

// Im sum_n M_n / Z^(n+1), Z = D - i g
__device__ __forceinline__ float complex_sum(const float2* __restrict__ m, float D, float g) {
  const float q = bartw::rcp_approx(fmaf(D, D, g * g)), rr = D * q, ri = g * q;   // 1 / Z
  const float4* p = reinterpret_cast<const float4*>(m);
  float vr = 0.0f, vi = 0.0f;
#pragma unroll
  for (int n = DN_PC / 2 - 1; n >= 0; --n) {
    const float4 c = p[n];                       // M_2n, M_(2n+1)
    float t = fmaf(vr, rr, fmaf(-vi, ri, c.z));
    vi = fmaf(vr, ri, fmaf(vi, rr, c.w));
    vr = t;
    t = fmaf(vr, rr, fmaf(-vi, ri, c.x));
    vi = fmaf(vr, ri, fmaf(vi, rr, c.y));
    vr = t;
  }
  return fmaf(vr, ri, vi * rr);
}

// One point per thread: the warp's 32 points are one block of 32, so its lanes
// agree on the far blocks and almost on the mid ones (uniform loops, one
// broadcast read per block).
__global__ void __launch_bounds__(256)
dense_sum_kernel(const __grid_constant__ DenseArgs a) {
  const int cell = a.c0 + blockIdx.y;
  const DensePlan plan = a.plan[cell];
  if (plan.kind == DN_NONE) return;
  const int j0 = (blockIdx.x * blockDim.x + threadIdx.x) & ~31;
  if (j0 >= a.n_nu) return;
  const int lane = threadIdx.x & 31, j = min(j0 + lane, a.n_nu - 1);
  const DensePoint p = a.pts[j];
  const int t = (j >> 3) + a.boff, T = t >> 2;
  const float* m8 = a.m8 + (int64_t)blockIdx.y * a.nb * DN_P;
  const float* m32 = a.m32 + (int64_t)blockIdx.y * (a.nb / 4) * DN_P;
  const float* mg = a.mg + (int64_t)blockIdx.y * a.g_stride * DN_P;
  const float* win = a.window + (int64_t)blockIdx.y * a.nb * DN_WIN;
  const float jf = (float)(j - j0);                          // positions relative to j0: exact
  // centre of block b and of parent P, relative to j0
  auto centre8 = [&](int b) { return (float)((b - a.boff) * DN_B - j0) + 3.5f; };
  auto centre32 = [&](int P) { return (float)((4 * P - a.boff) * DN_B - j0) + 15.5f; };

  // ---- near: the windows of the blocks around the point
  float near = 0.0f;
  for (int b = t - plan.m1 + 1; b < t + plan.m1; ++b)
    near += win[(int64_t)b * DN_WIN + (t - b + plan.m1 - 1) * DN_B + (j & 7)];

  // ---- blocks inside the point's cutoff [bl, br), outside the near ones
  const int PL = (p.bl + 3) >> 2, PR = p.br >> 2;            // parents inside it
  float far = 0.0f, mid = 0.0f;
  if (plan.kind == DN_COMPLEX) {
    const DenseBins bn = *a.bins;
    const float scale = a.cells[cell].gfac * a.inv_dnu;
    const float2* mc8 = a.mc8 + (int64_t)blockIdx.y * a.nb * DN_BINS * DN_PC;
    const float2* mc32 = a.mc32 + (int64_t)blockIdx.y * (a.nb / 4) * DN_BINS * DN_PC;
    // parents inside the cutoff: real centre far away, complex centres nearer
    const int u0 = __reduce_min_sync(0xffffffffu, PL), u1 = __reduce_max_sync(0xffffffffu, PR);
    for (int P = u0; P < u1; ++P) {
      const int m = abs(P - T);                  // the same for the warp
      const bool in = P >= PL && P < PR;
      const float D = jf - centre32(P);
      if (m >= plan.m2) {
        if (in) far += moment_sum(m32 + (int64_t)P * DN_P, D);
      } else if (m >= plan.mh) {
        for (int q = 0; q < bn.n; ++q)
          if (in) far += complex_sum(mc32 + ((int64_t)P * DN_BINS + q) * DN_PC, D, bn.c[q] * scale);
      }
    }
    // blocks of the parents closer than that, and those beside the parents
    auto blocks8 = [&](int b0, int b1) {
      const int v0 = __reduce_min_sync(0xffffffffu, b0 < b1 ? b0 : 0x7fffffff);
      const int v1 = __reduce_max_sync(0xffffffffu, b0 < b1 ? b1 : -0x7fffffff);
      for (int b = v0; b < v1; ++b) {
        const bool in = b >= b0 && b < b1 && abs(b - t) >= plan.m1;
        const float D = jf - centre8(b);
        for (int q = 0; q < bn.n; ++q)
          if (in) mid += complex_sum(mc8 + ((int64_t)b * DN_BINS + q) * DN_PC, D, bn.c[q] * scale);
      }
    };
    const int c0 = max(4 * (T - plan.mh + 1), 4 * PL), c1 = min(4 * (T + plan.mh), 4 * PR);
    if (PL < PR) {
      blocks8(p.bl, 4 * PL);
      blocks8(c0, c1);
      blocks8(4 * PR, p.br);
    } else {
      blocks8(p.bl, p.br);
    }
  } else {
  // left of the point: parents [PL, PE), blocks before and after them
  const int PE = min(T - plan.m2 + 1, PR), lend = min(t - plan.m1 + 1, p.br);
  const int PS = max(T + plan.m2, PL), rbeg = max(t + plan.m1, p.bl);
  {
    const int u0 = __reduce_min_sync(0xffffffffu, PL), u1 = __reduce_max_sync(0xffffffffu, PE);
    for (int P = u0; P < u1; ++P)
      if (P >= PL && P < PE) far += moment_sum(m32 + (int64_t)P * DN_P, jf - centre32(P));
    const int v0 = __reduce_min_sync(0xffffffffu, PS), v1 = __reduce_max_sync(0xffffffffu, PR);
    for (int P = v0; P < v1; ++P)
      if (P >= PS && P < PR) far += moment_sum(m32 + (int64_t)P * DN_P, jf - centre32(P));
  }
  auto blocks = [&](int b0, int b1) {                        // [b0, b1), possibly empty
    const int u0 = __reduce_min_sync(0xffffffffu, b0 < b1 ? b0 : 0x7fffffff);
    const int u1 = __reduce_max_sync(0xffffffffu, b0 < b1 ? b1 : -0x7fffffff);
    for (int b = u0; b < u1; ++b)
      if (b >= b0 && b < b1) mid += moment_sum(m8 + (int64_t)b * DN_P, jf - centre8(b));
  };
  const bool hasL = PE > PL, hasR = PR > PS;
  blocks(p.bl, hasL ? min(4 * PL, lend) : lend);
  blocks(hasL ? 4 * PE : lend, lend);
  blocks(rbeg, hasR ? 4 * PS : p.br);
  blocks(hasR ? max(4 * PR, rbeg) : p.br, p.br);
  }

  // ---- edges: the block that a cutoff edge divides, group by group (blocks
  // within the near radius were taken line by line)
  float edge = 0.0f;
  auto groups = [&](int g0, int g1, int b) {
    if (abs(b - t) < plan.m1) return;
    const float D = jf - centre8(b);
    for (int g = max(g0, 0); g < min(g1, (int)a.g_stride); ++g) edge += moment_sum(mg + (int64_t)g * DN_P, D);
  };
  if (p.bl > p.br) {                                         // both edges divide the same block
    groups(p.gl, p.gr, p.br);
  } else {
    if (p.bl > 0) groups(p.gl, min(a.gfirst[p.bl], p.gr), p.bl - 1);
    if (p.br < a.nb) groups(max(a.gfirst[p.br], p.gl), p.gr, p.br);
  }
  if (j0 + lane < a.n_nu) a.out[(int64_t)cell * a.n_nu + j] = ((edge + far) + (mid + near)) * INV_SCALE;
}

}  // namespace

bool bartop::dense_applies(const bart_linelist& lines, const bart_nugrid& nu, double cutoff, CellConst* cells,
                           int n_cells) {
  const double reach = cutoff / nu.dnu_cm;
  if (lines.n_lines < 64 || lines.n_lines > (int64_t)1 << 30 || (double)lines.n_lines < DN_DENSITY * (double)nu.n_nu)
    return false;
  // The near window (4 blocks of 8 points and more) is checked line by line
  // against the cutoff where it passes it; below three blocks there is little else.
  if (!(reach >= 3.0 * DN_B) || reach > 1e6 || nu.n_nu > (1 << 30)) return false;
  const double lo = nu.nu_start_cm - cutoff, hi = nu.nu_start_cm + (double)nu.n_nu * nu.dnu_cm + cutoff;
  if (!(lo > 0.0)) return false;
  bool any = false;
  for (int c = 0; c < n_cells; ++c) {
    // x of one grid interval: |x| >= 9 at the 8 m1 - 3.5 - 4 >= 24.5 points that
    // a mid block's lines are away at least keeps the moments' asymptotic series
    // below 1e-6; the near window's products of four squared x (within 12
    // points of a line's) stay in the FP32 range
    const double dx_min = nu.dnu_cm / (hi * cells[c].dfac), dx_max = nu.dnu_cm / (lo * cells[c].dfac);
    cells[c].dense = dx_min >= 0.4 && dx_max <= 3000.0;
    any = any || cells[c].dense;
  }
  return any;
}

bart_status bartop::dense_cells(bart_ctx* ctx, const LineWin* win, const int* jlo, const int* jhi, const float* gref,
                                int64_t n_lines, const CellConst* cells, int n_cells, const bart_nugrid& nu,
                                double cutoff, const int* smax, const int* tmap, float ln_rel, float* out,
                                const DensePlan** plan) {
  const int n_nu = (int)nu.n_nu, n = (int)n_lines;
  const int reach = (int)std::floor(cutoff / nu.dnu_cm);
  const int boff = ((reach + 2) / DN_B + DN_M1_MAX + 4) / 4 * 4;         // blocks before the grid, whole parents
  const int nb = (boff + n_nu / DN_B + (reach + 2) / DN_B + DN_M1_MAX + 8) / 4 * 4;
  const int tiles = (n + GR_TILE - 1) / GR_TILE;
  const int64_t g_max = std::min<int64_t>(n, (int64_t)nb * DN_GROUPS) + 1;
  const size_t per_cell = ((size_t)nb * (DN_WIN + DN_P) + (size_t)(nb / 4) * DN_P + (size_t)g_max * DN_P +
                           (size_t)(nb + nb / 4) * DN_BINS * DN_PC * 2) * 4;
  const int batch = (int)std::max<size_t>(1, std::min<size_t>(n_cells, DN_SCRATCH / per_cell));
  DenseBins* bins;
  int *range, *lstart, *gfirst, *gid, *count, *stat;
  DensePlan* pl;
  DensePoint* pts;
  float* scratch;
  *plan = nullptr;
  const struct {
    const char* name;
    size_t bytes;
    void** p;
  } need[] = {{"dn_range", 8 * sizeof(int), (void**)&range},
              {"dn_bins", sizeof(DenseBins), (void**)&bins},
              {"dn_lstart", (size_t)(nb + 1) * sizeof(int), (void**)&lstart},
              {"dn_gfirst", (size_t)(nb + 1) * sizeof(int), (void**)&gfirst},
              {"dn_gid", (size_t)n * sizeof(int), (void**)&gid},
              {"dn_count", (size_t)(tiles + 1) * sizeof(int), (void**)&count},
              {"dn_plan", (size_t)n_cells * sizeof(DensePlan), (void**)&pl},
              {"dn_pts", (size_t)n_nu * sizeof(DensePoint), (void**)&pts},
              {"dn_moments", per_cell * batch, (void**)&scratch}};
  for (const auto& q : need)
    if (bart_scratch(ctx, q.name, q.bytes, q.p) != BART_OK) {
      ctx->err.clear();       // no room (or a capture that cannot grow it): every cell goes line by line
      return BART_OK;
    }
  stat = range + 4;
  bart_status st;
  cudaStream_t s = ctx->stream;
  BART_CUDA(ctx, cudaMemsetAsync(stat, 0, 3 * sizeof(int), s));
  const int* total = count + tiles;
  dense_range_kernel<<<1, 1, 0, s>>>(jlo, jhi, n, n_nu, range);
  dense_block_kernel<<<nb / 256 + 1, 256, 0, s>>>(win, range, boff, nb, lstart);
  dense_group_count_kernel<<<tiles, GR_TILE, 0, s>>>(win, range, count);
  dense_group_scan_kernel<<<1, GR_TILE, 0, s>>>(count, tiles);
  dense_group_kernel<<<tiles, GR_TILE, 0, s>>>(win, range, count, n, gid);
  dense_first_group_kernel<<<nb / 256 + 1, 256, 0, s>>>(lstart, range, gid, total, nb, gfirst);
  dense_point_kernel<<<(n_nu + 255) / 256, 256, 0, s>>>(win, jlo, jhi, range, gid, total, lstart, boff, nb, n_nu, pts);
  dense_gamma_kernel<<<std::min(tiles, 4 * ctx->sm_count), 256, 0, s>>>(gref, n, stat);
  dense_plan_kernel<<<(n_cells + 127) / 128, 128, 0, s>>>(cells, n_cells, stat, (float)(1.0 / nu.dnu_cm), reach, pl, bins);
  if ((st = bart_check_launch(ctx, "dense opacity prologue")) != BART_OK) return st;
  DenseArgs a{};
  a.win = win;
  a.gref = gref;
  a.lstart = lstart;
  a.gid = gid;
  a.gfirst = gfirst;
  a.cells = cells;
  a.plan = pl;
  a.pts = pts;
  a.bins = bins;
  a.smax = smax;
  a.tmap = tmap;
  a.wtab = ctx->d_wtable;
  a.ln_rel = ln_rel;
  a.dnu = (float)nu.dnu_cm;
  a.inv_dnu = (float)(1.0 / nu.dnu_cm);
  a.w_scale = (float)(1.0 / (bartc::PI * nu.dnu_cm));
  a.boff = boff;
  a.nb = nb;
  a.n_nu = n_nu;
  a.reach = reach;
  a.g_stride = g_max;
  a.window = scratch;
  a.m8 = a.window + (size_t)batch * nb * DN_WIN;
  a.m32 = a.m8 + (size_t)batch * nb * DN_P;
  a.mc8 = reinterpret_cast<float2*>(a.m32 + (size_t)batch * (nb / 4) * DN_P);
  a.mc32 = a.mc8 + (size_t)batch * nb * DN_BINS * DN_PC;
  a.mg = reinterpret_cast<float*>(a.mc32 + (size_t)batch * (nb / 4) * DN_BINS * DN_PC);
  a.out = out;
  BART_CUDA(ctx, cudaFuncSetAttribute(dense_near_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)sizeof(NearShared)));
  for (a.c0 = 0; a.c0 < n_cells; a.c0 += batch) {
    const unsigned nc = (unsigned)std::min(batch, n_cells - a.c0);
    dense_near_kernel<<<dim3((unsigned)((nb + DN_WARPS - 1) / DN_WARPS), nc), 32 * DN_WARPS, sizeof(NearShared), s>>>(a);
    dense_up_kernel<<<dim3((unsigned)((nb / 4 + 127) / 128), nc), 128, 0, s>>>(a);
    dense_sum_kernel<<<dim3((unsigned)((n_nu + 255) / 256), nc), 256, 0, s>>>(a);
    if ((st = bart_check_launch(ctx, "dense opacity kernels")) != BART_OK) return st;
  }
  *plan = pl;
  return BART_OK;
}
