// Opacity of dense line lists: the same sum over lines as opacity_kernel,
// arranged by distance so that the cost of a line far from a point is shared
// with its neighbours.
//
// The 5e6-line grid holds 17 lines per wavenumber point and each line reaches
// 2,500 points, so most of the work of a line-by-line sum is far wings of lines
// that lie within a fraction of a point of one another.  Lines are taken in
// source blocks of 8 grid points (by their nearest point jc).  For a point j
//   near   source blocks closer than m1 (5) blocks: every line evaluated on its own
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
// DN_P.  m1 and m2 keep sqrt(r^2 + gamma^2) <= DN_RHO x the distance, r^8 =
// E[(half + g)^8] (reach8): the first term left out is then below 9 DN_RHO^8 =
// 1.3e-6 of a line's own at the nearest point for the line farthest from the
// centre, far below that in a sum.
//
// Lengths are in units of a power of two near the widest profile, so that no
// power of a width leaves the FP32 range.
//
// Lorentz widths beyond about 3 points need moments about a complex centre:
// with the lines of a block in bins of gamma_ref (ratio <= sqrt 2 within a bin),
// u = delta + g + i (gamma - gamma_c) about the bin's middle gamma_c and
// Z = d - i gamma_c, V = (S / pi) Im sum_n E[u^n] / Z^(n+1): |Z| >= gamma_c, so a
// wide profile is smooth on the scale of a block and needs no near lines at
// all.  DN_PC terms hold where E[|u|^14] <= (DN_RHOC |Z|)^14 (reach14; 15
// DN_RHOC^14 = 9e-7; against the Faddeeva function in 64 bits, for x of a grid
// interval from 0.4 on: 1.2e-6 of a line on its block's edge).
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
// pair every 8 chunks; the moments of a block's lines and a point's sums over
// blocks are folded the same way (FoldedSum), so that rounding does not grow with
// the number of lines or blocks.  dense_sum_kernel adds the near windows of the
// 2 m1 - 1 blocks around a point, then the moments.  No atomics: every sum has a
// fixed order.
//
// Used (dense_applies, dense_plan_kernel) for lists of at least DN_DENSITY lines
// per point, where blocks pay for their fixed cost, and for cells whose widths
// fit: Doppler deviations up to 1.8 grid points (x of an interval 0.4); Lorentz
// widths up to about 3 grid points, or gamma_ref within a factor 4 over the
// list (4 bins), or a cutoff so short that the near window holds all of it.
// Other cells go line by line.  From a sixth of the cutoff on a divided block's
// moments about the real centre do not converge, and its lines count one by one
// (130 of them per point; line by line the cell has 42,000).
// Measured: one species of the 5e6-line grid (1.67e6 lines, 100,000 points), 10
// layers over 1e-8 .. 100 bar x 20 temperatures: 169 ms line by line, 58 ms with
// the 160 cells of widths up to 3 points here, 44 ms with widths up to a sixth of
// the cutoff, 40 ms with the near points in packed pairs, 28.3 ms with all cells,
// 28.8 ms with the moments' sums compensated (100 to 170 us of the near kernel
// and 15 of the sums per cell; the near kernel's per-lane sums in shared memory
// and its profiles bound it: L1 data pipe 87%, issue 53% of the slots at 0.1 bar); 2 species x 10,000 lines, 60 cells, 2,000 points 1 cm^-1 apart:
// 2.59 ms and 0.32 ms.
#include <algorithm>
#include <cmath>

#include "opacity.cuh"

using namespace bartop;

namespace {

constexpr int DN_B = 8;                     // points of a source block
constexpr int DN_P = 8;                     // moments
constexpr int DN_M1 = 5;                    // near radius in blocks about real centres (a mid block's centre is 36.5
                                            // points away; 4 blocks, 28.5 points, would not do for a half width of 4),
                                            // and the largest about complex ones
constexpr int DN_WIN = (2 * DN_M1 - 1) * DN_B;   // near points of a block, at most
constexpr int DN_GROUPS = 20;               // groups of a block: jlo and jhi each step at most 9 times
constexpr float DN_RHO = 0.14f;
constexpr int DN_BINS = 4;                  // bins of gamma_ref
constexpr int DN_PC = 14;                   // moments about a complex centre
constexpr float DN_RHOC = 0.305f;
constexpr float DN_RHO_EDGE = 0.175f;       // divided blocks: 9e-7 of a line at its cutoff (against the Faddeeva
                                            // function in 64 bits; 9 x 0.175^8 = 8e-6 would be a half width's share)
constexpr double DN_DENSITY = 0.5;          // lines per point
constexpr int DN_WARPS = 4;
constexpr int DN_FOLD = 8;                  // chunks of 32 lines between two folds
constexpr float DN_EPS_L = 2e-6f;           // bound of the shifted Lorentz form
constexpr size_t DN_SCRATCH = (size_t)256 << 20;     // moments and windows of a batch of cells (a third of it is
                                                     // touched for a cell: within L2)

struct DensePoint {           // per grid point (indexes of groups and blocks)
  int gl, gr;                 // groups whose window holds the point: [gl, gr)
  int bl, br;                 // blocks all of whose lines do: [bl, br)
  int il, ir;                 // lines: [il, ir)
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
  p.il = il;
  p.ir = ir;
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

// (E[(h + g)^8])^(1/8) and (E[(h + g)^14])^(1/14) of a Gaussian g of deviation s:
// how far a line h from its block's centre reaches into the moments.
__device__ __forceinline__ float reach8(float h, float s) {
  const float r = s / h, q = r * r;
  return h * powf(fmaf(q, fmaf(q, fmaf(q, fmaf(q, 105.0f, 420.0f), 210.0f), 28.0f), 1.0f), 0.125f);
}
__device__ __forceinline__ float reach14(float h, float s) {
  const float r = s / h, q = r * r;
  float v = fmaf(q, 135135.0f, 945945.0f);
  v = fmaf(q, v, 945945.0f);
  v = fmaf(q, v, 315315.0f);
  v = fmaf(q, v, 45045.0f);
  v = fmaf(q, v, 3003.0f);
  v = fmaf(q, v, 91.0f);
  return h * powf(fmaf(q, v, 1.0f), 1.0f / 14.0f);
}

// sigma: the widest Doppler deviation of a cell in points, over dfac.
__global__ void dense_plan_kernel(const CellConst* __restrict__ cells, int n_cells, const int* __restrict__ stat,
                                  float inv_dnu, float sigma, int reach, DensePlan* __restrict__ plan,
                                  DenseBins* __restrict__ bins) {
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  const DenseBins bn = dense_bins(stat);
  if (c == 0) *bins = bn;
  if (c >= n_cells) return;
  DensePlan p{DN_NONE, 0, 0, 0, 1.0f, 0};
  const float scale = cells[c].gfac * inv_dnu, g = __int_as_float(stat[0]) * scale;   // widest line, in points
  if (cells[c].dense && !stat[1] && g < 1e6f) {
    // a point of block t is at least 8 m - 3.5 points from the centre of block t +- m
    const float sd = sigma * cells[c].dfac;
    const float r8 = reach8(4.0f, sd), r32 = reach8(16.0f, sd), c8 = reach14(4.0f, sd), c32 = reach14(16.0f, sd);
    const int m2 = max(4, (int)ceilf((sqrtf(r32 * r32 + g * g) / DN_RHO + 15.5f) / 32.0f));
    if (sqrtf(r8 * r8 + g * g) <= DN_RHO * (8.0f * DN_M1 - 3.5f) ||
        8 * (DN_M1 - 1) > reach) {               // (or the near window holds every line's points)
      p = {DN_REAL, DN_M1, 0, m2, 1.0f, 0};
    } else if (bn.n > 0) {
      float d8 = 0.0f, d32 = 0.0f;               // squared distances from which the complex moments hold
      for (int q = 0; q < bn.n; ++q) {
        const float gc = bn.c[q] * scale, e2 = bn.eta * bn.eta * gc * gc;
        d8 = fmaxf(d8, (c8 * c8 + e2) / (DN_RHOC * DN_RHOC) - gc * gc);
        d32 = fmaxf(d32, (c32 * c32 + e2) / (DN_RHOC * DN_RHOC) - gc * gc);
      }
      p.kind = DN_COMPLEX;
      p.m1 = d8 > 0.0f ? (int)ceilf((sqrtf(d8) + 3.5f) / 8.0f) : 0;
      p.mh = d32 > 0.0f ? (int)ceilf((sqrtf(d32) + 15.5f) / 32.0f) : 0;
      p.m2 = max(m2, p.mh);
      // the moments of the divided blocks' groups are about the real centre
      p.lines = sqrtf(r8 * r8 + g * g) > DN_RHO_EDGE * (float)(reach - 8);
      if (p.m1 > DN_M1) p.kind = DN_NONE;
    }
    // lengths up to sqrt(16^2 + g^2): their 14th powers times a strength stay in range
    p.ih = exp2f(-ceilf(0.5f * log2f(c32 * c32 + g * g)));
  }
  plan[c] = p;
}

// Pairs of points in packed FP32 (one issue slot for both; the near kernel is
// bound by its instructions and its sums in shared memory).
__device__ __forceinline__ float2 f2(float v) { return make_float2(v, v); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 rcp2(float2 d) { return make_float2(bartw::rcp_approx(d.x), bartw::rcp_approx(d.y)); }

// G(x) = -Im w'(x) = (2 / sqrt(pi)) (2 x F(x) - 1), F Dawson's integral, u = x^2:
// up to x = 9.3 a rational function of u fitted (least squares, reweighted
// towards the largest error) to |dG| <= 1e-6 (50 e^(-x^2) + |G|) in FP32 -- near
// its zero at 0.92 the Gaussian term of the profile is far larger -- and its
// asymptotic series beyond.
__device__ __forceinline__ float2 dawson_g(float2 u) {
  float2 n = f2(4.43394788e-06f), d = f2(7.85838861e-06f);
  n = fma2(n, u, f2(-3.46022744e-05f));
  n = fma2(n, u, f2(4.63677612e-04f));
  n = fma2(n, u, f2(-2.12909611e-04f));
  n = fma2(n, u, f2(2.23139278e-02f));
  n = fma2(n, u, f2(-9.76259707e-02f));
  n = fma2(n, u, f2(1.38819137f));
  n = fma2(n, u, f2(-1.12835006f));
  d = fma2(d, u, f2(-7.29758443e-05f));
  d = fma2(d, u, f2(8.88062378e-04f));
  d = fma2(d, u, f2(-8.60452054e-04f));
  d = fma2(d, u, f2(1.95862562e-02f));
  d = fma2(d, u, f2(6.41052559e-02f));
  d = fma2(d, u, f2(2.97722797e-01f));
  d = fma2(d, u, f2(7.68709942e-01f));
  d = fma2(d, u, f2(1.0f));
  const bool fx = u.x > 9.3f * 9.3f, fy = u.y > 9.3f * 9.3f;
  const float2 t = rcp2(make_float2(fx ? u.x : d.x, fy ? u.y : d.y));
  constexpr float C = 1.1283791670955126f;
  float2 s = fma2(t, f2(29.53125f * C), f2(6.5625f * C));    // (2 / sqrt(pi)) (2k-1)!! / 2^k, k = 5 .. 1
  s = fma2(s, t, f2(1.875f * C));
  s = fma2(s, t, f2(0.75f * C));
  s = fma2(s, t, f2(0.5f * C));
  return mul2(t, make_float2(fx ? s.x : n.x, fy ? s.y : n.y));
}

// Re w(x + i y) for 0 <= y <= SMALL_Y: the expansion in y of small_y_re
// (faddeeva.cuh) without a branch or a table.
__device__ __forceinline__ float2 core_small(float2 x, float y) {
  constexpr float L2E_LO = (float)(1.4426950408889634 - (double)LOG2EF);
  const float2 u = mul2(x, x), lo = fma2(x, x, make_float2(-u.x, -u.y));     // x^2 = u + lo
  const float2 ah = mul2(u, f2(-LOG2EF));
  const float2 al = add2(fma2(u, f2(LOG2EF), ah), fma2(lo, f2(LOG2EF), mul2(u, f2(L2E_LO))));
  const float2 e = mul2(make_float2(ex2f_approx(ah.x), ex2f_approx(ah.y)), fma2(al, f2(-LN2F_), f2(1.0f)));
  const float2 g = dawson_g(u);
  const float y2 = y * y, y26 = y2 * (1.0f / 6.0f);
  const float2 q = make_float2(u.x < 1600.0f ? y26 : 0.0f, u.y < 1600.0f ? y26 : 0.0f);
  const float2 gy = fma2(q, fma2(g, fma2(u, f2(-4.0f), f2(6.0f)), f2(2.2567583341910252f)), g);
  return fma2(e, fma2(f2(y2), fma2(u, f2(-2.0f), f2(1.0f)), f2(1.0f)), mul2(f2(y), gy));
}

// (sqrt(pi) / y) Re w by Gauss-Hermite quadrature of w = (i / pi) int e^(-t^2) /
// (z - t) dt: Re w = (y / pi) sum_k w_k / ((x - t_k)^2 + y^2), the two nodes +-t
// as 2 w s / (s^2 - 4 x^2 t^2) with s = x^2 + y^2 + t^2.  Weights divided by
// sqrt(pi) here.  4 nodes: <= 4e-7 from |x| = gh4_from(y) on.
__device__ __forceinline__ float2 gh4_ratio(float2 x, float y2) {
  constexpr float T1 = 0.27525512860841095f, T2 = 2.7247448713915889f;      // t^2
  constexpr float W1 = 0.90824829046386302f, W2 = 0.091751709536136983f;    // 2 w / sqrt(pi)
  const float2 u = mul2(x, x), s1 = add2(u, f2(y2 + T1)), s2 = add2(u, f2(y2 + T2));
  const float2 d1 = fma2(s1, s1, mul2(u, f2(-4.0f * T1))), d2 = fma2(s2, s2, mul2(u, f2(-4.0f * T2)));
  const float2 n = fma2(mul2(s2, f2(W2)), d1, mul2(mul2(s1, f2(W1)), d2));
  return mul2(n, rcp2(mul2(d1, d2)));
}
// |x| from which it holds for widths of at least y; negative: everywhere.
__device__ __forceinline__ float gh4_from(float y) { return y >= 7.0f ? -1.0f : y >= 4.0f ? 5.0f : y >= 2.0f ? 7.1f : 9.0f; }
// 8 nodes: <= 3e-7 for |z| >= 5 and for y >= 3, plus the residue e^(y^2 - x^2)
// cos 2xy that the quadrature misses near the real axis.
constexpr float GH8_Y = 3.0f;
constexpr float LORENTZ_Y = 1000.0f;        // from here on the shifted Lorentz form holds at any x (2 / y^2), and
                                            // not much farther the products of the others leave the FP32 range
template <bool RESIDUE>
__device__ __forceinline__ float2 gh8_re(float2 x, float y) {
  constexpr float T[4] = {0.14530352150331707f, 1.3390972881263614f, 3.9269635013582872f, 8.5886356890120343f};
  constexpr float Wt[4] = {0.746024515358155f, 0.234479815323518f, 0.0192704402415765f, 0.00022522907675073f};
  const float y2 = y * y;
  const float2 u = mul2(x, x);
  float2 r = f2(0.0f);
#pragma unroll
  for (int k = 0; k < 4; k += 2) {
    const float2 s1 = add2(u, f2(y2 + T[k])), s2 = add2(u, f2(y2 + T[k + 1]));
    const float2 d1 = fma2(s1, s1, mul2(u, f2(-4.0f * T[k]))), d2 = fma2(s2, s2, mul2(u, f2(-4.0f * T[k + 1])));
    r = fma2(fma2(mul2(s2, f2(Wt[k + 1])), d1, mul2(mul2(s1, f2(Wt[k])), d2)), rcp2(mul2(d1, d2)), r);
  }
  r = mul2(r, f2(bartw::INV_SQRTPI * y));
  if (RESIDUE) {
    const float gx = fmaf(y, y, -u.x), gy = fmaf(y, y, -u.y);
    if (y < 1.0f && gx > -87.0f) r.x += __expf(gx) * __cosf(2.0f * x.x * y);
    if (y < 1.0f && gy > -87.0f) r.y += __expf(gy) * __cosf(2.0f * x.y * y);
  }
  return r;
}
// (sqrt(pi) / y) Re w for |z| >= 9: three terms of the asymptotic series from
// |z| = 100 on (4e-8), else four nodes.
__device__ __forceinline__ float far_ratio(float x, float y2) {
  const float u = x * x, s = u + y2, r = bartw::rcp_approx(s);
  if (s >= 1e4f) return r * fmaf(r * r, fmaf(1.5f, u, -0.5f * y2), 1.0f);
  return gh4_ratio(f2(x), y2).x;
}
__device__ __forceinline__ float2 core_any(float2 x, float y, const float2* __restrict__ wtab) {
  const bool tx = fmaf(x.x, x.x, y * y) < 25.0f, ty = fmaf(x.y, x.y, y * y) < 25.0f;
  float2 r = f2(0.0f);
  if (!tx || !ty) r = gh8_re<true>(x, y);
  if (tx) r.x = bartw::taylor_re<>(fabsf(x.x), y, wtab);
  if (ty) r.y = bartw::taylor_re<>(fabsf(x.y), y, wtab);
  return r;
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

// hi + lo += v, exactly but for the rounding of lo (TwoSum).
__device__ __forceinline__ void two_sum(float& hi, float& lo, float v) {
  const float t = hi + v, bp = t - hi;
  lo += (hi - (t - bp)) + (v - bp);
  hi = t;
}
// A running sum of few terms, folded into a compensated pair now and then.
struct FoldedSum {
  float s = 0.0f, hi = 0.0f, lo = 0.0f;
  __device__ __forceinline__ void fold() {
    two_sum(hi, lo, s);
    s = 0.0f;
  }
  __device__ __forceinline__ float total() {
    fold();
    return hi + lo;
  }
};
// term(i) for i in [from, to), folding the sum every 16 of them.
template <typename F>
__device__ __forceinline__ void folded_range(int from, int to, FoldedSum& sum, F term) {
  for (int i = from; i < to;) {
    const int stop = min(i + 16, to);
    for (; i < stop; ++i) term(i);
    if (i < to) sum.fold();
  }
}

struct NearShared {
  float4 acc[DN_WARPS][DN_WIN / 4][32];      // per lane, four neighbouring points
  float group[DN_WARPS][DN_GROUPS * DN_P];
  float2 folded[DN_WARPS][DN_GROUPS * DN_P]; // the groups' sums before the last fold, compensated pairs
  int list[DN_WARPS][64];                    // lines of a bin, being gathered
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
  float* grp = sh.group[warp];
  float2* grp_folded = sh.folded[warp];
  for (int s = 0; s < steps; ++s) acc[s][lane] = make_float4(0.f, 0.f, 0.f, 0.f);
  for (int q = lane; q < DN_GROUPS * DN_P; q += 32) {
    grp[q] = 0.0f;
    grp_folded[q] = make_float2(0.f, 0.f);
  }
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
      two_sum(hi[q], lo[q], v);
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

    // ---- moments about the block's centre, in points (times ih)
    {
      const float de = ((off - centre) - w.delta * a.inv_dnu) * plan.ih, ga = gam * (a.inv_dnu * plan.ih);
      const float rdx = bartw::rcp_approx(dx) * plan.ih, s2 = 0.5f * rdx * rdx;
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
        for (int n = 0; n < DN_P; ++n) grp[g * DN_P + n] += M[n];
      }
      __syncwarp();
    }

    // ---- near points.  The warp's lines lie in [cmin, cmax] (window
    // coordinates); a point's smallest |x| over them decides the form.
    const float pos = off - w.delta * a.inv_dnu;
    // (a window of one block has lines up to half a point left of its first point)
    const float cmin = ordered_float(__reduce_min_sync(0xffffffffu, ordered_int(pos)));
    const float cmax = ordered_float(__reduce_max_sync(0xffffffffu, ordered_int(pos)));
    const float dxm = __uint_as_float(__reduce_min_sync(0xffffffffu, __float_as_uint(dx)));
    const float ymax = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(y)));
    const float ymin = __uint_as_float(__reduce_min_sync(0xffffffffu, __float_as_uint(y)));
    const bool small = ymax <= bartw::SMALL_Y;
    // |x| from which the shifted Lorentz form holds for every lane
    const bool lorentz = ymin >= LORENTZ_Y;
    const float xl = sqrtf(sqrtf(fmaf(2.0f * ymax, ymax, 1.5f) * (1.0f / DN_EPS_L)) * 1.001f);
    const float x_core = gh4_from(ymin);
    const float rdm = bartw::rcp_approx(dxm);
    const float p_far = xl * rdm, p_core = x_core * rdm;      // the same distances in points
    const float p_tab = 5.0f * rdm;                           // |z| >= 5: no table
    const float2 qL = f2(q - 1.5f), dx2 = f2(dx), xc2 = f2(xc);
    const int jl = w.jlo - w0, jh = w.jhi - w0;
    // steps of four points [0, s1) and [s4, steps) are far from every line,
    // [s1, s2) and [s3, s4) beyond the core, [s2, s3) within it for some
    auto left = [&](float d) { return min(max((int)floorf((cmin - d + 1.0f) * 0.25f), 0), steps); };
    auto right = [&](float d, int from) { return min(max((int)ceilf((cmax + d) * 0.25f), from), steps); };
    const int s1 = lorentz ? steps : left(p_far), s2 = max(left(p_core), s1);
    const int s3 = x_core < 0.0f ? s2 : right(p_core, s2), s4 = right(p_far, s3);
    auto add = [&](int s, float A0, float2 r0, float2 r1) {   // acc += A0 r
      float4 t = acc[s][lane];
      if (check) {                                            // (an infinite A0 stays within the line's window)
        const float2 v0 = mul2(f2(A0), r0), v1 = mul2(f2(A0), r1);
        const int j = 4 * s;
        if (j >= jl && j <= jh) t.x += v0.x;
        if (j + 1 >= jl && j + 1 <= jh) t.y += v0.y;
        if (j + 2 >= jl && j + 2 <= jh) t.z += v1.x;
        if (j + 3 >= jl && j + 3 <= jh) t.w += v1.y;
      } else {
        const float2 t0 = fma2(f2(A0), r0, make_float2(t.x, t.y)), t1 = fma2(f2(A0), r1, make_float2(t.z, t.w));
        t = make_float4(t0.x, t0.y, t1.x, t1.y);
      }
      acc[s][lane] = t;
    };
    auto at = [&](int s, int k) {                             // x of points 4 s + k and the next
      const float k0 = (float)(4 * s) - off;
      return fma2(add2(f2(k0), make_float2((float)k, (float)(k + 1))), dx2, xc2);
    };
    for (int e = steps - s4 + s1; e > 0; --e) {
      const int s = e > s1 ? steps - (e - s1) : s1 - e;
      const float2 xa = at(s, 0), xb = at(s, 2);
      add(s, A, rcp2(fma2(xa, xa, qL)), rcp2(fma2(xb, xb, qL)));
    }
    for (int e = (s2 - s1) + (s4 - s3); e > 0; --e) {
      const int s = e > s2 - s1 ? s4 - (e - (s2 - s1)) : s2 - e;
      add(s, A, gh4_ratio(at(s, 0), q), gh4_ratio(at(s, 2), q));
    }
    if (small) {
      for (int s = s2; s < s3; ++s) add(s, B, core_small(at(s, 0), y), core_small(at(s, 2), y));
    } else if (ymin >= GH8_Y) {
      for (int s = s2; s < s3; ++s) add(s, B, gh8_re<false>(at(s, 0), y), gh8_re<false>(at(s, 2), y));
    } else {
      for (int s = s2; s < s3; ++s) {
        const float p0 = (float)(4 * s);
        float2 r[2];
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          const float2 x = at(s, 2 * k);
          const float p = p0 + (float)(2 * k);
          r[k] = fmaxf(cmin - (p + 1.0f), p - cmax) >= p_tab ? gh8_re<true>(x, y) : core_any(x, y, a.wtab);
        }
        add(s, B, r[0], r[1]);
      }
    }
    if (++chunks % DN_FOLD == 0 && base + 32 < l1) {
      fold();
      for (int s = 0; s < steps; ++s) acc[s][lane] = make_float4(0.f, 0.f, 0.f, 0.f);
      for (int e = lane; e < DN_GROUPS * DN_P; e += 32) {
        float2 v = grp_folded[e];
        two_sum(v.x, v.y, grp[e]);
        grp_folded[e] = v;
        grp[e] = 0.0f;
      }
      __syncwarp();
    }
  }
  if (l1 > l0) fold();
  const int64_t at = (int64_t)blockIdx.y * a.nb + b;
#pragma unroll
  for (int q = 0; q < 3; ++q)
    if (lane + 32 * q < n_pts) a.window[at * DN_WIN + lane + 32 * q] = hi[q] + lo[q];
  // the groups' moments, and the block's from them
  for (int e = lane; e < ng * DN_P; e += 32)
    a.mg[((int64_t)blockIdx.y * a.g_stride + g0) * DN_P + e] = grp_folded[e].x + (grp_folded[e].y + grp[e]);
  if (lane < DN_P) {
    float t = 0.0f, l = 0.0f;
    for (int g = 0; g < ng; ++g) {
      const float2 v = grp_folded[g * DN_P + lane];
      two_sum(t, l, v.x);
      two_sum(t, l, grp[g * DN_P + lane]);
      l += v.y;
    }
    a.m8[at * DN_P + lane] = t + l;
  }
  if (plan.kind != DN_COMPLEX) return;
  // ---- moments about the complex centres, bin by bin; the bin's lines are
  // gathered in shared memory first, so that 32 of them are taken at a time
  const DenseBins bn = *a.bins;
  int* list = sh.list[warp];
  for (int bin = 0; bin < bn.n; ++bin) {
    float2 M[DN_PC];
#pragma unroll
    for (int n = 0; n < DN_PC; ++n) M[n] = make_float2(0.f, 0.f);
    const float gc = bn.c[bin] * cc.gfac;
    float2 mine = make_float2(0.f, 0.f), low = mine;          // lane n: moment n, a compensated pair
    int have = 0, taken = 0;                                  // taken: chunks of 32 since the last fold
    for (int base = l0; base < l1; base += 32) {
      const int next = base + lane;
      const bool in = next < l1 &&
                      min(max((int)floorf(log2f(a.gref[min(next, l1 - 1)] * bn.inv_g0) * bn.inv_lr), 0), bn.n - 1) == bin;
      const unsigned m = __ballot_sync(0xffffffffu, in);
      if (in) list[have + __popc(m & ((1u << lane) - 1u))] = next;
      have += __popc(m);
      __syncwarp();
      if (have < 32 && base + 32 < l1) continue;
      do {                                       // 32 lines, or at the end what is left
        const bool on = lane < have;
        const int i = list[on ? lane : 0];
        const LineWin w = a.win[have > 0 ? i : l0];
        const float gr = a.gref[have > 0 ? i : l0];
        const float ln_s = line_ln_s(w, cc);
        const float wt = (on && ln_s >= ln_thr) ? ex2f_approx((ln_s + LN_SCALE) * LOG2EF) * a.w_scale : 0.0f;
        const float inv = bartw::rcp_approx(w.nu0f * cc.dfac), rdx = bartw::rcp_approx(a.dnu * inv) * plan.ih, s2 = 0.5f * rdx * rdx;
        const float de = (((float)(w.jc - w0) - centre) - w.delta * a.inv_dnu) * plan.ih;
        const float ga = (gr * cc.gfac - gc) * (a.inv_dnu * plan.ih);
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
        __syncwarp();
        const int rest = list[32 + lane];        // those beyond the 32 taken, at most 31
        __syncwarp();
        list[lane] = rest;
        __syncwarp();
        have -= 32;
      } while (have > 0 && base + 32 >= l1);
      have = max(have, 0);
      if (++taken < DN_FOLD && base + 32 < l1) continue;
      taken = 0;
      float2 sum = make_float2(0.f, 0.f);
#pragma unroll
      for (int n = 0; n < DN_PC; ++n) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
          M[n].x += __shfl_xor_sync(0xffffffffu, M[n].x, o);
          M[n].y += __shfl_xor_sync(0xffffffffu, M[n].y, o);
        }
        if (lane == n) sum = M[n];
        M[n] = make_float2(0.f, 0.f);
      }
      two_sum(mine.x, low.x, sum.x);
      two_sum(mine.y, low.y, sum.y);
    }
    if (lane < DN_PC) a.mc8[(at * DN_BINS + bin) * DN_PC + lane] = make_float2(mine.x + low.x, mine.y + low.y);
  }
}

// Moments of the blocks of 32 points from their four blocks of 8: with t the
// offset of a block's centre, I'_n = sum_k C(n, k) t^(n-k) I_k (k >= 1).
__global__ void __launch_bounds__(128)
dense_up_kernel(const __grid_constant__ DenseArgs a) {
  const int P = blockIdx.x * blockDim.x + threadIdx.x;
  const DensePlan plan = a.plan[a.c0 + blockIdx.y];
  if (P >= a.nb / 4 || plan.kind == DN_NONE) return;
  const float* m = a.m8 + ((int64_t)blockIdx.y * a.nb + 4 * P) * DN_P;
  float o[DN_P] = {};
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    const float t = (float)(8 * c - 12) * plan.ih;
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
  if (plan.kind != DN_COMPLEX) return;
  for (int bin = 0; bin < a.bins->n; ++bin) {
    float2 u[DN_PC] = {};
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const float t = (float)(8 * c - 12) * plan.ih;
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

// sum_n I_n / D^(n+1), D in the moments' unit (the sums are in it, too)
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
  // distances from the centres of block b and parent P, in the moments' unit (exact)
  const float e8 = ((float)(j & 7) - 3.5f) * plan.ih, f8 = -8.0f * plan.ih;
  const float e32 = ((float)(j & 31) - 15.5f) * plan.ih, f32 = -32.0f * plan.ih;
  auto dist8 = [&](int b) { return fmaf((float)(b - t), f8, e8); };
  auto dist32 = [&](int P) { return fmaf((float)(P - T), f32, e32); };

  // ---- near: the windows of the blocks around the point
  float near = 0.0f;
  for (int b = t - plan.m1 + 1; b < t + plan.m1; ++b)
    near += win[(int64_t)b * DN_WIN + (t - b + plan.m1 - 1) * DN_B + (j & 7)];

  // ---- blocks inside the point's cutoff [bl, br), outside the near ones
  const int PL = (p.bl + 3) >> 2, PR = p.br >> 2;            // parents inside it
  FoldedSum far, mid;
  if (plan.kind == DN_COMPLEX) {
    const DenseBins bn = *a.bins;
    const float scale = a.cells[cell].gfac * a.inv_dnu * plan.ih;
    const float2* mc8 = a.mc8 + (int64_t)blockIdx.y * a.nb * DN_BINS * DN_PC;
    const float2* mc32 = a.mc32 + (int64_t)blockIdx.y * (a.nb / 4) * DN_BINS * DN_PC;
    // parents inside the cutoff: real centre far away, complex centres nearer
    const int u0 = __reduce_min_sync(0xffffffffu, PL), u1 = __reduce_max_sync(0xffffffffu, PR);
    folded_range(u0, u1, far, [&](int P) {
      const int m = abs(P - T);                  // the same for the warp
      const bool in = P >= PL && P < PR;
      const float D = dist32(P);
      if (m >= plan.m2) {
        if (in) far.s += moment_sum(m32 + (int64_t)P * DN_P, D);
      } else if (m >= plan.mh) {
        for (int q = 0; q < bn.n; ++q)
          if (in) far.s += complex_sum(mc32 + ((int64_t)P * DN_BINS + q) * DN_PC, D, bn.c[q] * scale);
      }
    });
    // blocks of the parents closer than that, and those beside the parents
    auto blocks8 = [&](int b0, int b1) {
      const int v0 = __reduce_min_sync(0xffffffffu, b0 < b1 ? b0 : 0x7fffffff);
      const int v1 = __reduce_max_sync(0xffffffffu, b0 < b1 ? b1 : -0x7fffffff);
      folded_range(v0, v1, mid, [&](int b) {
        const bool in = b >= b0 && b < b1 && abs(b - t) >= plan.m1;
        const float D = dist8(b);
        for (int q = 0; q < bn.n; ++q)
          if (in) mid.s += complex_sum(mc8 + ((int64_t)b * DN_BINS + q) * DN_PC, D, bn.c[q] * scale);
      });
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
    folded_range(u0, u1, far, [&](int P) {
      if (P >= PL && P < PE) far.s += moment_sum(m32 + (int64_t)P * DN_P, dist32(P));
    });
    const int v0 = __reduce_min_sync(0xffffffffu, PS), v1 = __reduce_max_sync(0xffffffffu, PR);
    far.fold();
    folded_range(v0, v1, far, [&](int P) {
      if (P >= PS && P < PR) far.s += moment_sum(m32 + (int64_t)P * DN_P, dist32(P));
    });
  }
  auto blocks = [&](int b0, int b1) {                        // [b0, b1), possibly empty
    const int u0 = __reduce_min_sync(0xffffffffu, b0 < b1 ? b0 : 0x7fffffff);
    const int u1 = __reduce_max_sync(0xffffffffu, b0 < b1 ? b1 : -0x7fffffff);
    folded_range(u0, u1, mid, [&](int b) {
      if (b >= b0 && b < b1) mid.s += moment_sum(m8 + (int64_t)b * DN_P, dist8(b));
    });
  };
  const bool hasL = PE > PL, hasR = PR > PS;
  blocks(p.bl, hasL ? min(4 * PL, lend) : lend);
  blocks(hasL ? 4 * PE : lend, lend);
  blocks(rbeg, hasR ? 4 * PS : p.br);
  blocks(hasR ? max(4 * PR, rbeg) : p.br, p.br);
  }

  // ---- edges: the block that a cutoff edge divides, group by group (blocks
  // within the near radius were taken line by line), or, where the profiles
  // are too wide for their moments about the real centre, line by line: at
  // least 23 points away, |x| > 9 (dense_applies), by the far form
  float edge = 0.0f;                                         // (of 2 DN_GROUPS terms at most)
  FoldedSum direct;
  const bool both = p.bl > p.br;                             // both edges divide the same block
  if (plan.lines) {
    const CellConst cc = a.cells[cell];
    const float ln_thr = a.smax ? ordered_float(a.smax[a.tmap[cell]]) + a.ln_rel : -3.0e38f;
    auto lines = [&](int i0, int i1, int b) {
      if (abs(b - t) < plan.m1) return;
      folded_range(i0, i1, direct, [&](int i) {
        const LineWin w = a.win[i];
        const float ln_s = line_ln_s(w, cc);
        if (!(ln_s >= ln_thr)) return;
        const float inv = bartw::rcp_approx(w.nu0f * cc.dfac), y = a.gref[i] * cc.gfac * inv;
        const float S = ex2f_approx((ln_s + LN_SCALE) * LOG2EF);
        const float x = fmaf((float)(j - w.jc), a.dnu * inv, w.delta * inv);
        direct.s = fmaf(S * inv * bartw::INV_SQRTPI * (y * bartw::INV_SQRTPI), far_ratio(x, y * y), direct.s);
      });
    };
    if (both) {
      lines(p.il, p.ir, p.br);
    } else {
      if (p.bl > 0) lines(p.il, min(a.lstart[p.bl], p.ir), p.bl - 1);
      if (p.br < a.nb) lines(max(a.lstart[p.br], p.il), p.ir, p.br);
    }
  } else {
    auto groups = [&](int g0, int g1, int b) {
      if (abs(b - t) < plan.m1) return;
      const float D = dist8(b);
      for (int g = max(g0, 0); g < min(g1, (int)a.g_stride); ++g) edge += moment_sum(mg + (int64_t)g * DN_P, D);
    };
    if (both) {
      groups(p.gl, p.gr, p.br);
    } else {
      if (p.bl > 0) groups(p.gl, min(a.gfirst[p.bl], p.gr), p.bl - 1);
      if (p.br < a.nb) groups(max(a.gfirst[p.br], p.gl), p.gr, p.br);
    }
  }
  if (j0 + lane < a.n_nu) a.out[(int64_t)cell * a.n_nu + j] = (((edge + far.total()) + mid.total()) * plan.ih + (near + direct.total())) * INV_SCALE;
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
    // x of one grid interval: from 0.4 on (a Doppler deviation of 1.8 points) the
    // reach of a line's moments (dense_plan_kernel) stays within the near radii;
    // the near window's products of four squared x (within 12 points of a
    // line's) stay in the FP32 range
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
  const int boff = ((reach + 2) / DN_B + DN_M1 + 4) / 4 * 4;         // blocks before the grid, whole parents
  const int nb = (boff + n_nu / DN_B + (reach + 2) / DN_B + DN_M1 + 8) / 4 * 4;
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
  const double hi = nu.nu_start_cm + (double)n_nu * nu.dnu_cm + cutoff;
  dense_plan_kernel<<<(n_cells + 127) / 128, 128, 0, s>>>(cells, n_cells, stat, (float)(1.0 / nu.dnu_cm),
                                                         (float)(hi / nu.dnu_cm * 0.70710678118654752), reach, pl, bins);
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
