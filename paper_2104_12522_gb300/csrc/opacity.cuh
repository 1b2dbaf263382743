// What the line-by-line opacity kernels share: the per-line and per-cell
// constants, the line strength, and the plan of the kernels for dense line
// lists (opacity_dense.cu).
#pragma once

#include <vector>

#include "bart_internal.cuh"
#include "faddeeva.cuh"

namespace bartop {

constexpr float LN_SCALE = 69.314718055994531f;   // ln(2^100): internal scale of all terms
constexpr float INV_SCALE = 7.888609052210118e-31f; // 2^-100
constexpr float LOG2EF = 1.4426950408889634f;
constexpr float LN2F_ = 0.6931471805599453f;

__device__ __forceinline__ float ex2f_approx(float a) {
  float r;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(a));
  return r;
}
__device__ __forceinline__ float lg2f_approx(float a) {
  float r;
  asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(a));
  return r;
}

struct LineWin {            // per line, from the FP64 prologue
  int jlo, jhi, jc;
  float delta;              // nu_jc - nu0 (cm^-1)
  float ln_s0;              // ln S_ref + c2 E''/T_ref - ln(1 - exp(-c2 nu0/T_ref)): the T-free part of ln S(T)
  float c2e;                // c2 E''
  float c2nu;               // c2 nu0
  float nu0f;               // nu0 in FP32
};

struct CellConst {
  float inv_t;              // 1 / T
  float ln_q;               // 1.5 ln(296 / T): partition-function ratio
  float gfac;               // P sqrt(296 / T)  (bar)
  float dfac;               // sqrt(2 k T / m) / c: sigma*sqrt2 = nu0 * dfac
  float c2_t;               // c2 / T
  int dense;                // the widths suit the kernels for dense lists (dense_applies)
};

__device__ __forceinline__ double nu_minus(double nu_start, double dnu, int64_t j, double nu0) {
  // (nu_start + j*dnu) - nu0, each operation rounded separately (no FMA).
  return __dadd_rn(__dadd_rn(nu_start, __dmul_rn((double)j, dnu)), -nu0);
}

// ln S(T) = ln_s0 + 1.5 ln(T_ref/T) - c2 E''/T + ln(1 - exp(-c2 nu0/T)), in FP32
// (the staging of the opacity kernel and the threshold prologue share it).
__device__ __forceinline__ float line_ln_s(const LineWin& w, const CellConst& cc) {
  const float stim = 1.0f - ex2f_approx(-w.c2nu * cc.inv_t * LOG2EF);
  return w.ln_s0 + cc.ln_q - w.c2e * cc.inv_t + LN2F_ * lg2f_approx(stim);
}

// Order-preserving map of floats to ints (for atomicMax on floats).
__device__ __forceinline__ int ordered_int(float f) {
  const int i = __float_as_int(f);
  return i >= 0 ? i : i ^ 0x7fffffff;
}
__device__ __forceinline__ float ordered_float(int i) { return __int_as_float(i >= 0 ? i : i ^ 0x7fffffff); }

// First index in [lo, hi) with key[i] >= v (key nondecreasing).
__device__ inline int64_t lower_bound_i(const int* __restrict__ key, int64_t lo, int64_t hi, int v) {
  while (lo < hi) {
    int64_t mid = (lo + hi) >> 1;
    if (key[mid] < v) lo = mid + 1; else hi = mid;
  }
  return lo;
}

// Per (P, T) cell, what the kernels for dense lists do (opacity_dense.cu): near
// radius m1 in blocks of 8 points; blocks of 32 points from m2 blocks on by
// their moments about the centre, from mh on by those about complex centres
// (DN_COMPLEX).
enum { DN_NONE = 0, DN_REAL = 1, DN_COMPLEX = 2 };   // DN_NONE: line by line (opacity_kernel)
struct DensePlan {
  int kind, m1, mh, m2;
  float ih;                 // moments are of lengths times ih (a power of two)
  int lines;                // divided blocks line by line, not by their groups' moments
};

// Whether a species' list is dense enough on this grid for those kernels;
// marks the cells whose line widths allow them (cells[c].dense).
bool dense_applies(const bart_linelist& lines, const bart_nugrid& nu, double cutoff, CellConst* cells, int n_cells);

// The marked cells of one species: win, jlo and jhi from
// line_window_kernel; *plan (device, [n_cells]) tells opacity_kernel which
// cells it has left.  out [n_cells][n_nu].
bart_status dense_cells(bart_ctx* ctx, const LineWin* win, const int* jlo, const int* jhi, const float* gref,
                        int64_t n_lines, const CellConst* cells, int n_cells, const bart_nugrid& nu, double cutoff,
                        const int* smax, const int* tmap, float ln_rel, float* out,
                        const DensePlan** plan);

}  // namespace bartop
