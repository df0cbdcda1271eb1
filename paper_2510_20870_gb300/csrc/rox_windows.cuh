// a3: the cutoff window and centre decomposition of one line on a uniform grid (shared by the
// kernels of rox_geometry.cu and rox_prep.cu).
#pragma once
#include <math.h>
#include "rox_internal.cuh"

namespace {

// d_j = (nu_min + j*dnu) - nu0 with each operation rounded separately (no contraction),
// exactly the double-precision expression of the cutoff test.
__device__ __forceinline__ double node_offset(double nu_min, double dnu, long long j, double nu0) {
  return __dsub_rn(__dadd_rn(nu_min, __dmul_rn((double)j, dnu)), nu0);
}

// This GPU issues about two FP64 operations per clock per SM, and a window has some twenty of them if
// its floor, ceiling and comparisons are done in FP64 (0.50 ms for 1e7 lines). So the line centre in
// index units u = (nu0 - nu_min)/dnu is formed in FP64, scaled by 2^ROX_U_BITS (exactly) and
// rounded down to a 64-bit integer, and everything else is integer arithmetic: three FP64
// operations a line, 0.08 ms. `guard` bounds, in index units, the rounding of the candidates
// u -+ cutoff/dnu and of the cutoff test for every line within reach of the grid: a candidate
// farther than that from an integer is the exact answer, and the exact FP64 test only runs for the
// others (about one line in 1e6). Centres beyond +-2^24 grid steps, out of any grid's reach, are
// held there.
#define ROX_U_BITS 38
struct RoxWindows {
  double nu_min, dnu, scale, cutoff;   // scale: 2^ROX_U_BITS / dnu
  double inv_dnu;
  long long c_fix, guard_fix;          // cutoff/dnu and guard in units of 2^-ROX_U_BITS
  long long n_grid;
  float dnu_hi, dnu_lo;                // dnu as a float pair
  float k_lo, k_hi;                    // centres of lines beyond reach in the geometry records
};
struct LineWindow {
  int jl, jh, k0;
  float4 geo;       // {k0, f dnu, jlo, jhi} (RoxListDev::geo)
};
__device__ __forceinline__ LineWindow line_window(const RoxWindows& W, double nu0) {
  const long long mask = (1LL << ROX_U_BITS) - 1, far = 1LL << (24 + ROX_U_BITS);
  const int n_grid = (int)W.n_grid;
  LineWindow w;
  // first j with d_j >= -cutoff, last j with d_j <= cutoff (d_j non-decreasing in j): a
  // candidate from the line centre, then the exact test moves it where it could be off. The
  // conversion saturates; a NaN centre becomes the lowest value, an empty window.
  const long long U = max(-far, min(far, __double2ll_rd((nu0 - W.nu_min) * W.scale)));
  const long long r_lo = U - W.c_fix, r_hi = U + W.c_fix;
  int jlo = (int)((r_lo + mask) >> ROX_U_BITS), jhi = (int)(r_hi >> ROX_U_BITS);
  jlo = min(max(jlo, -4), n_grid + 4);
  jhi = min(max(jhi, -4), n_grid + 4);
  // within the guard of an integer on either side
  if (((r_lo + W.guard_fix) & mask) <= 2 * W.guard_fix) {
    for (int it = 0; it < 4 && node_offset(W.nu_min, W.dnu, jlo - 1, nu0) >= -W.cutoff; it++) jlo--;
    for (int it = 0; it < 4 && node_offset(W.nu_min, W.dnu, jlo, nu0) < -W.cutoff; it++) jlo++;
  }
  if (((r_hi + W.guard_fix) & mask) <= 2 * W.guard_fix) {
    for (int it = 0; it < 4 && node_offset(W.nu_min, W.dnu, jhi + 1, nu0) <= W.cutoff; it++) jhi++;
    for (int it = 0; it < 4 && node_offset(W.nu_min, W.dnu, jhi, nu0) > W.cutoff; it++) jhi--;
  }
  w.jl = min(max(jlo, 0), n_grid);
  w.jh = min(max(jhi, -1), n_grid - 1);
  w.k0 = (int)(U >> ROX_U_BITS);      // centre decomposition (nu0 - nu_min)/dnu = k0 + f, f in [0, 1)
  // f dnu from the fraction in two parts of 24 and 14 bits, rounded once but for 2^-38. The
  // record's centre must not decrease along the list: a line beyond the grid's reach, never
  // evaluated, is put just outside the centres that reach it.
  const float fh = (float)(int)((U >> 14) & 0xffffff) * 0x1p-24f, fl = (float)(int)(U & 0x3fff) * 0x1p-38f;
  const float k = (float)w.k0, kg = fminf(fmaxf(k, W.k_lo), W.k_hi);
  const float fd = fmaf(fh, W.dnu_hi, fmaf(fh, W.dnu_lo, fl * W.dnu_hi));
  w.geo = make_float4(kg, kg == k ? fd : 0.0f, __int_as_float(w.jl), __int_as_float(w.jh));
  return w;
}

inline RoxWindows rox_windows(const rox_grid* g, double cutoff) {
  // rounding bound of the candidates and of the cutoff test, in index units: every quantity
  // involved is at most |nu| + 2 cutoff in cm^-1 (or n + 8 in index units) for a line within
  // reach; 16 double-precision ulps of each is a generous margin
  const double inv_dnu = 1.0 / g->dnu;
  const double nu_abs = fmax(fabs(g->nu_min), fabs(g->nu_min + (double)(g->n - 1) * g->dnu));
  const double guard = 16.0 * 2.3e-16 * ((nu_abs + 2.0 * cutoff) * inv_dnu + (double)g->n + 8.0);
  const double one = (double)(1LL << ROX_U_BITS), c_idx = cutoff * inv_dnu;
  RoxWindows W;
  W.nu_min = g->nu_min;
  W.dnu = g->dnu;
  W.scale = inv_dnu * one;
  W.inv_dnu = inv_dnu;
  W.cutoff = cutoff;
  W.c_fix = (long long)rint(c_idx * one);
  // two units more for the roundings to fixed point; a guard of half a step or more tests every line
  W.guard_fix = guard < 0.5 ? (long long)ceil(guard * one) + 2 : (1LL << ROX_U_BITS);
  W.n_grid = g->n;
  W.dnu_hi = (float)g->dnu;
  W.dnu_lo = (float)(g->dnu - (double)W.dnu_hi);
  W.k_lo = -(float)(ceil(c_idx) + 8.0);
  W.k_hi = (float)((double)g->n + ceil(c_idx) + 8.0);
  return W;
}

}  // namespace
