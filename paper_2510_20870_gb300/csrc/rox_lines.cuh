// Per-line constants of the Voigt kernel at one (P,T) point: widths, far-form constants, slow zone
// (shared by the kernels of rox_voigt.cu and rox_prep.cu).
#pragma once
#include <cuda_fp16.h>
#include "rox_internal.cuh"
#include "rox_faddeeva.cuh"

namespace {

#define ROX_INV_PI 0.318309886183790672f

__device__ __forceinline__ float load_width(const void* p, int f16, long long i) {
  return f16 ? __half2float(reinterpret_cast<const __half*>(p)[i])
             : reinterpret_cast<const float*>(p)[i];
}

// the two per-line width inputs of line i: {gamma_ref, n_T} of the single power law, or, for
// broadened lists (BRD), {the broadeners' sum at the job's temperature, the natural width}
template <bool BRD>
__device__ __forceinline__ void load_widths(const RoxJobDev& J, const RoxListDev& L, int f16, long long i, float& a,
                                            float& b) {
  if constexpr (BRD) {
    a = L.gLT[(long long)J.t_row * L.gLT_stride + i];
    b = L.gN ? L.gN[i] : 0.0f;
  } else {
    a = load_width(L.gamma_ref, f16, i);
    b = load_width(L.n_t, f16, i);
  }
}

// Whether a line whose window covers the span and whose slow zone misses it is smooth there: its
// far form at the span's 32 Chebyshev points then gives it at every point of the span by
// polynomial interpolation. D: |offset| of the span's centre from the line, h: the span's
// half-width. The far form's poles X^2 = -A +- sqrt(-B) have real parts of at most
// Rp = sqrt(max(0, -A) + sqrt|B|); with none within 1.25 h of the centre the error of degree 31 is
// below 1e-7 (a Bernstein ellipse of parameter 2: 2^-32 times 128 / (1.25^2 - 1)).
#define ROX_SMOOTH_R 1.25f
__device__ __forceinline__ float smooth_dmin(float A, float B, float h) {
  const float b = fabsf(B) + 1e-30f;
  const float rp2 = fmaxf(0.0f, -A) + b * rox_rsqrt(b) + 1e-30f;
  return fmaf(ROX_SMOOTH_R, h, rp2 * rox_rsqrt(rp2));
}

// Per-line constants of one (P,T) point that do not depend on the span: the far-form
// constants, the slow zone's half-width hz (at least the precision margin) and threshold t_z,
// and what pass 2 needs. nu0f: the line centre in FP32; Sp: S 2^-e; gref, nt: the width inputs
// (see load_widths). The Voigt kernel computes them per line and span, or (ROX_VX_PRE) reads
// them from the record that the preparation kernel (rox_prep.cu) computes once per line with this same function.
struct LineK {
  float A, B, P, Q, tz, iG, y, pc, zc, hz;
};
template <bool BRD>
__device__ __forceinline__ LineK line_consts(float nu0f, float Sp, float gref, float nt, const RoxJobDev& J,
                                             float margin_cm) {
  LineK k;
  const float gG = nu0f * J.gG_fac;
  const float gL = BRD ? fmaf(gref, J.p_fac, nt) : gref * rox_exp2(nt * J.l2_ratio) * J.p_fac;
  const float gG2 = gG * gG, gL2 = gL * gL;
  const float pY = Sp * gL * ROX_INV_PI;
  const float invG = rox_rcp(gG);
  k.y = gL * invG;
  const rox_far fc = rox_far_coefs(k.y);      // far-zone form of this line (rox_faddeeva.cuh)
  // slow zone: |X| < sqrt(r2 gamma_G^2 - gamma_L^2), at least the precision margin (see below)
  const float hz2 = fmaxf(0.0f, fc.r2 * gG2 - gL2);
  float hz = hz2 * rox_rsqrt(hz2);            // 0 for hz2 = 0 (rsqrt(0) = inf, product taken as 0 below)
  hz = hz2 > 0.0f ? hz : 0.0f;
  // the margin keeps the offset's rounding small against |X|, or against gamma_L where that is the larger
  // scale of the profile (its poles lie gamma_L off the axis): a broad line needs less of it, or none
  const float mg2 = fmaxf(0.0f, fmaf(margin_cm, margin_cm, -gL2));
  const float mg = mg2 > 0.0f ? mg2 * rox_rsqrt(mg2) : 0.0f;
  k.zc = hz >= mg ? 3e38f : hz2;
  k.hz = fmaxf(hz, mg);
  k.A = fc.alpha * gG2;
  k.B = fc.beta * (gG2 * gG2);
  k.P = pY;
  k.Q = pY * (fc.kappa * gG2);
  k.tz = fmaf(k.hz, k.hz, k.A);
  k.iG = invG;
  k.pc = Sp * invG * ROX_INV_SQRT_PI;
  return k;
}

// Grid indices of a line's slow zone on a uniform grid, |j - (k0 + f)| < hz / dnu, widened by 1e-4
// relative and one point on each side (covers every point with t < t_z despite the roundings).
// g: the line's geometry record {k0, f dnu, jlo, jhi}.
__device__ __forceinline__ void zone_bounds(const float4& g, float hz, float inv_dnu, int& zlo, int& zhi) {
  const int k0 = (int)g.x;
  const float hzg = fminf(hz * inv_dnu * 1.0001f, 8.0e6f);
  const float fr = g.y * inv_dnu;
  zlo = k0 + __float2int_rd(fr - hzg) - 1;
  zhi = k0 + __float2int_ru(fr + hzg) + 1;
}

// the uniform grid's precision margin of the slow zones (cm^-1; see ROX_FAST_MARGIN)
__device__ __forceinline__ float fast_margin(float dnu_f) { return ROX_FAST_MARGIN * 32.0f * (ROX_K - 1) * dnu_f; }

}  // namespace
