// a1: the strength of one line, in the full FP64 and the reduced form, and its per-temperature
// constants (shared by the kernels of rox_params.cu and rox_prep.cu).
#pragma once
#include "rox_internal.cuh"

namespace {

struct StrengthConsts {
  int convention;
  double inv_T;        // 1/T
  double q_ratio;      // HITRAN: Q_ref/Q_T ; ExoMol: 1/Q_T
  double c2_dT;        // HITRAN: c2 (1/T - 1/T_ref) ; ExoMol: c2/T
  // for the reduced form: c2_dT / ln 2 as two floats, c2/T and q_ratio in FP32
  float g_hi, g_lo, c2_T, q_ratio_f;
};
__host__ __device__ inline void set_reduced(StrengthConsts* k) {
  const double g = k->c2_dT * 1.4426950408889634074;
  k->g_hi = (float)g;
  k->g_lo = (float)(g - (double)k->g_hi);
  k->c2_T = (float)(ROX_C2 * k->inv_T);
  k->q_ratio_f = (float)k->q_ratio;
}

// S(T) in FP64 for one line (HITRAN S_ref form or ExoMol Einstein-A form).
__device__ __forceinline__ double line_strength(const StrengthConsts& k, double nu0, double s_or_a,
                                                double g_up, double e_lower) {
  double stim_T = -expm1(-ROX_C2 * nu0 * k.inv_T);           // 1 - exp(-c2 nu0 / T)
  double boltz = exp(-e_lower * k.c2_dT);
  if (k.convention == ROX_HITRAN) {
    double stim_ref = -expm1(-ROX_C2 * nu0 / ROX_T_REF);
    return s_or_a * k.q_ratio * boltz * (stim_T / stim_ref);
  }
  return g_up * s_or_a / (8.0 * ROX_PI * ROX_C_CM * nu0 * nu0) * boltz * stim_T * k.q_ratio;
}

// The same S(T) for the cross-section launches, with almost no FP64 operation: this GPU runs FP64 at
// about two operations per clock per SM, FP64 exp, expm1 and a division cost ~70 of them per line,
// and the fourteen of an FP64 reduction of the exponent alone still took 0.32 ms for 1e7 lines, six
// times their bytes. Only the Boltzmann exponent needs more than FP32: a / ln 2 = -e_lower g with g
// held as two floats is formed as an exact product and its remainder (an FMA), so that k = rint and
// the fraction f = a/ln 2 - k, |f| <= 1/2, come out to 3e-8. 2^f, the stimulated-emission factor and
// the prefactor are FP32, and the FP32 product (pre-scaled by 2^64 against underflow) is put back in
// range by the exact power 2^(k - 64), an integer addition to the exponent of the double. Relative
// error a few 1e-7 (FP32 roundings), far below the cross-section tolerance; exponents beyond +-700 and
// FP32 products beyond 2^+-100 (or zero, or NaN) take the FP64 form.
__device__ __forceinline__ double line_strength_fast(const StrengthConsts& k, double nu0, float s_or_a, float g_up,
                                                     float e_lower) {
  const float q = -e_lower * k.g_hi;                           // a / ln 2, rounded
  if (!(fabsf(q) < 1009.88f)) return line_strength(k, nu0, (double)s_or_a, (double)g_up, (double)e_lower);
  const float rem = fmaf(-e_lower, k.g_lo, fmaf(-e_lower, k.g_hi, -q));
  const float kf = rintf(q);
  const float m = exp2f((q - kf) + rem);
  const float nu = (float)nu0;
  const float stim = -expm1f(-k.c2_T * nu);
  float p;
  if (k.convention == ROX_HITRAN) {
    const float stim_ref = -expm1f(-(float)(ROX_C2 / ROX_T_REF) * nu);
    p = (s_or_a * 0x1p64f) * k.q_ratio_f * (stim / stim_ref);
  } else {
    p = (g_up * s_or_a) * ((float)(0x1p64 / (8.0 * ROX_PI * ROX_C_CM)) / (nu * nu)) * stim * k.q_ratio_f;
  }
  const float pm = p * m;
  if (!(fabsf(pm) >= 0x1p-100f && fabsf(pm) <= 0x1p100f))   // outside FP32's comfortable range (or 0, NaN)
    return line_strength(k, nu0, (double)s_or_a, (double)g_up, (double)e_lower);
  const int ki = (int)kf;
  if (ki < -850) {   // may leave the normal range: two rounded products
    const double two_k = __longlong_as_double((long long)(ki + 1023) << 52);   // 2^k, |k| <= 1010
    return (double)pm * 0x1p-64 * two_k;
  }
  return __longlong_as_double(__double_as_longlong((double)pm) + ((long long)(ki - 64) << 52));
}

// Running maximum of strengths as double bits: non-negative values order like their bit patterns;
// negative and NaN ones count as 0.
__device__ __forceinline__ unsigned long long max_bits(unsigned long long mx, double s) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(s);
  return b <= 0x7ff0000000000000ULL && b > mx ? b : mx;
}
__device__ __forceinline__ void store_max(unsigned long long mx, unsigned long long* out) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long v = __shfl_xor_sync(0xffffffffu, mx, o);
    mx = v > mx ? v : mx;
  }
  if ((threadIdx.x & 31) == 0 && mx) atomicMax(out, mx);
}

inline StrengthConsts make_consts(int convention, double T, double Q_T, double Q_ref) {
  StrengthConsts k;
  k.convention = convention;
  k.inv_T = 1.0 / T;
  if (convention == ROX_HITRAN) {
    k.q_ratio = Q_ref / Q_T;
    k.c2_dT = ROX_C2 * (1.0 / T - 1.0 / ROX_T_REF);
  } else {
    k.q_ratio = 1.0 / Q_T;
    k.c2_dT = ROX_C2 / T;
  }
  set_reduced(&k);
  return k;
}

}  // namespace
