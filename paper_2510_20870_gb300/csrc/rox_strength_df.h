// The line strength in pairs of floats (an unevaluated sum hi + lo), for results that are rounded to
// FP32 (rox_line_strengths). FP64 arithmetic issues at about two operations per clock per SM here and the
// FP64 form needs some 65 of them per line; FP32 issues at 128. The pair form is good to
// ROX_DF_ERR; its rounding is taken where it is certain (hi + lo not within ROX_DF_ERR of the middle of
// two floats), otherwise the caller takes the FP64 form, so the results are those of the FP64 form.
// Sums and products without error after Knuth and Dekker; exp by a table of 2^(j/32) and a short
// Taylor series after Tang's method. Compiled for the host as well, where its error is measured.
#pragma once
#include <math.h>
#include <stdint.h>
#include <string.h>

#ifdef __CUDACC__
#define ROX_DF __host__ __device__ __forceinline__
#else
#define ROX_DF inline
#endif

#define ROX_DF_ERR 0x1p-35f   // relative error bound of the pair form; measured: below 2^-37

struct rox_df { float h, l; };

ROX_DF float rox_df_mul1(float a, float b) {      // a product that stays rounded by itself
#ifdef __CUDA_ARCH__
  return __fmul_rn(a, b);
#else
  return a * b;
#endif
}
ROX_DF rox_df rox_df_two_sum(float a, float b) {
  const float s = a + b, t = s - a;
  return {s, (a - (s - t)) + (b - t)};
}
ROX_DF rox_df rox_df_fast_sum(float a, float b) {   // |a| >= |b|, or a = 0
  const float s = a + b;
  return {s, b - (s - a)};
}
ROX_DF rox_df rox_df_prod(float a, float b) {
  const float p = rox_df_mul1(a, b);
  return {p, fmaf(a, b, -p)};
}
ROX_DF rox_df rox_df_mul(rox_df a, rox_df b) {
  const rox_df p = rox_df_prod(a.h, b.h);
  return rox_df_fast_sum(p.h, p.l + fmaf(a.h, b.l, a.l * b.h));
}
ROX_DF rox_df rox_df_div(rox_df a, rox_df b) {
  const float q = a.h / b.h;
  const float r = fmaf(-q, b.h, a.h) + fmaf(-q, b.l, a.l);
  return rox_df_fast_sum(q, r / b.h);
}
ROX_DF rox_df rox_df_split(double x) {   // host-side constants
  const float h = (float)x;
  return {h, (float)(x - (double)h)};
}
ROX_DF uint32_t rox_df_bits(float x) {
#ifdef __CUDA_ARCH__
  return __float_as_uint(x);
#else
  uint32_t u;
  memcpy(&u, &x, 4);
  return u;
#endif
}
ROX_DF float rox_df_float(uint32_t u) {
#ifdef __CUDA_ARCH__
  return __uint_as_float(u);
#else
  float x;
  memcpy(&x, &u, 4);
  return x;
#endif
}
ROX_DF uint64_t rox_df_bits64(double x) {
#ifdef __CUDA_ARCH__
  return (uint64_t)__double_as_longlong(x);
#else
  uint64_t u;
  memcpy(&u, &x, 8);
  return u;
#endif
}
ROX_DF double rox_df_double(uint64_t u) {
#ifdef __CUDA_ARCH__
  return __longlong_as_double((long long)u);
#else
  double x;
  memcpy(&x, &u, 8);
  return x;
#endif
}

// exp(a), a = a0 + a1 + a2 with |a0| < 700 and |a1| below 2^-14: exp(a) = tab[n & 31] 2^(n >> 5) (1 + s)
struct rox_df_exp_parts { int n; rox_df s; };
ROX_DF rox_df_exp_parts rox_df_exp(float a0, float a1, float a2) {
  // ln 2 / 32 as three floats; n L1 is exact to 2^-29, as is a0, so the first difference is exact
  const float L1 = 0x1.62e430p-6f, L2 = -0x1.05c610p-34f, L3 = -0x1.950d88p-59f;
  const float nf = rintf(a0 * 46.16624130844683f);
  const float r0 = fmaf(-nf, L1, a0);
  const rox_df p = rox_df_prod(nf, L2);
  const rox_df u = rox_df_two_sum(r0, a1), v = rox_df_two_sum(u.h, -p.h);
  const rox_df r = rox_df_two_sum(v.h, ((u.l + v.l) + (a2 - p.l)) - nf * L3);
  const rox_df q = rox_df_prod(r.h, r.h);
  const float t = q.h * r.h * fmaf(r.h, fmaf(r.h, 1.0f / 120.0f, 1.0f / 24.0f), 1.0f / 6.0f);
  const rox_df s = rox_df_fast_sum(r.h, 0.5f * q.h);
  return {(int)nf, rox_df_fast_sum(s.h, s.l + (fmaf(r.h, r.l, r.l) + fmaf(0.5f, q.l, t)))};
}
// tab[j] (1 + s)
ROX_DF rox_df rox_df_scale1p(rox_df T, rox_df s) {
  const rox_df p = rox_df_prod(T.h, s.h);
  const rox_df u = rox_df_fast_sum(T.h, p.h);
  return rox_df_fast_sum(u.h, u.l + (T.l + p.l + fmaf(T.h, s.l, T.l * s.h)));
}
// 1 - exp(-x), x = xh + xl in (0, 60]
ROX_DF rox_df rox_df_one_minus_exp(rox_df x, const rox_df* tab) {
  const rox_df_exp_parts e = rox_df_exp(-x.h, -x.l, 0.0f);
  const float two_k = rox_df_float((uint32_t)((e.n >> 5) + 127) << 23);
  const rox_df T = tab[e.n & 31];
  const float th = T.h * two_k, tl = T.l * two_k;
  const rox_df d = rox_df_two_sum(1.0f, -th), m = rox_df_prod(th, e.s.h);
  const rox_df g = rox_df_two_sum(d.h, -m.h);
  return rox_df_fast_sum(g.h, g.l + (d.l - tl - m.l - fmaf(th, e.s.l, tl * e.s.h)));
}

// constants of a temperature; c = c2_dT as three floats, x_T = c2/T, x_ref = c2/T_ref, q = the constant
// factors scaled by 2^-q_exp into [1, 2)
struct rox_df_consts {
  int hitran, q_exp, ok;
  float c0, c1, c2;
  rox_df x_T, x_ref, q;
};

// S = h 2^e (1 + d), |d| < ROX_DF_ERR; false where an operand is outside the pair form's range
ROX_DF bool rox_df_strength(const rox_df_consts& k, const rox_df* tab, double nu0, float s_or_a, float g_up,
                            float e_lower, rox_df* out, int* e_out) {
  const uint64_t nb = rox_df_bits64(nu0);
  const uint32_t ab = rox_df_bits(s_or_a), gb = rox_df_bits(k.hitran ? 1.0f : g_up);
  const int en = (int)(nb >> 52) - 1023, ea = (int)(ab >> 23) - 127, eg = (int)(gb >> 23) - 127;
  // positive normal operands, the centre within 2^+-20 cm^-1 (a sign bit makes the exponent large)
  if (!(k.ok && en >= -20 && en < 20 && ea > -127 && ea < 128 && eg > -127 && eg < 128)) return false;
  const rox_df a = rox_df_prod(-e_lower, k.c0), a1 = rox_df_prod(-e_lower, k.c1);
  if (!(fabsf(a.h) < 690.0f)) return false;
  const rox_df a01 = rox_df_two_sum(a.l, a1.h);
  const rox_df_exp_parts b = rox_df_exp(a.h, a01.h, a01.l + fmaf(-e_lower, k.c2, a1.l));
  // the centre: 24 leading bits and the other 29
  const float nh = rox_df_float((uint32_t)((nb >> 29) & 0x7fffffu) | ((uint32_t)(en + 127) << 23));
  const float nl = (float)(uint32_t)(nb & 0x1fffffffu) * rox_df_float((uint32_t)(en - 52 + 127) << 23);
  const rox_df nu = rox_df_fast_sum(nh, nl);
  rox_df x = rox_df_mul(nu, k.x_T);
  if (!(x.h > 0x1p-30f)) return false;
  if (x.h > 60.0f) x = {60.0f, 0.0f};              // exp(-60) = 2^-86: the factor is 1
  const rox_df stim = rox_df_one_minus_exp(x, tab);
  const rox_df A = {rox_df_float((ab & 0x7fffffu) | 0x3f800000u), 0.0f};
  rox_df f = rox_df_mul(rox_df_mul(A, k.q), rox_df_scale1p(tab[b.n & 31], b.s));
  rox_df den;
  if (k.hitran) {
    x = rox_df_mul(nu, k.x_ref);
    if (!(x.h > 0x1p-30f)) return false;
    if (x.h > 60.0f) x = {60.0f, 0.0f};
    den = rox_df_one_minus_exp(x, tab);
  } else {
    den = rox_df_mul(nu, nu);
    f = rox_df_mul(f, {rox_df_float((gb & 0x7fffffu) | 0x3f800000u), 0.0f});
  }
  *out = rox_df_mul(f, rox_df_div(stim, den));
  *e_out = ea + eg + k.q_exp + (b.n >> 5);
  return true;
}

// h 2^e rounded to FP32 if that is certain
ROX_DF bool rox_df_round(rox_df s, int e, float* out) {
  const int x = (int)(rox_df_bits(s.h) >> 23) + e;      // s.h is positive and normal
  if (x >= 1 && x < 255) {
    const float d = s.h * ROX_DF_ERR;
    if (s.h + (s.l + d) != s.h || s.h + (s.l - d) != s.h) return false;
    *out = rox_df_float(rox_df_bits(s.h) + ((uint32_t)e << 23));
    return true;
  }
  if (x >= 255) return false;
  if (x < -30) {                                        // below half of the smallest FP32 number
    *out = 0.0f;
    return true;
  }
  const double v = ((double)s.h + (double)s.l) * rox_df_double((uint64_t)(e + 1023) << 52);
  const float lo = (float)(v * (1.0 - (double)ROX_DF_ERR)), hi = (float)(v * (1.0 + (double)ROX_DF_ERR));
  *out = lo;
  return lo == hi;
}

inline rox_df_consts rox_df_make_consts(int hitran, double c2_dT, double q_fac, double c2_over_T, double c2_over_Tref) {
  rox_df_consts k;
  k.hitran = hitran;
  k.c0 = (float)c2_dT;
  k.c1 = (float)(c2_dT - (double)k.c0);
  k.c2 = (float)(c2_dT - (double)k.c0 - (double)k.c1);
  k.x_T = rox_df_split(c2_over_T);
  k.x_ref = rox_df_split(c2_over_Tref);
  int e = 0;
  const double m = frexp(q_fac, &e);
  k.q = rox_df_split(2.0 * m);
  k.q_exp = e - 1;
  // zero, negative, infinite or NaN factors and vanishing exponents are left to the FP64 form
  k.ok = q_fac > 0.0 && q_fac < 1e300 && fabs(c2_dT) < 1e6 && (c2_dT == 0.0 || fabs(c2_dT) > 1e-12) &&
         c2_over_T > 1e-12 && c2_over_T < 1e6;
  return k;
}
