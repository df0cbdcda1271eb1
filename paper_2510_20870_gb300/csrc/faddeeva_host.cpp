// Host (CPU) build of the FP32 Faddeeva code used by the CUDA kernels, so its accuracy
// can be measured against scipy.special.wofz without a GPU.
#include <stdint.h>
#include "rox_faddeeva.cuh"
#include "rox_strength_df.h"

extern "C" void rox_host_re_w(const float* x, const float* y, float* out, int64_t n) {
  for (int64_t i = 0; i < n; i++) out[i] = rox_re_w(&rox_daw_taylor[0][0], x[i], y[i]);
}

extern "C" void rox_host_re_w_far(const float* x, const float* y, float* out, int64_t n) {
  for (int64_t i = 0; i < n; i++) out[i] = rox_re_w_far(x[i], y[i]);
}

extern "C" float rox_host_far_r2(float y) { return rox_far_coefs(y).r2; }

extern "C" void rox_host_re_w_core(const float* x, const float* y, float* out, int64_t n) {
  for (int64_t i = 0; i < n; i++) out[i] = rox_re_w_core(&rox_daw_taylor[0][0], x[i], y[i]);
}

// the Voigt kernel's slow-zone forms, one point at a time
extern "C" void rox_host_core_zone(const float* x, const float* y, float* out, int64_t n) {
  for (int64_t i = 0; i < n; i++) {
    const float y2 = y[i] * y[i], x2 = x[i] * x[i];
    const bool small = y[i] < ROX_Y_CORE;
    float c[16];
    const int row = rox_core_row(y[i]);
    for (int k = 0; k < 16; k++) {
      const float* r = rox_core_r[k];
      c[k] = small ? rox_core_coef_r(y2, r[0], r[1], r[2], r[3]) : rox_core_coef(row, rox_core_arg(row, y[i]), k);
    }
    const int np = y[i] < 1.0f ? 7 : 5;
    const float U = x2 * (1.0f / (y2 + ROX_CORE_KAPPA));
    float a = c[np], d = c[8 + np];
    for (int k = np - 1; k >= 0; k--) a = fmaf(a, U, c[k]);
    for (int k = np - 1; k >= 0; k--) d = fmaf(d, U, c[8 + k]);
    const float r = a * rox_rcp(fmaf(d, U, 1.0f));
    if (small) {
      const float u2 = x2 * (4.0f * y2);
      const float g = fmaf(fmaf(fmaf(u2, ROX_COS_C6, ROX_COS_C4), u2, -0.5f), u2, 1.0f);
      out[i] = fmaf(rox_exp2(fmaf(x2, -ROX_LOG2E_F, y2 * ROX_LOG2E_F)), g, y[i] * r);
    } else {
      out[i] = r;
    }
  }
}

// the pair form of the line strength: hi, lo, exponent (e = INT32_MIN where it declines), and the
// rounded value with a flag for "certain"
extern "C" void rox_host_strength_df(int hitran, double c2_dT, double q_fac, double c2_T, double c2_Tref, const double* nu0,
                                     const float* s_or_a, const float* g_up, const float* e_lower, float* hi, float* lo,
                                     int32_t* ex, float* rounded, uint8_t* certain, int64_t n) {
  const rox_df_consts k = rox_df_make_consts(hitran, c2_dT, q_fac, c2_T, c2_Tref);
  rox_df tab[32];
  for (int j = 0; j < 32; j++) tab[j] = rox_df_split(exp2(j / 32.0));
  for (int64_t i = 0; i < n; i++) {
    rox_df s;
    int e;
    const bool ok = rox_df_strength(k, tab, nu0[i], s_or_a[i], hitran ? 1.0f : g_up[i], e_lower[i], &s, &e);
    hi[i] = ok ? s.h : 0.0f;
    lo[i] = ok ? s.l : 0.0f;
    ex[i] = ok ? e : INT32_MIN;
    certain[i] = ok && rox_df_round(s, e, &rounded[i]);
  }
}

// the rounding alone: h + l, scaled by 2^e
extern "C" void rox_host_df_round(const float* h, const float* l, const int32_t* e, float* rounded, uint8_t* certain,
                                  int64_t n) {
  for (int64_t i = 0; i < n; i++) {
    rounded[i] = 0.0f;
    certain[i] = rox_df_round({h[i], l[i]}, e[i], &rounded[i]);
  }
}
