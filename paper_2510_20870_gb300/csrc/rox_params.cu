// a1 / a2: per-line strength S(T) and widths gamma_G, gamma_L.
// pyROX paper, "Functionality of pyROX" -- "Compute line-strengths and -widths": the
// strength and broadening widths of every transition at the user's pressure and
// temperature. Each thread reads one line's SoA entries (coalesced) and writes its outputs.
// The strength exists in two forms: the full FP64 one (line_strength), and for the
// cross-section launches a reduced one (line_strength_fast) without FP64 arithmetic, its Boltzmann
// exponent a pair of floats. This GPU's FP64 rate, not the bytes, bounds the full form.
#include <algorithm>
#include <cuda_fp16.h>
#include "rox_internal.cuh"
#include "rox_lines.cuh"      // load_width
#include "rox_strength.cuh"
#include "rox_strength_df.h"

namespace {

// S(T) rounded to FP32: by pairs of floats where their rounding is certain (all but one line in a
// thousand), by the FP64 form otherwise, so the same bits as from the FP64 form alone. That one was
// bound by FP64 issue: 1.03 ms for 1e7 lines against 0.109 ms here; the bytes take 0.04 ms.
__global__ void k_strengths(rox_lines L, StrengthConsts k, rox_df_consts kd, float* S_out) {
  __shared__ rox_df tab[32];
  if (threadIdx.x < 32) tab[threadIdx.x] = rox_df_split(exp2((double)threadIdx.x / 32.0));
  __syncthreads();
  long long stride = (long long)gridDim.x * blockDim.x;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < L.n; i += stride) {
    const float g = (L.convention == ROX_EXOMOL) ? L.g_up[i] : 1.0f;
    const double nu0 = L.nu0[i];
    const float sa = L.s_or_a[i], el = L.e_lower[i];
    rox_df s;
    int e;
    float out;
    if (!rox_df_strength(kd, tab, nu0, sa, g, el, &s, &e) || !rox_df_round(s, e, &out))
      out = (float)line_strength(k, nu0, (double)sa, (double)g, (double)el);
    S_out[i] = out;
  }
}

// the reduced form alone, in double (rox_line_strengths_reduced: what the cross-section launches use)
__global__ void k_strengths_reduced(rox_lines L, StrengthConsts k, double* S_out) {
  long long stride = (long long)gridDim.x * blockDim.x;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < L.n; i += stride) {
    const float g = (L.convention == ROX_EXOMOL) ? L.g_up[i] : 1.0f;
    S_out[i] = line_strength_fast(k, L.nu0[i], L.s_or_a[i], g, L.e_lower[i]);
  }
}

__global__ void k_widths(rox_lines L, double gG_fac, float l2_ratio, float p_fac,
                         float* gG_out, float* gL_out) {
  long long stride = (long long)gridDim.x * blockDim.x;
  int f16 = L.width_dtype == ROX_WIDTH_F16;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < L.n; i += stride) {
    gG_out[i] = (float)(L.nu0[i] * gG_fac);
    float gref = load_width(L.gamma_ref, f16, i);
    float nt = load_width(L.n_t, f16, i);
    gL_out[i] = gref * exp2f(nt * l2_ratio) * p_fac;
  }
}

// S(T) for up to ROX_MAX_PT distinct temperatures in one launch, one sweep over the lines
// per temperature (FAST: the reduced form, bound by its bytes; else FP64 issue sets the
// cost); the per-temperature maximum (needed to
// scale S into FP32 range inside the Voigt kernel) is reduced per warp and combined with
// an atomic max on the (non-negative) double bit pattern, which is order-independent.
struct TempSet {
  int n;
  StrengthConsts k[ROX_MAX_PT];
};

template <bool FAST>
__global__ void k_strengths_multi(rox_lines L, TempSet ts,
                                  double* S_T, unsigned long long* smax_bits) {
  long long stride = (long long)gridDim.x * blockDim.x;
  for (int t = 0; t < ts.n; t++) {
    unsigned long long mx = 0;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < L.n; i += stride) {
      const float g = (L.convention == ROX_EXOMOL) ? L.g_up[i] : 1.0f;
      const double s = FAST ? line_strength_fast(ts.k[t], L.nu0[i], L.s_or_a[i], g, L.e_lower[i])
                            : line_strength(ts.k[t], L.nu0[i], (double)L.s_or_a[i], (double)g, (double)L.e_lower[i]);
      S_T[(long long)t * L.n + i] = s;
      mx = max_bits(mx, s);
    }
    store_max(mx, &smax_bits[t]);
  }
}

// S * 2^-e per temperature, e the exponent of the largest strength at that temperature,
// so the Voigt kernel works in FP32 well inside its range whatever the line strengths are: lines outside
// the selection's bins, or below rel times their bin's largest S at that temperature (the product rounded
// once in double precision), get -0.0, which the Voigt kernel tells apart from a kept strength that rounds
// to +0.0 in FP32.
__global__ void k_scale_strengths(const double* __restrict__ S_T, long long n, int n_temps,
                                  const unsigned long long* __restrict__ smax_bits, float* S32,
                                  const int32_t* __restrict__ bin, const unsigned long long* __restrict__ binmax_bits,
                                  long long n_bins, double rel) {
  long long stride = (long long)gridDim.x * blockDim.x;
  for (int t = 0; t < n_temps; t++) {
    double smax = __longlong_as_double((long long)smax_bits[t]);
    double sc = ldexp(1.0, smax > 0.0 ? -ilogb(smax) : 0);
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
      const double S = S_T[(long long)t * n + i];
      const int b = bin[i];
      const bool keep =
          b >= 0 && S >= __dmul_rn(rel, __longlong_as_double((long long)binmax_bits[(long long)t * n_bins + b]));
      S32[(long long)t * n + i] = keep ? (float)(S * sc) : -0.0f;   // -0: dropped (+0: kept, below FP32)
    }
  }
}

// ---- a2 broadening descriptions: sum_b vmr_b gamma_b (296/T)^n_b of line i, l2 = log2(296/T)
__device__ __forceinline__ float broad_sum(const RoxBroadDev& B, long long i, float l2) {
  long long j = 0;
  if (B.j_lower) {
    j = B.j_lower[i];
    j = j < 0 ? 0 : (j >= B.tab_len ? B.tab_len - 1 : j);
  }
  float g = 0.0f;
  for (int b = 0; b < B.n_b; b++) {
    float gb, nb;
    if (B.tab_gamma[b]) {
      gb = B.tab_gamma[b][j];
      nb = B.tab_n[b][j];
    } else {
      gb = load_width(B.gamma[b], B.f16, i);
      nb = load_width(B.n[b], B.f16, i);
    }
    g = fmaf(B.vmr[b] * gb, exp2f(nb * l2), g);
  }
  return g;
}
#define ROX_INV_4PI_C 2.6544187294380724e-12f   // 1 / (4 pi c), c in cm/s

struct BroadTemps {
  int32_t n;
  float l2[ROX_MAX_PT];
};

// per distinct temperature the broadeners' sum of every line (G[t][i]); natural widths once
__global__ void k_broad_T(RoxBroadDev B, const float* __restrict__ a_coef, long long n, BroadTemps ts, float* G,
                          float* gN) {
  long long stride = (long long)gridDim.x * blockDim.x;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
    for (int t = 0; t < ts.n; t++) G[(long long)t * n + i] = broad_sum(B, i, ts.l2[t]);
    if (gN) gN[i] = a_coef[i] * ROX_INV_4PI_C;
  }
}

__global__ void k_lorentz_out(RoxBroadDev B, const float* __restrict__ a_coef, long long n, float l2, float p_fac,
                              float* out) {
  long long stride = (long long)gridDim.x * blockDim.x;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride)
    out[i] = fmaf(broad_sum(B, i, l2), p_fac, B.natural ? a_coef[i] * ROX_INV_4PI_C : 0.0f);
}

// Main-contributor selection, bin of every line: floor((nu0 - origin) / width) with the
// subtraction and the division each rounded once in double precision; -1 outside [0, n_bins). An FP64
// division is some twenty operations at two per clock per SM, so the quotient is a product with the
// reciprocal in units of 2^-21 bins (below 2^31 bins, where it is off by a few units at most), and the division itself
// decides only within four units of a bin's edge.
#define ROX_BIN_BITS 21
__global__ void k_line_bins(const double* __restrict__ nu0, long long n, double origin, double width, double scale,
                            long long n_bins, int32_t* bin) {
  long long stride = (long long)gridDim.x * blockDim.x;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
    const double d = __dsub_rn(nu0[i], origin);
    const long long u = __double2ll_rd(d * scale);             // saturates; a NaN centre: lowest value
    long long b = u >> ROX_BIN_BITS;
    const long long f = u & ((1LL << ROX_BIN_BITS) - 1);
    if (f < 4 || f > (1LL << ROX_BIN_BITS) - 5) {
      const double q = floor(__ddiv_rn(d, width));
      b = q >= 0.0 && q < (double)n_bins ? (long long)q : -1;
    }
    bin[i] = b >= 0 && b < n_bins ? (int32_t)b : -1;
  }
}

// Largest S per temperature and bin (as double bits; S >= 0, so the bit patterns order like
// the values). The list is sorted by nu0, so each bin is a run of lines: every thread folds
// a run of ROX_BIN_RUN consecutive lines and issues one atomic max per bin it meets.
#define ROX_BIN_RUN 16
__global__ void k_bin_max(const int32_t* __restrict__ bin, const double* __restrict__ S_T, long long n, int n_temps,
                          long long n_bins, unsigned long long* binmax_bits) {
  const long long runs = (n + ROX_BIN_RUN - 1) / ROX_BIN_RUN;
  long long stride = (long long)gridDim.x * blockDim.x;
  for (int t = 0; t < n_temps; t++) {
    const double* S = S_T + (long long)t * n;
    unsigned long long* bm = binmax_bits + (long long)t * n_bins;
    for (long long r = (long long)blockIdx.x * blockDim.x + threadIdx.x; r < runs; r += stride) {
      const long long i0 = r * ROX_BIN_RUN, i1 = min(n, i0 + ROX_BIN_RUN);
      int cur = -1;
      double mx = 0.0;
      for (long long i = i0; i < i1; i++) {
        const int b = bin[i];
        if (b != cur) {
          if (cur >= 0) atomicMax(&bm[cur], (unsigned long long)__double_as_longlong(mx));
          cur = b;
          mx = S[i];
        } else {
          mx = fmax(mx, S[i]);
        }
      }
      if (cur >= 0) atomicMax(&bm[cur], (unsigned long long)__double_as_longlong(mx));
    }
  }
}

// Selection on reduced-form strengths (relative error below 5e-7, see line_strength_fast):
// every decision is taken as on the full FP64 strengths. A line whose reduced value is within
// ROX_SEL_EPS of its bin's reduced maximum may hold the exact maximum: its FP64 strength
// replaces the reduced one in S_T and the exact bin maxima are taken over those lines
// (k_bin_candidates lists them, k_bin_max_fix treats the list: about two in a bin, and one of them
// among 32 lines would have the whole warp wait for its FP64 exponentials). A line within
// ROX_SEL_EPS of its threshold rel * (exact maximum) is decided on its FP64 strength; any other line
// lies on the same side of the threshold whichever form is used (k_select_scale).
// Strengths are compared as integers that order like their values (strength_key):
// ROX_SEL_BITS is at least a relative difference of ROX_SEL_EPS. With FP64 comparisons and
// products, and the candidates' strengths taken where they lie, bins, maxima and decisions took 0.95 ms
// for 1e7 lines, here 0.42 ms.
#define ROX_SEL_EPS 1e-5
#define ROX_SEL_BITS 90071992548LL     // 1e-5 2^53: one bit is a relative 2^-53 to 2^-52
__device__ __forceinline__ long long strength_key(double S) {   // -0 and 0: 0
  const long long b = __double_as_longlong(S);
  return b >= 0 ? b : (long long)(0x8000000000000000ULL - (unsigned long long)b);
}
#define ROX_KEY_INF 0x7ff0000000000000LL   // NaN lies above it (or below its negative)
__global__ void k_bin_candidates(const int32_t* __restrict__ bin, const double* __restrict__ S_T, long long n, int n_temps,
                                 long long n_bins, const unsigned long long* __restrict__ binmax_fast, int32_t* list,
                                 long long* count) {
  long long stride = (long long)gridDim.x * blockDim.x;
  const int lane = threadIdx.x & 31;
  const long long rounds = (n + stride - 1) / stride;          // whole warps to the end
  for (int t = 0; t < n_temps; t++) {
    long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    for (long long r = 0; r < rounds; r++, i += stride) {
      const int b = i < n ? bin[i] : -1;
      bool cand = false;
      if (b >= 0) {
        const long long sb = strength_key(S_T[(long long)t * n + i]);
        cand = sb >= strength_key(__longlong_as_double((long long)binmax_fast[(long long)t * n_bins + b])) - ROX_SEL_BITS && sb <= ROX_KEY_INF;
      }
      const unsigned m = __ballot_sync(0xffffffffu, cand);
      if (m == 0) continue;
      long long base = 0;
      if (lane == 0) base = (long long)atomicAdd((unsigned long long*)&count[t], (unsigned long long)__popc(m));
      base = __shfl_sync(0xffffffffu, base, 0);
      if (cand) list[(long long)t * n + base + __popc(m & ((1u << lane) - 1u))] = (int32_t)i;
    }
  }
}
__global__ void k_bin_max_fix(const rox_lines L, const __grid_constant__ TempSet ts, const int32_t* __restrict__ bin,
                              double* S_T, long long n_bins, const int32_t* __restrict__ list,
                              const long long* __restrict__ count, unsigned long long* binmax_exact) {
  const long long stride = (long long)gridDim.x * blockDim.x;
  const int t = blockIdx.y;
  const long long m = count[t];
  for (long long j = (long long)blockIdx.x * blockDim.x + threadIdx.x; j < m; j += stride) {
    const long long i = list[(long long)t * L.n + j];
    const double g = (L.convention == ROX_EXOMOL) ? (double)L.g_up[i] : 1.0;
    const double sx = line_strength(ts.k[t], L.nu0[i], (double)L.s_or_a[i], g, (double)L.e_lower[i]);
    S_T[(long long)t * L.n + i] = sx;
    atomicMax(&binmax_exact[(long long)t * n_bins + bin[i]], (unsigned long long)__double_as_longlong(sx));
  }
}

// thresholds rel * (exact maximum) of every temperature and bin, in place of the reduced maxima
__global__ void k_bin_thresholds(const unsigned long long* __restrict__ binmax_exact, long long total, double rel, double* thr) {
  long long stride = (long long)gridDim.x * blockDim.x;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += stride)
    thr[i] = __dmul_rn(rel, __longlong_as_double((long long)binmax_exact[i]));
}

__global__ void k_select_scale(const rox_lines L, const __grid_constant__ TempSet ts, const double* __restrict__ S_T,
                               const unsigned long long* __restrict__ smax_bits, const int32_t* __restrict__ bin,
                               const double* __restrict__ thr_T, long long n_bins, float* S32) {
  long long stride = (long long)gridDim.x * blockDim.x;
  for (int t = 0; t < ts.n; t++) {
    const double smax = __longlong_as_double((long long)smax_bits[t]);
    const int e = smax > 0.0 ? ilogb(smax) : 0;
    const double sc = ldexp(1.0, -e);
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < L.n; i += stride) {
      const int b = bin[i];
      float out = -0.0f;               // -0: dropped (+0: kept, below FP32)
      if (b >= 0) {
        double S = S_T[(long long)t * L.n + i];
        const long long tb = strength_key(thr_T[(long long)t * n_bins + b]);
        long long sb = strength_key(S);
        if (llabs(sb - tb) <= ROX_SEL_BITS) {   // near the threshold: the FP64 form decides
          const double g = (L.convention == ROX_EXOMOL) ? (double)L.g_up[i] : 1.0;
          S = line_strength(ts.k[t], L.nu0[i], (double)L.s_or_a[i], g, (double)L.e_lower[i]);
          sb = strength_key(S);
        }
        if (sb >= tb && sb <= ROX_KEY_INF) {
          // S 2^-e: an integer subtraction from the exponent while both are normal
          const int x = (int)(sb >> 52);
          out = x > 0 && x < 2047 && x - e > 0 && x - e < 2047 ? (float)__longlong_as_double(sb - (long long)e * (1LL << 52)) : (float)(S * sc);
        }
      }
      S32[(long long)t * L.n + i] = out;
    }
  }
}

// keep flags of the first temperature: the same test as k_scale_strengths
__global__ void k_keep_flags(const double* __restrict__ S_T, const int32_t* __restrict__ bin,
                             const unsigned long long* __restrict__ binmax_bits, long long n, double rel,
                             uint8_t* keep) {
  long long stride = (long long)gridDim.x * blockDim.x;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
    const int b = bin[i];
    keep[i] = b >= 0 && S_T[i] >= __dmul_rn(rel, __longlong_as_double((long long)binmax_bits[b]));
  }
}

// Per-job strengths (rox_xsec_jobs): each job's line range at its own temperature, the
// per-job maximum, then the job's FP32 scaled copy (second kernel, after the maximum is known).
__global__ void k_strengths_jobs(const __grid_constant__ RoxStrengthJobs J) {
  long long stride = (long long)gridDim.x * blockDim.x;
  for (int q = 0; q < J.n_jobs; q++) {
    const RoxStrengthJob& jb = J.job[q];
    const RoxStrengthList& L = J.list[jb.list];
    StrengthConsts k;
    k.convention = L.convention;
    k.inv_T = jb.inv_T;
    k.q_ratio = jb.q_ratio;
    k.c2_dT = jb.c2_dT;
    set_reduced(&k);
    unsigned long long mx = 0;
    for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < jb.count; t += stride) {
      const long long i = jb.l0 + t;
      const float g = (L.convention == ROX_EXOMOL) ? L.g_up[i] : 1.0f;
      const double sv = line_strength_fast(k, L.nu0[i], L.s_or_a[i], g, L.e_lower[i]);
      jb.S64[t] = sv;
      mx = max_bits(mx, sv);
    }
    store_max(mx, jb.smax_bits);
  }
}

__global__ void k_scale_jobs(const __grid_constant__ RoxStrengthJobs J) {
  long long stride = (long long)gridDim.x * blockDim.x;
  for (int q = 0; q < J.n_jobs; q++) {
    const RoxStrengthJob& jb = J.job[q];
    const double smax = __longlong_as_double((long long)*jb.smax_bits);
    const double sc = ldexp(1.0, smax > 0.0 ? -ilogb(smax) : 0);
    for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < jb.count; t += stride)
      jb.S32[t] = (float)(jb.S64[t] * sc);
  }
}

int grid_for(long long n) {
  long long b = (n + 255) / 256;
  return (int)(b < 152 * 16 ? (b < 1 ? 1 : b) : 152 * 16);
}

}  // namespace

cudaError_t rox_launch_strengths(const rox_lines* L, double T, double Q_T, double Q_ref,
                                 float* S_out, cudaStream_t s) {
  const StrengthConsts k = make_consts(L->convention, T, Q_T, Q_ref);
  const int hitran = L->convention == ROX_HITRAN;
  const rox_df_consts kd = rox_df_make_consts(hitran, k.c2_dT, hitran ? k.q_ratio : k.q_ratio / (8.0 * ROX_PI * ROX_C_CM),
                                              ROX_C2 * k.inv_T, ROX_C2 / ROX_T_REF);
  k_strengths<<<grid_for(L->n), 256, 0, s>>>(*L, k, kd, S_out);
  return cudaGetLastError();
}

cudaError_t rox_launch_strengths_reduced(const rox_lines* L, double T, double Q_T, double Q_ref, double* S_out,
                                         cudaStream_t s) {
  k_strengths_reduced<<<grid_for(L->n), 256, 0, s>>>(*L, make_consts(L->convention, T, Q_T, Q_ref), S_out);
  return cudaGetLastError();
}

cudaError_t rox_launch_widths(const rox_lines* L, double mass_amu, double P_bar, double T,
                              float* gG, float* gL, cudaStream_t s) {
  double gG_fac = sqrt(2.0 * ROX_KB * T / (mass_amu * ROX_AMU)) / ROX_C_M;
  float l2 = (float)log2(ROX_T_REF / T);
  float pf = (float)(P_bar / ROX_P_REF);
  k_widths<<<grid_for(L->n), 256, 0, s>>>(*L, gG_fac, l2, pf, gG, gL);
  return cudaGetLastError();
}

cudaError_t rox_launch_strengths_multi(const rox_lines* L, int n_temps, const double* temps,
                                       const double* q_of_temp, double Q_ref, double* S_T,
                                       unsigned long long* smax_bits, bool exact, cudaStream_t s) {
  TempSet ts;
  ts.n = n_temps;
  for (int t = 0; t < n_temps; t++) ts.k[t] = make_consts(L->convention, temps[t], q_of_temp[t], Q_ref);
  if (exact)
    k_strengths_multi<false><<<grid_for(L->n), 256, 0, s>>>(*L, ts, S_T, smax_bits);
  else
    k_strengths_multi<true><<<grid_for(L->n), 256, 0, s>>>(*L, ts, S_T, smax_bits);
  return cudaGetLastError();
}

void rox_fill_strength_consts(int convention, double T, double Q_T, double Q_ref, RoxStrengthJob* jb) {
  StrengthConsts k = make_consts(convention, T, Q_T, Q_ref);
  jb->inv_T = k.inv_T;
  jb->q_ratio = k.q_ratio;
  jb->c2_dT = k.c2_dT;
}

cudaError_t rox_launch_strengths_jobs(const RoxStrengthJobs& J, long long max_count, cudaStream_t s) {
  k_strengths_jobs<<<grid_for(max_count), 256, 0, s>>>(J);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  k_scale_jobs<<<grid_for(max_count), 256, 0, s>>>(J);
  return cudaGetLastError();
}

cudaError_t rox_launch_select(const double* nu0, const double* S_T, long long n, int n_temps,
                              const unsigned long long* smax_bits, double origin, double width, long long n_bins,
                              double rel, int32_t* bin, unsigned long long* binmax_bits, float* S32, cudaStream_t s) {
  cudaError_t e = cudaMemsetAsync(binmax_bits, 0, (size_t)n_temps * (size_t)n_bins * 8, s);
  if (e != cudaSuccess) return e;
  k_line_bins<<<grid_for(n), 256, 0, s>>>(nu0, n, origin, width, (double)(1LL << ROX_BIN_BITS) / width, n_bins, bin);
  k_bin_max<<<grid_for((n + ROX_BIN_RUN - 1) / ROX_BIN_RUN), 256, 0, s>>>(bin, S_T, n, n_temps, n_bins, binmax_bits);
  k_scale_strengths<<<grid_for(n), 256, 0, s>>>(S_T, n, n_temps, smax_bits, S32, bin, binmax_bits, n_bins, rel);
  return cudaGetLastError();
}

// Selection for the cross-section launches, on strengths from k_strengths_multi<true> (the
// reduced form): bins, reduced maxima, exact maxima over the candidate lines (list [n_temps][n], count
// [n_temps]: scratch), then the decisions and the scaled FP32 strengths (-0.0 for dropped lines).
cudaError_t rox_launch_select_reduced(const rox_lines* L, int n_temps, const double* temps, const double* q_of_temp,
                                      double Q_ref, double* S_T, const unsigned long long* smax_bits, double origin,
                                      double width, long long n_bins, double rel, int32_t* bin,
                                      unsigned long long* binmax_fast, unsigned long long* binmax_exact, float* S32,
                                      int32_t* list, long long* count, cudaStream_t s) {
  const long long n = L->n;
  cudaError_t e = cudaMemsetAsync(binmax_fast, 0, (size_t)n_temps * (size_t)n_bins * 8, s);
  if (e != cudaSuccess) return e;
  if ((e = cudaMemsetAsync(binmax_exact, 0, (size_t)n_temps * (size_t)n_bins * 8, s)) != cudaSuccess) return e;
  TempSet ts;
  ts.n = n_temps;
  for (int t = 0; t < n_temps; t++) ts.k[t] = make_consts(L->convention, temps[t], q_of_temp[t], Q_ref);
  k_line_bins<<<grid_for(n), 256, 0, s>>>(L->nu0, n, origin, width, (double)(1LL << ROX_BIN_BITS) / width, n_bins, bin);
  k_bin_max<<<grid_for((n + ROX_BIN_RUN - 1) / ROX_BIN_RUN), 256, 0, s>>>(bin, S_T, n, n_temps, n_bins, binmax_fast);
  if ((e = cudaMemsetAsync(count, 0, (size_t)n_temps * 8, s)) != cudaSuccess) return e;
  k_bin_candidates<<<grid_for(n), 256, 0, s>>>(bin, S_T, n, n_temps, n_bins, binmax_fast, list, count);
  // a thread per four lines, two warps a block: a short list's candidates (about two in a bin) spread over
  // the SMs' FP64 units, each some 2 us a strength (3e4 lines, three temperatures: 39.9 us with a thread
  // per 32 lines and the temperatures in turn)
  const dim3 fix((unsigned)std::max(1LL, std::min(152LL * 16, (n / 4 + 63) / 64)), (unsigned)n_temps);
  k_bin_max_fix<<<fix, 64, 0, s>>>(*L, ts, bin, S_T, n_bins, list, count, binmax_exact);
  double* thr = reinterpret_cast<double*>(binmax_fast);
  k_bin_thresholds<<<grid_for(n_temps * n_bins), 256, 0, s>>>(binmax_exact, (long long)n_temps * n_bins, rel, thr);
  k_select_scale<<<grid_for(n), 256, 0, s>>>(*L, ts, S_T, smax_bits, bin, thr, n_bins, S32);
  return cudaGetLastError();
}

cudaError_t rox_launch_broad_T(const RoxBroadDev& B, const float* a_coef, long long n, int n_temps,
                               const double* temps, float* G, float* gN, cudaStream_t s) {
  BroadTemps ts;
  ts.n = n_temps;
  for (int t = 0; t < n_temps; t++) ts.l2[t] = (float)log2(ROX_T_REF / temps[t]);
  k_broad_T<<<grid_for(n), 256, 0, s>>>(B, a_coef, n, ts, G, gN);
  return cudaGetLastError();
}

cudaError_t rox_launch_lorentz_out(const RoxBroadDev& B, const float* a_coef, long long n, double P_bar, double T,
                                   float* out, cudaStream_t s) {
  k_lorentz_out<<<grid_for(n), 256, 0, s>>>(B, a_coef, n, (float)log2(ROX_T_REF / T), (float)(P_bar / ROX_P_REF),
                                            out);
  return cudaGetLastError();
}

cudaError_t rox_launch_keep_flags(const double* S_T, const int32_t* bin, const unsigned long long* binmax_bits,
                                  long long n, double rel, uint8_t* keep, cudaStream_t s) {
  k_keep_flags<<<grid_for(n), 256, 0, s>>>(S_T, bin, binmax_bits, n, rel, keep);
  return cudaGetLastError();
}
