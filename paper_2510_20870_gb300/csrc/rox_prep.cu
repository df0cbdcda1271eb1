// The per-line passes ahead of the Voigt launch on a uniform grid, in two kernels: what needs only
// the list (k_prep_lines: a3 windows, a1 strengths and their maxima) and what needs the maxima or
// the neighbouring line's window (k_prep_scaled: scaled strengths, a3 span ranges, and for
// one (P,T) point, on nodes up to ROX_PRE_POINTS of them, the Voigt kernel's per-line constants). pyROX paper, "Compute line-strengths and
// -widths" and "Combine and save".
//
// Separate kernels (windows, strengths, scaling, span ranges, constants) read the line centres and
// the records between them twice and cost five launches, each of about 2.3 us on a list of 1e4 lines,
// where a call takes some 50; the fused ones are bound by their bytes on long lists.
#include "rox_internal.cuh"
#include "rox_lines.cuh"
#include "rox_strength.cuh"
#include "rox_windows.cuh"

namespace {

// NT: temperatures that the argument block holds (8 or ROX_MAX_PT: the large block alone is 28 KB)
template <int NT>
struct PrepTemps {
  int n;
  StrengthConsts k[NT];
};

template <int NT>
__global__ void k_prep_lines(const rox_lines L, const RoxWindows W, const __grid_constant__ PrepTemps<NT> ts,
                             double* S_T, RoxWsHeader* hdr, float4* geo) {
  const long long stride = (long long)gridDim.x * blockDim.x;
  const long long i0 = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  unsigned long long ev = 0;
  for (int t = 0; t < ts.n; t++) {
    unsigned long long mx = 0;
    for (long long i = i0; i < L.n; i += stride) {
      const double nu0 = L.nu0[i];
      if (t == 0) {
        if (i > 0 && L.nu0[i - 1] > nu0) hdr->status = ROX_EUNSORTED;
        const LineWindow w = line_window(W, nu0);
        if (w.jh >= w.jl) ev += (unsigned)(w.jh - w.jl + 1);
        geo[i] = w.geo;
      }
      const float g = L.convention == ROX_EXOMOL ? L.g_up[i] : 1.0f;
      const double s = line_strength_fast(ts.k[t], nu0, L.s_or_a[i], g, L.e_lower[i]);
      S_T[(long long)t * L.n + i] = s;
      mx = max_bits(mx, s);
    }
    store_max(mx, &hdr->smax_bits[t]);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) ev += __shfl_xor_sync(0xffffffffu, ev, o);
  if ((threadIdx.x & 31) == 0 && ev) atomicAdd(&hdr->evals_lines, ev);
}

// S * 2^-e per temperature (e the exponent of the temperature's largest S), so that the Voigt kernel
// works in FP32 well inside its range whatever the line strengths are.
// Span t meets line i iff jhi_i >= 256 t and jlo_i <= 256 t + 255, both non-decreasing along the list:
// each line writes the boundaries between its predecessor's span count and its own (the sorted-order
// form of a histogram prefix sum).
template <bool PRE>
__global__ void k_prep_scaled(const RoxListDev L, const RoxJobDev J, long long n, int n_temps,
                              const double* __restrict__ S_T, const unsigned long long* __restrict__ smax_bits, float* S32,
                              const float4* __restrict__ geo, int n_spans, long long* lo_out, long long* hi_out,
                              float4* rec) {
  const long long stride = (long long)gridDim.x * blockDim.x;
  const long long i0 = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const bool nodes = L.node_d != nullptr;
  const float margin_cm = nodes ? 0.f : fast_margin(L.dnu_f);
  for (int t = 0; t < n_temps; t++) {
    const double smax = __longlong_as_double((long long)smax_bits[t]);
    const double sc = ldexp(1.0, smax > 0.0 ? -ilogb(smax) : 0);
    for (long long i = i0; i <= n; i += stride) {
      if (t == 0) {
        int ch0 = 0, cl0 = 0, ch = n_spans, cl = n_spans;
        float4 g = make_float4(0.f, 0.f, 0.f, 0.f);
        if (lo_out && i > 0) {
          const float4 p = geo[i - 1];
          ch0 = min((__float_as_int(p.w) + ROX_SPAN) / ROX_SPAN, n_spans);     // jhi = -1: 0
          cl0 = min(__float_as_int(p.z) / ROX_SPAN, n_spans);
        }
        if (i < n) {
          g = geo[i];
          ch = min((__float_as_int(g.w) + ROX_SPAN) / ROX_SPAN, n_spans);
          cl = min(__float_as_int(g.z) / ROX_SPAN, n_spans);
        }
        if (lo_out) {
          for (int s = ch0; s < ch; s++) lo_out[s] = i;
          for (int s = cl0; s < cl; s++) hi_out[s] = i;
        }
        if (i == n) continue;
        const float S = (float)(S_T[i] * sc);
        if constexpr (PRE) {
          const float gref = load_width(L.gamma_ref, L.width_f16, i), nt = load_width(L.n_t, L.width_f16, i);
          const LineK k = line_consts<false>(nodes ? g.x : L.nu_min_f + fmaf(g.x, L.dnu_f, g.y), S, gref, nt, J, margin_cm);
          rec[3 * i] = make_float4(k.A, k.B, k.P, k.Q);
          rec[3 * i + 1] = make_float4(k.tz, k.iG, k.y, k.pc);
          if (nodes) {      // the zone's nodes and the spans' widths differ: half-width and distance at width 0
            rec[3 * i + 2] = make_float4(k.zc, k.hz, 0.f, smooth_dmin(k.A, k.B, 0.f));
          } else {
            int zlo, zhi;
            zone_bounds(g, k.hz, L.inv_dnu_f, zlo, zhi);
            rec[3 * i + 2] = make_float4(k.zc, __int_as_float(zlo), __int_as_float(zhi),
                                         smooth_dmin(k.A, k.B, 0.5f * (ROX_SPAN - 1) * L.dnu_f));
          }
        } else {
          S32[i] = S;
        }
      } else if (i < n) {
        S32[(long long)t * n + i] = (float)(S_T[(long long)t * n + i] * sc);
      }
    }
  }
}

int grid_for(long long n) {
  const long long b = (n + 255) / 256;
  return (int)(b < 152 * 16 ? (b < 1 ? 1 : b) : 152 * 16);
}

template <int NT>
cudaError_t prep_lines(const rox_lines* L, const rox_grid* g, double cutoff, int n_temps, const double* temps,
                       const double* q_of_temp, double Q_ref, double* S_T, RoxWsHeader* hdr, float4* geo, cudaStream_t s) {
  PrepTemps<NT> ts;
  ts.n = n_temps;
  for (int t = 0; t < n_temps; t++) ts.k[t] = make_consts(L->convention, temps[t], q_of_temp[t], Q_ref);
  k_prep_lines<NT><<<grid_for(L->n), 256, 0, s>>>(*L, rox_windows(g, cutoff), ts, S_T, hdr, geo);
  return cudaGetLastError();
}

}  // namespace

// windows, strengths S_T[t][i] at every temperature and their maxima, evaluation count and order check
cudaError_t rox_launch_prep_lines(const rox_lines* L, const rox_grid* g, double cutoff, int n_temps, const double* temps,
                                  const double* q_of_temp, double Q_ref, double* S_T, RoxWsHeader* hdr, float4* geo,
                                  cudaStream_t s) {
  if (n_temps <= 8) return prep_lines<8>(L, g, cutoff, n_temps, temps, q_of_temp, Q_ref, S_T, hdr, geo, s);
  return prep_lines<ROX_MAX_PT>(L, g, cutoff, n_temps, temps, q_of_temp, Q_ref, S_T, hdr, geo, s);
}

// scaled strengths and span ranges (lo != NULL) of n lines; with rec, the constants of the one job J in
// place of its scaled strengths
cudaError_t rox_launch_prep_scaled(const RoxListDev& L, const RoxJobDev& J, long long n, int n_temps, const double* S_T,
                                   const unsigned long long* smax_bits, float* S32, const float4* geo, long long n_spans,
                                   long long* lo, long long* hi, float4* rec, cudaStream_t s) {
  const int b = grid_for(n + 1);
  if (rec) k_prep_scaled<true><<<b, 256, 0, s>>>(L, J, n, n_temps, S_T, smax_bits, S32, geo, (int)n_spans, lo, hi, rec);
  else k_prep_scaled<false><<<b, 256, 0, s>>>(L, J, n, n_temps, S_T, smax_bits, S32, geo, (int)n_spans, lo, hi, rec);
  return cudaGetLastError();
}
