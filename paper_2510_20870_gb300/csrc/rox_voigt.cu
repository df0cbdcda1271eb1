// a4 / a5: Voigt evaluation and accumulation onto the wavenumber grid, for every (P,T).
// pyROX paper, "Compute line profiles" (Voigt = Re of the Faddeeva function, Gandhi et al.
// 2020 Eq. 12) and "Combine and save" (profiles summed into a cross-section per
// temperature-pressure point).
//
// Persistent kernel; the unit of work is one warp and one span of ROX_SPAN consecutive grid
// points at one (P,T) point, taken from an atomic counter by the warp itself, so warps never
// wait for one another. Each lane owns ROX_K points of the span, strided by 32. The lines that reach
// the span form a contiguous range of the nu0-sorted list (precomputed per span). The span is
// written once at the end and every sum has a fixed order, so results are reproducible bit for bit.
//
// A line's profile outside its slow zone is a rational in X = nu - nu0 (rox_re_w_far: per-line
// coefficients of y = gamma_L/gamma_G): S V = (P t + Q)/(t^2 + B), t = X^2 + A; two lines share one
// reciprocal. Far from its poles that function is smooth, so a line is evaluated at every point of
// a span only where it has to be:
//  1. Cells (uniform grids). Lines whose window covers the span, at least four times their cell's
//     half-width plus pole modulus away: k_moments has summed the lines of each cell of 64 grid points
//     into 14 moments of a multipole expansion, evaluated once per cell at the span's 32 Chebyshev
//     points.
//  2. Edge runs. Lines beyond the cells, cut by the window's end inside the span: running sums of 8
//     moments per line, one evaluation per point (edge_batch).
//  3. The rest, in batches of 32, a lane setting up a line. Lines smooth on the span are evaluated
//     at the 32 Chebyshev points (one step a pair in place of ROX_K); lines covering it, with their
//     poles near, at every point, t clamped to the slow zone's boundary; window-edge lines near
//     the span under masks; then, inside the slow zones, the Faddeeva forms minus the boundary
//     value added before (zone_batch, a lane a line; zone_line where zones lie apart).
// The sums at the Chebyshev points go to the span's points by one interpolation per span (error
// 1e-7 of a line's value at the distances admitted: smooth_dmin).
//
// Every form but the slow zones' works per line and span, not per line and point: on the 1e7-line
// ExoMol list the kernel took 16.0 ms with each line at each of its 5,001 points, 3.27 ms so. It is bound
// by instruction issue and, as the code is long, by instruction fetch (4.2 of 9.2 stalled warps
// per issue before the loops were kept short): a form that saves a few instructions with a second
// copy of a loop costs more than it gives.
#include <cuda_fp16.h>
#include "rox_internal.cuh"
#include "rox_lines.cuh"
#include "rox_interp_table.h"   // generated by gen_interp_table.py

namespace {


// Per-line constants of one (P,T) point for the batch in hand. Each line has a slot; slots are
// ordered by class -- lines that are smooth on the span first, then the others whose window covers all
// of it, then the lines cut by a window edge that are not scanned -- and slots 2k, 2k+1 form pair k. The pair tables hold both lines' far-form constants side by side,
// so one 16-byte load brings a field of both; the line table holds what window edges and pass 2
// need per slot. S is scaled by 2^-e (e the exponent of the largest strength at this
// temperature).
struct PairTab {
  float4 ab[16];   // {A0, A1, B0, B1}: far form t = X^2 + A, d = t^2 + B
  float4 pq[16];   // {P0, P1, Q0, Q1}: S V = (P t + Q) / d, P = S Y / pi, Q = P K
  float4 ef[16];   // uniform grid {E0, E1, F0, F1}: X at the lane's first point = (lane + E) dnu + F,
                   // E = (span start) - k0 (exact), F = -f dnu; nodes {ch0, ch1, cl0, cl1}: X = (D.hi - ch) + (D.lo - cl)
  float2 tz[16];   // {t_z0, t_z1}: the far form holds for t >= t_z; pass 1 evaluates it at max(t, t_z)
};
struct LineTab {
  int2 W[32];      // window [jlo, jhi] (grid indices)
  int2 Z[32];      // slow zone [zlo, zhi] (grid indices; nodes: the window)
  float4 z[32];    // {1/gamma_G, y = gamma_L/gamma_G, S/(gamma_G sqrt(pi)), X^2 of the end of the
                   // line's own zone where the precision margin widens it, else huge}
};
// The warp's tables of a batch; before they are written the same memory holds the edge lines' scan.
#define ROX_EDGE_TERMS 8
struct __align__(16) EdgeRec {
  float m[ROX_EDGE_TERMS];   // moments of the edge lines up to this one
  int key;                   // first point (counted from the side the lines come from) that has them
  int pad[3];
};
struct BatchTab {
  union {
    struct {
      PairTab pairs;
      LineTab lines;
    };
    EdgeRec scan[33];        // [0]: the lines before the batch
  };
  __device__ BatchTab() {}
};
// one line's field out of a pair table row: half h (0, 1) of {lo, hi} pairs
__device__ __forceinline__ float row_lo(const float4& v, int h) { return h ? v.y : v.x; }
__device__ __forceinline__ float row_hi(const float4& v, int h) { return h ? v.w : v.z; }

__device__ __forceinline__ void cp_async16(void* smem, const void* gmem) {
  unsigned s = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(s), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async4(void* smem, const void* gmem) {
  unsigned s = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(s), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait0() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }

// Two FP32 values in one 64-bit register pair, for the paired FP32 instructions of sm_100 and
// later (fma.rn.f32x2 / add.rn.f32x2: two IEEE operations, each rounded as the scalar one). A
// paired instruction takes one issue slot for two operations, which leaves issue slots to the
// reciprocal, the clamps and the loads while the FMA pipes stay busy.
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 f2_pack(float lo, float hi) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ void f2_unpack(f32x2 v, float& lo, float& hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ f32x2 f2_fma(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ f32x2 f2_add(f32x2 a, f32x2 b) {
  f32x2 d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}

// v += x with the running compensation c (Kahan) weighted by kw: 1 keeps it, 0 leaves the plain sum
__device__ __forceinline__ void sum_add(float& v, float& c, float x, float kw) {
  const float y = x - c, t = v + y;
  c = ((t - v) - y) * kw;
  v = t;
}

// Far-form constants of pair k, packed for the paired instructions.
struct PairC {
  f32x2 A, B, P, Q;
  float2 T;
  float e0, e1, f0, f1;
};
template <bool CLAMP>
__device__ __forceinline__ PairC pair_consts(const PairTab& P, int k) {
  PairC c;
  const float4 ab = P.ab[k], pq = P.pq[k], ef = P.ef[k];
  c.A = f2_pack(ab.x, ab.y);
  c.B = f2_pack(ab.z, ab.w);
  c.P = f2_pack(pq.x, pq.y);
  c.Q = f2_pack(pq.z, pq.w);
  c.T = CLAMP ? P.tz[k] : make_float2(0.0f, 0.0f);
  c.e0 = ef.x;
  c.e1 = ef.y;
  c.f0 = ef.z;
  c.f1 = ef.w;
  return c;
}

// acc + S0 V0 + S1 V1 for the pair's offsets x0, x1 at one point, the two fractions over one
// reciprocal, n0/d0 + n1/d1 = (n0 d1 + n1 d0)/(d0 d1). CLAMP: t = max(X^2 + A, t_z) per line
// (inside its slow zone a line contributes the far form's value at the zone boundary, which
// pass 2 takes out again). MASK: u0, u1 tell whether the point is in each line's window.
// Paired: X^2 + A, t^2 + B, P t + Q; scalar: 4 FP32 operations and 1 MUFU (+ 2 clamps).
template <bool CLAMP, bool MASK>
__device__ __forceinline__ float pair_add(float x0, float x1, const PairC& c, bool u0, bool u1, float acc) {
  const f32x2 x = f2_pack(x0, x1);
  f32x2 t = f2_fma(x, x, c.A);
  if (CLAMP) {
    float t0, t1;
    f2_unpack(t, t0, t1);
    t = f2_pack(fmaxf(t0, c.T.x), fmaxf(t1, c.T.y));
  }
  float d0, d1, n0, n1;
  f2_unpack(f2_fma(t, t, c.B), d0, d1);
  f2_unpack(f2_fma(t, c.P, c.Q), n0, n1);
  if (MASK) {
    n0 = u0 ? n0 : 0.0f;
    n1 = u1 ? n1 : 0.0f;
  }
  return fmaf(fmaf(n1, d0, n0 * d1), rox_rcp(d0 * d1), acc);
}

// The pair's offsets at this lane's first point (uniform grid): X = (lane + E) dnu + F, with
// lane + E = (span start + lane) - k0 exact, so X is the exact index decomposition rounded once.
template <bool NU>
__device__ __forceinline__ void pair_x0(const PairC& c, float lanef, float dnu_f, float& X0, float& X1) {
  if constexpr (NU) {
    X0 = X1 = 0.0f;
  } else {
    f2_unpack(f2_fma(f2_add(f2_pack(lanef, lanef), f2_pack(c.e0, c.e1)), f2_pack(dnu_f, dnu_f), f2_pack(c.f0, c.f1)),
              X0, X1);
  }
}

// X = nu - nu0 at this lane's point of sub-span m. Uniform grid: X0 + 32 m dnu (one rounding more).
// User-provided nodes: the node's double-float offset from the span's first node, D[32 m] =
// {hi, lo}, minus the line's {ch, cl}; the hi parts cancel exactly near the line, so X keeps
// its relative accuracy.
template <bool NU>
__device__ __forceinline__ float pos(int m, float X0, float ch, float cl, const float2* D, float dnu_f) {
  if constexpr (NU) {
    const float2 d = D[32 * m];
    return (d.x - ch) + (d.y - cl);
  } else {
    return fmaf((float)(32 * m), dnu_f, X0);
  }
}

// Pass 1 for covering pair k: every point of the span, t clamped to each line's zone boundary.
template <bool NU>
__device__ __forceinline__ void cover_pair(const PairTab& P, int k, float lanef, float dnu_f, const float2* D,
                                           float (&acc)[ROX_K]) {
  const PairC c = pair_consts<true>(P, k);
  float X0, X1;
  pair_x0<NU>(c, lanef, dnu_f, X0, X1);
#pragma unroll
  for (int m = 0; m < ROX_K; m++)
    acc[m] = pair_add<true, false>(pos<NU>(m, X0, c.e0, c.f0, D, dnu_f), pos<NU>(m, X1, c.e1, c.f1, D, dnu_f), c,
                                   true, true, acc[m]);
}

// Pass 1 for pair k of lines that are smooth on the span: their sum at this lane's Chebyshev
// point of the span (tau: its position in grid steps, or on nodes in cm^-1, from the span's first
// point). One step in place of ROX_K.
template <bool NU>
__device__ __forceinline__ float smooth_pair(const PairTab& P, int k, float tau, float dnu_f, float nacc) {
  const PairC c = pair_consts<false>(P, k);
  float x0, x1;
  if constexpr (NU) {
    x0 = (tau - c.e0) - c.f0;
    x1 = (tau - c.e1) - c.f1;
  } else {
    pair_x0<NU>(c, tau, dnu_f, x0, x1);
  }
  return pair_add<false, false>(x0, x1, c, true, true, nacc);
}

// Adds to stot (the span's points) the polynomial through the values v at the span's 32 Chebyshev
// points (lane k holds point k). Uniform grid: the cardinal functions are a table; nodes: the
// barycentric quotient, evaluated at each node's position.
template <bool NU>
__device__ __forceinline__ void interp_span(float v, int lane, const float2* D, float half, float* stot) {
  if constexpr (NU) {
    const float inv = half > 0.f ? 1.0f / half : 0.f;
    for (int m = 0; m < ROX_K; m++) {
      const float x = fmaf(D[32 * m].x, inv, -1.0f);
      float num = 0.f, den = 0.f;
#pragma unroll 8
      for (int k = 0; k < ROX_NODES; k++) {
        float d = x - rox_cheb_x[k];
        d = d == 0.f ? 1e-20f : d;
        const float q = rox_cheb_w[k] * rox_rcp(d);
        num = fmaf(q, __shfl_sync(0xffffffffu, v, k), num);
        den += q;
      }
      stot[32 * m + lane] += num / den;
    }
  } else {
    float r[ROX_K];
#pragma unroll
    for (int m = 0; m < ROX_K; m++) r[m] = 0.f;
#pragma unroll 4
    for (int k = 0; k < ROX_NODES; k++) {
      const float vk = __shfl_sync(0xffffffffu, v, k);
#pragma unroll
      for (int m = 0; m < ROX_K; m++) r[m] = fmaf(__ldg(&rox_interp[m][k][lane]), vk, r[m]);
    }
#pragma unroll
    for (int m = 0; m < ROX_K; m++) stot[32 * m + lane] += r[m];
  }
}

// Pass 1 for pair k of which at least one line is cut by a window edge that the edge scan does not
// take: the sub-spans outside both windows are skipped; elsewhere each point takes line i iff it lies
// in the line's window (the exact integer window). Rare on long cutoffs, so the loop is kept short
// rather than fast, and adds into the warp's row zacc.
template <bool NU>
__device__ __forceinline__ void edge_pair(const PairTab& P, const LineTab& L, int k, int Aw, int lane, float lanef,
                                          float dnu_f, const float2* D, float* zacc) {
  const PairC c = pair_consts<true>(P, k);
  const int2 w0 = L.W[2 * k], w1 = L.W[2 * k + 1];
  const int lo0 = w0.x - Aw, hi0 = w0.y - Aw, lo1 = w1.x - Aw, hi1 = w1.y - Aw;
  const int mf = max(0, min(lo0, lo1) >> 5), ml = min(ROX_K - 1, max(hi0, hi1) >> 5);
  float X0, X1;
  pair_x0<NU>(c, lanef, dnu_f, X0, X1);
#pragma unroll 1
  for (int m = mf; m <= ml; m++) {
    const int q = 32 * m + lane;
    zacc[q] = pair_add<true, true>(pos<NU>(m, X0, c.e0, c.f0, D, dnu_f), pos<NU>(m, X1, c.e1, c.f1, D, dnu_f), c,
                                   q >= lo0 && q <= hi0, q >= lo1 && q <= hi1, zacc[q]);
  }
}

// Pass 2 for the line in slot s, whose slow zone meets the span: at exactly the points where
// pass 1 clamped t (t < t_z on the same rounded t, inside the window), the FP32 Faddeeva form of
// the line's y (rox_faddeeva.cuh) replaces the far form's boundary value cf that pass 1 added there:
// + S V - cf. In a zone widened to the precision margin the points beyond the form's own zone (X^2 >= zc) take the far form on an offset rounded once.
// The pass is bound by instruction issue, so a lane takes two points at once in paired FP32
// instructions (two neighbouring points of the uniform grid: 64 points a warp step, one 8-byte
// update of the warp's shared-memory row zacc; on nodes two sub-spans), the polynomials' coefficients
// come from shared memory as ready pairs, and points outside the zone are selected away rather than
// branched over. Within a warp step the lanes touch distinct points.
struct ZoneC {
  float A, B, P, Q, tz, cf, zc;
  f32x2 gU;                    // x2 -> U
  f32x2 ge, ge0, gc, gy, gp;   // Gaussian part (y < 0.1): exponent ge x2 + ge0, (2xy)^2 = gc x2, factor gp; N/D's factor gy
};
__device__ __forceinline__ f32x2 f2_dup(float v) { return f2_pack(v, v); }
__device__ __forceinline__ f32x2 f2_mul(f32x2 a, f32x2 b) {
  f32x2 d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
// N(U)/D(U); cb: the 16 coefficients as pairs
__device__ __forceinline__ f32x2 rat_pair(const ulonglong2* cb, f32x2 U) {
  f32x2 c[16];
#pragma unroll
  for (int i = 0; i < 8; i++) {
    const ulonglong2 v = cb[i];
    c[2 * i] = v.x;
    c[2 * i + 1] = v.y;
  }
  f32x2 n = c[7], d = c[15];
#pragma unroll
  for (int k = 6; k >= 0; k--) {
    n = f2_fma(n, U, c[k]);
    d = f2_fma(d, U, c[8 + k]);
  }
  d = f2_fma(d, U, f2_dup(1.0f));
  float d0, d1;
  f2_unpack(d, d0, d1);
  return f2_mul(n, f2_pack(rox_rcp(d0), rox_rcp(d1)));
}
// S V - cf for the pair of offsets X
__device__ __forceinline__ f32x2 zone_pair(const ZoneC& z, const ulonglong2* cb, f32x2 X) {
  const f32x2 x2 = f2_mul(X, X);
  const f32x2 r = rat_pair(cb, f2_mul(x2, z.gU));
  float e0, e1;
  f2_unpack(f2_fma(x2, z.ge, z.ge0), e0, e1);
  const f32x2 u2 = f2_mul(x2, z.gc);
  f32x2 g = f2_fma(u2, f2_dup(ROX_COS_C6), f2_dup(ROX_COS_C4));
  g = f2_fma(u2, g, f2_dup(-0.5f));
  g = f2_fma(u2, g, f2_dup(1.0f));
  f32x2 v = f2_fma(f2_pack(rox_exp2(e0), rox_exp2(e1)), f2_mul(g, z.gp), f2_dup(-z.cf));
  v = f2_fma(r, z.gy, v);
  if (z.zc < 1e38f) {
    float x0, x1, v0, v1, d0, d1, w0, w1;
    const f32x2 t = f2_add(x2, f2_dup(z.A));
    f2_unpack(x2, x0, x1);
    f2_unpack(v, v0, v1);
    f2_unpack(f2_fma(t, t, f2_dup(z.B)), d0, d1);
    f2_unpack(f2_fma(t, f2_dup(z.P), f2_dup(z.Q)), w0, w1);
    v = f2_pack(x0 < z.zc ? v0 : fmaf(w0, rox_rcp(d0), -z.cf), x1 < z.zc ? v1 : fmaf(w1, rox_rcp(d1), -z.cf));
  }
  return v;
}
template <bool NU>
__device__ __forceinline__ void zone_points(const ZoneC& z, const ulonglong2* cb, float e, float f, int q0, int q1,
                                            int lane, float dnu_f, const float2* D, float* zacc) {
  float t0, t1, v0, v1;
  if constexpr (NU) {
    for (int m = (q0 >> 5) & ~1; m <= q1 >> 5; m += 2) {
      const int q = 32 * m + lane;
      const f32x2 X = f2_pack(pos<NU>(m, 0.f, e, f, D, dnu_f), pos<NU>(m + 1, 0.f, e, f, D, dnu_f));   // exact already
      f2_unpack(f2_fma(X, X, f2_dup(z.A)), t0, t1);
      const bool u0 = t0 < z.tz && q >= q0 && q <= q1, u1 = t1 < z.tz && q + 32 >= q0 && q + 32 <= q1;
      if (!__any_sync(0xffffffffu, u0 || u1)) continue;
      f2_unpack(zone_pair(z, cb, X), v0, v1);
      if (u0) zacc[q] += v0;
      if (u1) zacc[q + 32] += v1;
    }
  } else {
    int q = (q0 & ~1) + 2 * lane;
    float mf = (float)(q & ~31);
    const f32x2 dn = f2_dup(dnu_f), ff = f2_dup(f);
    const float l0 = (float)(q & 31);
    const f32x2 le = f2_add(f2_pack(l0, l0 + 1.0f), f2_dup(e));
    const f32x2 X0 = f2_fma(le, dn, ff);                       // t rounded exactly as pass 1 rounds it
    for (; q <= q1; q += 64, mf += 64.0f) {
      const f32x2 Xm = f2_fma(f2_dup(mf), dn, X0);
      f2_unpack(f2_fma(Xm, Xm, f2_dup(z.A)), t0, t1);
      const f32x2 X = f2_fma(f2_add(le, f2_dup(mf)), dn, ff);  // the offset rounded once
      f2_unpack(zone_pair(z, cb, X), v0, v1);
      float2* p = reinterpret_cast<float2*>(zacc + q);
      float2 s = *p;
      s.x += t0 < z.tz && q >= q0 ? v0 : 0.0f;
      s.y += t1 < z.tz && q < q1 ? v1 : 0.0f;
      *p = s;
    }
  }
}
template <bool NU>
__device__ __forceinline__ void zone_line(const PairTab& P, const LineTab& L, int s, int Aw, int lane, float dnu_f,
                                          const float4& r, const float2* D, f32x2* cbuf, float* zacc) {
  const int2 w = L.W[s], zw = L.Z[s];
  const int lo = max(max(zw.x, w.x) - Aw, 0), hi = min(min(zw.y, w.y) - Aw, ROX_SPAN - 1);
  if (lo > hi) return;
  const int k = s >> 1, h = s & 1;
  const float4 ab = P.ab[k], pq = P.pq[k], ef = P.ef[k];
  const float4 zl = L.z[s];                     // {1/gamma_G, y, S/(gamma_G sqrt(pi)), zc}
  const float y = zl.y, y2 = y * y;
  // the form's coefficients, one a lane, handed round through shared memory
  const int row = rox_core_row(y);
  const float c = y < ROX_Y_CORE ? rox_core_coef_r(y2, r.x, r.y, r.z, r.w)
                                 : rox_core_coef(row, rox_core_arg(row, y), lane & 15);
  __syncwarp();
  if (lane < 16) cbuf[lane] = f2_dup(c);
  __syncwarp();
  ZoneC z;
  z.A = row_lo(ab, h);
  z.B = row_hi(ab, h);
  z.P = row_lo(pq, h);
  z.Q = row_hi(pq, h);
  z.tz = h ? P.tz[k].y : P.tz[k].x;
  z.cf = fmaf(z.tz, z.P, z.Q) * rox_rcp(fmaf(z.tz, z.tz, z.B));
  z.zc = zl.w;
  const float g2 = zl.x * zl.x;
  z.gU = f2_dup(g2 * rox_rcp(y2 + ROX_CORE_KAPPA));
  const bool small = y < ROX_Y_CORE;
  z.ge = f2_dup(small ? -ROX_LOG2E_F * g2 : 0.0f);
  z.ge0 = f2_dup(small ? ROX_LOG2E_F * y2 : 0.0f);
  z.gc = f2_dup(small ? 4.0f * y2 * g2 : 0.0f);
  z.gp = f2_dup(small ? zl.z : 0.0f);
  z.gy = f2_dup(small ? zl.z * y : zl.z);
  zone_points<NU>(z, reinterpret_cast<const ulonglong2*>(cbuf), row_lo(ef, h), row_hi(ef, h), lo, hi, lane, dnu_f, D,
                  zacc);
}


// Points of the common zone per zoned line up to which the batch form is taken. With 8 a table of 40 points
// takes 29.2 ms in place of 27.9, sparse lists up to 5% less; with 32 the table is the same and
// sparse lists take up to 25% longer.
#define ROX_ZONE_DENSE 16
// Pass 2 for all zoned lines of a batch at once, one line a lane: where the lines lie close together
// their zones share most of their points, and the warp walks those points [qa, qb] with every
// lane evaluating its own line (coefficients in registers, computed once for the batch) and a
// warp sum of eight points at a time. Against the line by line form this takes a point's work
// to a thirty-second of 23 instructions per line, where that takes some 70 for 32 points plus 60
// per line (measured: 297 + 62 warp instructions a line on the 1e7-line ExoMol list). on: this
// lane's line is zoned; [q0, q1]: its zone inside its window (span positions).
template <bool NU>
__device__ __forceinline__ void zone_batch(bool on, int q0, int q1, int qa, int qb, bool cut, const LineK& k, float e,
                                           float f, float dnu_f, const float2* Drow, int lane, float* sm, float* zacc) {
  const bool small = k.y < ROX_Y_CORE;
  const float y2 = k.y * k.y;
  float c[16];
#pragma unroll
  for (int i = 0; i < 16; i++)
    c[i] = rox_core_coef_r(y2, rox_core_r[i][0], rox_core_r[i][1], rox_core_r[i][2], rox_core_r[i][3]);
  if (__any_sync(0xffffffffu, on && !small)) {
    const int row = rox_core_row(k.y);
    const float t = rox_core_arg(row, k.y);
#pragma unroll
    for (int i = 0; i < 16; i++) {
      const float v = rox_core_coef(row, t, i);
      c[i] = small ? c[i] : v;
    }
  }
  const float g2 = k.iG * k.iG;
  const f32x2 gU = f2_dup(g2 * rox_rcp(y2 + ROX_CORE_KAPPA));
  // the Gaussian part: none above y = 0.1 (exponent 0, factor 0)
  const f32x2 ge = f2_dup(small ? -ROX_LOG2E_F * g2 : 0.0f), ge0 = f2_dup(small ? ROX_LOG2E_F * y2 : 0.0f);
  const f32x2 gc = f2_dup(small ? 4.0f * y2 * g2 : 0.0f), gp = f2_dup(small ? k.pc : 0.0f);
  const f32x2 gy = f2_dup(small ? k.pc * k.y : k.pc);
  const f32x2 ncf = f2_dup(-fmaf(k.tz, k.P, k.Q) * rox_rcp(fmaf(k.tz, k.tz, k.B)));
  const float zt = on ? k.tz - k.A : -1.0f;                 // the zone: X^2 < t_z - A
  const bool wide = __any_sync(0xffffffffu, on && k.zc < 1e38f);
  const f32x2 ee = f2_dup(e), ff = f2_dup(f), dn = f2_dup(dnu_f), one = f2_dup(1.0f);
  // sum over the lanes, eight points at a time through shared memory: row i holds point q + i of every
  // line; lane l then adds eight lines of row l / 4, conflict-free with rows 36 floats apart
  const float* row = sm + 36 * (lane >> 2) + 8 * (lane & 3);
  for (int q = qa & ~7; q <= qb; q += 8) {
    // two pairs of points a round, not all four: the kernel's code is larger than the instruction
    // caches (fully unrolled, warps spent 46% of their stalls waiting for instructions)
#pragma unroll 2
    for (int i = 0; i < 8; i += 2) {
      f32x2 X;
      if constexpr (NU) {
        const float2 da = Drow[q + i], db = Drow[q + i + 1];
        X = f2_pack((da.x - e) + (da.y - f), (db.x - e) + (db.y - f));
      } else {
        const float qf = (float)(q + i);
        X = f2_fma(f2_add(f2_pack(qf, qf + 1.0f), ee), dn, ff);
      }
      const f32x2 x2 = f2_mul(X, X), U = f2_mul(x2, gU);
      f32x2 n = f2_dup(c[7]), d = f2_dup(c[15]);
#pragma unroll
      for (int j = 6; j >= 0; j--) {
        n = f2_fma(n, U, f2_dup(c[j]));
        d = f2_fma(d, U, f2_dup(c[8 + j]));
      }
      float d0, d1, e0, e1, x0, x1, v0, v1;
      f2_unpack(f2_fma(d, U, one), d0, d1);
      f2_unpack(f2_fma(x2, ge, ge0), e0, e1);
      const f32x2 u2 = f2_mul(x2, gc);
      f32x2 g = f2_fma(u2, f2_dup(ROX_COS_C6), f2_dup(ROX_COS_C4));
      g = f2_fma(u2, g, f2_dup(-0.5f));
      g = f2_fma(u2, g, one);
      f32x2 s = f2_fma(f2_pack(rox_exp2(e0), rox_exp2(e1)), f2_mul(g, gp), ncf);
      s = f2_fma(f2_mul(n, f2_pack(rox_rcp(d0), rox_rcp(d1))), gy, s);
      f2_unpack(s, v0, v1);
      f2_unpack(x2, x0, x1);
      if (wide) {
        float w0, w1, n0, n1, c0, c1;
        const f32x2 t = f2_add(x2, f2_dup(k.A));
        f2_unpack(f2_fma(t, f2_dup(k.P), f2_dup(k.Q)), n0, n1);
        f2_unpack(f2_fma(t, t, f2_dup(k.B)), w0, w1);
        f2_unpack(ncf, c0, c1);
        v0 = x0 < k.zc ? v0 : fmaf(n0, rox_rcp(w0), c0);
        v1 = x1 < k.zc ? v1 : fmaf(n1, rox_rcp(w1), c1);
      }
      v0 = x0 < zt ? v0 : 0.0f;
      v1 = x1 < zt ? v1 : 0.0f;
      if (cut) {
        v0 = q + i >= q0 && q + i <= q1 ? v0 : 0.0f;
        v1 = q + i + 1 >= q0 && q + i + 1 <= q1 ? v1 : 0.0f;
      }
      sm[36 * i + lane] = v0;
      sm[36 * i + 36 + lane] = v1;
    }
    __syncwarp();
    const float4 a = *reinterpret_cast<const float4*>(row), b = *reinterpret_cast<const float4*>(row + 4);
    float r = ((a.x + a.y) + (a.z + a.w)) + ((b.x + b.y) + (b.z + b.w));
    r += __shfl_xor_sync(0xffffffffu, r, 1);
    r += __shfl_xor_sync(0xffffffffu, r, 2);
    if ((lane & 3) == 0) zacc[q + (lane >> 2)] += r;
    __syncwarp();
  }
}

// ---- Window edges. A line whose window ends inside the span reaches only the points on one
// side of its last (or first) point; at a cutoff many spans away its far form is as smooth there as a
// cell's. Sorted by centre, such lines have sorted edges, so point j has the lines up to some i(j):
// the lanes, one line each, form their moments about a common centre (the span's centre minus or
// plus the cutoff), a warp scan turns them into running sums, and each point evaluates the sum
// that belongs to it once. Per line about 8 warp instructions, where evaluating its points
// under a mask took 95. The left lines (edge jhi) run through the list downwards, so that both sides
// count points from the side the lines come from: key = Bw - jhi or jlo - Aw, non-decreasing.
// Centre distances are one cutoff give or take the span's half-width; with (half-width + pole
// modulus) / (cutoff - half-width) at most ROX_EDGE_R, eight terms err by 9 r^8 = 1e-7.
// The sums carried from batch to batch are compensated: a part may have 1e5 and more lines of a side, and
// 3e5 lines of 1e-9 beside one of 1 were dropped whole by a plain sum (2.6e-4 of the value).
#define ROX_EDGE_R 0.1f
#define ROX_CARRY (2 * ROX_EDGE_TERMS)   // floats of a side's running sums and their compensations
// Lines of a side in a general batch from which it is scanned: a scan takes some 250 instructions whatever
// it holds, a masked pair about 100. At cutoffs of two to four spans most batches hold a few such lines
// only (30,000 lines, 300,001 points, 10 points (P,T), cutoff 5 cm^-1: 0.470 ms with every batch scanned,
// 0.43 from 16 lines on); with never a scan, long lists lose (the 3e6-line fixed-resolution grid 4.62 -> 5.1 ms).
#define ROX_EDGE_SCAN 16
// points [k0, k1) of one side: their line's sum from the records rec[0 .. n_rec - 1] (n_rec 33, or 1 to take rec[0])
template <bool NU>
__device__ __forceinline__ void edge_points(const EdgeRec* rec, int n_rec, bool left, int k0, int k1, int lane,
                                            float centre, float inv_cut, float dnu_f, const float2* Drow, float* zacc) {
  for (int k = k0 + lane; k < k1; k += 32) {
    int i = 0;                       // records 1 .. i have key <= k
    if (n_rec > 1) {
#pragma unroll
      for (int st = 16; st > 0; st >>= 1)
        if (rec[i + st].key <= k) i += st;
      if (i == 31 && rec[32].key <= k) i = 32;
    }
    const float4 ra = reinterpret_cast<const float4*>(rec[i].m)[0], rb = reinterpret_cast<const float4*>(rec[i].m)[1];
    const int q = left ? ROX_SPAN - 1 - k : k;
    const float y = ((NU ? Drow[q].x : (float)q * dnu_f) - centre) * inv_cut;
    const float z = rox_rcp(y);
    float f = fmaf(rb.w, z, rb.z);
    f = fmaf(fmaf(fmaf(f, z, rb.y), z, rb.x), z, ra.w);
    f = fmaf(fmaf(fmaf(f, z, ra.z), z, ra.y), z, ra.x);
    zacc[q] += z * z * f;
  }
}
// one batch's lines of one side (mine: this lane's line is one of them, at d = offset of its centre from
// `centre` in cutoffs): kcur is the side's first point without its final sum
template <bool NU>
__device__ __forceinline__ void edge_batch(EdgeRec* rec, float* carry, bool left, bool mine, int key, float d,
                                           const LineK& k, int& kcur, int lane, float centre, float inv_cut,
                                           float dnu_f, const float2* Drow, float* zacc) {
  const float i2 = inv_cut * inv_cut, i4 = i2 * i2;
  const float pu = mine ? k.P * i2 : 0.f, qu = mine ? k.Q * i4 : 0.f, bu = mine ? k.B * i4 : 0.f;
  const float dd = mine ? d : 0.f, e = fmaf(dd, dd, mine ? k.A * i2 : 0.f);
  const float d3 = 4.0f * dd, d2 = -fmaf(d3, dd, 2.0f * e), d1 = d3 * e, d0 = -fmaf(e, e, bu);
  float m[ROX_EDGE_TERMS];
  m[0] = pu;
  m[1] = 2.0f * pu * dd;
  m[2] = fmaf(d3, m[1], fmaf(d2, m[0], fmaf(pu, e, qu)));
  m[3] = fmaf(d3, m[2], fmaf(d2, m[1], d1 * m[0]));
#pragma unroll
  for (int l = 4; l < ROX_EDGE_TERMS; l++) m[l] = fmaf(d3, m[l - 1], fmaf(d2, m[l - 2], fmaf(d1, m[l - 3], d0 * m[l - 4])));
  int kk = mine ? key : -1;
  __syncwarp();                      // the tables of the batch before are no longer read
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int ko = __shfl_up_sync(0xffffffffu, kk, o);
    kk = lane >= o ? max(kk, ko) : kk;
#pragma unroll
    for (int l = 0; l < ROX_EDGE_TERMS; l++) {
      const float t = __shfl_up_sync(0xffffffffu, m[l], o);
      if (lane >= o) m[l] += t;
    }
  }
  const float4 ca = reinterpret_cast<const float4*>(carry)[0], cb = reinterpret_cast<const float4*>(carry)[1];
  const float c[ROX_EDGE_TERMS] = {ca.x, ca.y, ca.z, ca.w, cb.x, cb.y, cb.z, cb.w};
  if (lane == 0) {
    reinterpret_cast<float4*>(rec[0].m)[0] = ca;
    reinterpret_cast<float4*>(rec[0].m)[1] = cb;
  }
  float4* r = reinterpret_cast<float4*>(rec[lane + 1].m);
  r[0] = make_float4(c[0] + m[0], c[1] + m[1], c[2] + m[2], c[3] + m[3]);
  r[1] = make_float4(c[4] + m[4], c[5] + m[5], c[6] + m[6], c[7] + m[7]);
  rec[lane + 1].key = kk;
  __syncwarp();
  if (lane == 31) {                  // the batch's sum into the carried one, read by all lanes above
#pragma unroll
    for (int l = 0; l < ROX_EDGE_TERMS; l++) {
      float v = c[l], e = carry[ROX_EDGE_TERMS + l];
      sum_add(v, e, m[l], 1.0f);
      carry[l] = v;
      carry[ROX_EDGE_TERMS + l] = e;
    }
  }
  const int klast = min(__shfl_sync(0xffffffffu, kk, 31), ROX_SPAN);
  edge_points<NU>(rec, 33, left, kcur, klast, lane, centre, inv_cut, dnu_f, Drow, zacc);
  kcur = max(kcur, klast);
  __syncwarp();
}

// k_moments: the far forms of a cell's lines summed into one multipole expansion. With the cell's
// centre as origin and its half-width as unit, a line at d has f(Y) = (P t + Q)/(t^2 + B),
// t = (Y - d)^2 + A, a rational function whose expansion f = sum_l m_l / Y^(l+2) follows from
// f (Y^4 + d3 Y^3 + d2 Y^2 + d1 Y + d0) = P Y^2 - 2 P d Y + P (d^2 + A) + Q by a four-term
// recurrence, exact for every order. One warp takes four consecutive cells of one job (one where
// there are too few to fill the GPU: 9.8 us with four against 5.2 on a list of 1e4 lines),
// finds the first by a 32-way search of the sorted centres and walks its lines 32 at a time; the lanes'
// sums are added by a fixed tree, every ROX_CELL_FOLD rounds of 32 lines into a compensated total (a cell
// of 2.4e5 lines, one of them 4e7 times the others', was 1.7e-4 off with one plain sum per lane).
// Truncated after ROX_MOMENTS terms the expansion errs by (r^14)(15 - 14 r) of a line's value,
// r = (half-width + pole modulus)/|Y|: k_voigt takes a cell only where r <= 1/4 (5e-8).
#define ROX_CELL_FOLD 16
// Whether an indexed list (the kept lines of a selection) has a line a cell: how many are kept is known
// only here. k_moments and k_voigt decide alike (3e4 lines, most of them dropped: 8.3 us of moments saved).
__device__ __forceinline__ bool kept_fill_cells(const RoxListDev& L, const RoxJobDev& J) {
  return min(L.span_hi[J.span_first + J.n_spans - 1], J.l1) - max(L.span_lo[J.span_first], J.l0) >= J.n_cells;
}
__device__ __forceinline__ float cell_k0(const RoxListDev& L, long long pos) {
  return L.geo[L.idx ? (long long)L.idx[pos] : pos].x;
}
template <int X>
__global__ void __launch_bounds__(256) k_moments(const __grid_constant__ RoxVoigtArgs A) {
  constexpr bool IDX = (X & ROX_VX_INDEX) != 0;
  constexpr bool BRD = (X & ROX_VX_BROAD) != 0;
  constexpr bool PRE = (X & ROX_VX_PRE) != 0;
  if (*(volatile int32_t*)&A.hdr->status != ROX_OK) return;
  const int lane = threadIdx.x & 31;
  const int nw = (int)((gridDim.x * blockDim.x) >> 5);
  for (int task = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5); A.cells_task * task < A.n_slots; task += nw) {
    const int slot = A.cells_task * task;
    int k = 0, k_hi = A.n_jobs - 1;            // last job with mom_off <= slot
    while (k < k_hi) {
      const int mid = (k + k_hi + 1) >> 1;
      if (A.job[mid].mom_off <= slot) k = mid; else k_hi = mid - 1;
    }
    const RoxJobDev& J = A.job[k];
    const RoxListDev& L = A.list[J.list];
    if (J.n_cells <= 0 || *L.status != ROX_OK || (IDX && !kept_fill_cells(L, J))) continue;
    const int s0 = slot - J.mom_off;
    const long long p0 = max(L.span_lo[J.span_first], J.l0);
    const long long p1 = min(L.span_hi[J.span_first + J.n_spans - 1], J.l1);
    const float dnu_f = L.dnu_f, margin_cm = fast_margin(dnu_f);
    const float half = 0.5f * ROX_CELL * dnu_f, ih = 1.0f / half, ih2 = ih * ih;
    const float* S_row = J.S32 - J.l0;
    // first line of cell s0: p0 plus the lines before it
    long long lo = p0, len = max(0LL, p1 - p0);
    const float first = (float)(ROX_CELL * (J.c_first + s0));
    while (len > 0) {
      const long long step = (len + 31) >> 5, off = (long long)lane * step;
      const bool less = off < len && cell_k0(L, lo + off) < first;
      const int c = __popc(__ballot_sync(0xffffffffu, less));
      if (c == 0) break;
      const long long nlo = lo + (c - 1) * step + 1;
      len = min(step - 1, lo + len - nlo);
      lo = nlo;
    }
    for (int s = s0; s < s0 + A.cells_task && s <= J.n_cells; s++) {
      const int cell = J.c_first + s;
      const float centre = (float)(ROX_CELL * cell) + 0.5f * ROX_CELL, end = (float)(ROX_CELL * (cell + 1));
      if (lane == 0) A.cstart[J.mom_off + s] = (int32_t)lo;
      if (s == J.n_cells) break;               // the end of the last cell
      float M[ROX_MOMENTS], pm = 0.f, zm = 0.f;
      float sum = 0.f, cmp = 0.f;              // lane l: moment l of the rounds folded so far
      int rounds = 0;
#pragma unroll
      for (int l = 0; l < ROX_MOMENTS; l++) M[l] = 0.f;
      for (;;) {
        const long long pos = lo + lane;
        bool in = pos < p1;
        long long li = 0;
        float4 g = make_float4(0.f, 0.f, 0.f, 0.f);
        if (in) {
          li = IDX ? (long long)L.idx[pos] : pos;
          g = L.geo[li];
          in = g.x < end;
        }
        const int nb = __popc(__ballot_sync(0xffffffffu, in));
        if (in) {
          float a, b, p, q, tz;
          if constexpr (PRE) {
            const float4* rec = reinterpret_cast<const float4*>(J.S32);
            const float4 r0 = rec[3 * li];
            a = r0.x;
            b = r0.y;
            p = r0.z;
            q = r0.w;
            tz = rec[3 * li + 1].x;
          } else {
            float gref, nt;
            load_widths<BRD>(J, L, L.width_f16, li, gref, nt);
            const LineK kc = line_consts<BRD>(L.nu_min_f + fmaf(g.x, dnu_f, g.y), S_row[li], gref, nt, J, margin_cm);
            a = kc.A;
            b = kc.B;
            p = kc.P;
            q = kc.Q;
            tz = kc.tz;
          }
          // the zone's half-width, t_z = hz^2 + A: from what the records hold too, so that a point has the same
          // cells alone (with records) and in a call of several
          const float z2 = fmaxf(tz - a, 0.f) + 1e-30f;
          const float hz = z2 * rox_rsqrt(z2) * 1.001f;
          const float bm = fabsf(b) + 1e-30f;
          const float r2 = fabsf(a) + bm * rox_rsqrt(bm) + 1e-30f;      // |pole|^2 at most
          pm = fmaxf(pm, r2 * rox_rsqrt(r2) * 1.001f);
          zm = fmaxf(zm, hz);
          const float d = fmaf(g.y, ih, (g.x - centre) * (2.0f / ROX_CELL));
          const float pu = p * ih2, qu = q * (ih2 * ih2), bu = b * (ih2 * ih2);
          const float e = fmaf(d, d, a * ih2);
          const float d3 = 4.0f * d, d2 = -fmaf(d3, d, 2.0f * e), d1 = d3 * e, d0 = -fmaf(e, e, bu);
          float m0 = pu, m1 = 2.0f * pu * d;
          float m2 = fmaf(d3, m1, fmaf(d2, m0, fmaf(pu, e, qu)));
          float m3 = fmaf(d3, m2, fmaf(d2, m1, d1 * m0));
          M[0] += m0;
          M[1] += m1;
          M[2] += m2;
          M[3] += m3;
#pragma unroll
          for (int l = 4; l < ROX_MOMENTS; l++) {
            const float m = fmaf(d3, m3, fmaf(d2, m2, fmaf(d1, m1, d0 * m0)));
            M[l] += m;
            m0 = m1;
            m1 = m2;
            m2 = m3;
            m3 = m;
          }
        }
        lo += nb;
        if (nb == 32 && ++rounds < ROX_CELL_FOLD) continue;
        rounds = 0;
        float v = 0.f;
#pragma unroll
        for (int l = 0; l < ROX_MOMENTS; l++) {
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) M[l] += __shfl_xor_sync(0xffffffffu, M[l], o);
          v = lane == l ? M[l] : v;
          M[l] = 0.f;
        }
        sum_add(sum, cmp, v, 1.0f);
        if (nb < 32) break;
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        pm = fmaxf(pm, __shfl_xor_sync(0xffffffffu, pm, o));
        zm = fmaxf(zm, __shfl_xor_sync(0xffffffffu, zm, o));
      }
      if (!(pm <= 64.0f * half)) pm = 1e30f;   // powers of the poles beyond FP32's range: not to be used
      const float v = lane == ROX_MOMENTS ? pm : (lane == ROX_MOMENTS + 1 ? zm : sum);
      if (lane < 16) reinterpret_cast<float*>(A.mom + 4 * (size_t)(J.mom_off + s))[lane] = v;
    }
  }
}

// NU: the lists are on user-provided nodes (node offsets in dynamic shared memory, one
// ROX_SPAN row of float2 per warp). X: ROX_VX_INDEX (each list is a subset of the sorted lines,
// given by RoxListDev::idx, e.g. the kept lines of a main-contributor selection; span ranges
// then count positions in that index), ROX_VX_BROAD (widths from the broadening pass) and
// ROX_VX_PRE (per-line constants from the preparation kernel). Each
// extra is compiled only into the instantiations that use it: in this kernel even a few added
// instructions per line batch cost several percent of the plain launch.
template <bool NU, int X, int W>
__global__ void __launch_bounds__(W * 32, 20 / W) k_voigt(const __grid_constant__ RoxVoigtArgs A) {
  constexpr bool IDX = (X & ROX_VX_INDEX) != 0;
  constexpr bool BRD = (X & ROX_VX_BROAD) != 0;
  constexpr bool PRE = (X & ROX_VX_PRE) != 0;
  extern __shared__ __align__(16) float2 s_nodes[];   // NU: node offsets; PRE: the staged per-line constants
  __shared__ float4 s_geo[W][32];
  __shared__ float s_S[PRE ? 1 : W][32];
  __shared__ __align__(16) unsigned char s_tab[W][sizeof(BatchTab)];
  __shared__ __align__(16) float s_carry[W][2][ROX_CARRY];   // moments of the edge lines so far, per side
  __shared__ __align__(8) float s_zacc[W][ROX_SPAN];
  __shared__ float s_tot[W][ROX_SPAN];    // the span's sum over its parts
  // a part's sum and its compensation, side by side: one 8-byte access each way a point (rows apart, the
  // exomol list took 0.9% longer)
  __shared__ __align__(8) float2 s_part[W][ROX_SPAN];
  __shared__ float s_totc[W][ROX_SPAN];   // the compensation of s_tot
  __shared__ __align__(16) f32x2 s_cf[W][16];   // a zoned line's form coefficients
  __shared__ int s_status;

  const int tid = threadIdx.x;
  const int lane = tid & 31, w = tid >> 5;
  if (tid == 0) s_status = *(volatile int32_t*)&A.hdr->status;
  __syncthreads();
  if (s_status != ROX_OK) return;   // e.g. unsorted input: leave sigma untouched

  float4* geo_st = s_geo[w];   // this lane's line of the batch; the next batch's copy starts once it is read
  float* S_st = s_S[PRE ? 0 : w];
  BatchTab& BT = *reinterpret_cast<BatchTab*>(s_tab[w]);
  PairTab& PT = BT.pairs;
  LineTab& LT = BT.lines;
  const float lanef = (float)lane;
  const float cheb = rox_cheb_x[lane];
  float* zacc = s_zacc[w];
  float* stot = s_tot[w];
  float2* psum = s_part[w] + lane;        // [32 m]: this lane's points
  float* tot_cmp = s_totc[w] + lane;
  f32x2* cbuf = s_cf[w];
  float* carry = s_carry[w][0];
  const float* cr = rox_core_r[lane & 15];
  const float4 core_r = make_float4(cr[0], cr[1], cr[2], cr[3]);
  float2* Drow = NU ? s_nodes + w * ROX_SPAN : nullptr;   // this span's node offsets
  // PRE: per warp 32 lines x 3 float4 of per-line constants
  float4(*rec_st)[3] = PRE ? reinterpret_cast<float4(*)[3]>(s_nodes + (NU ? W * ROX_SPAN : 0)) + 32 * w : nullptr;
  const float2* D = NU ? Drow + lane : nullptr;
  unsigned long long evals = 0;   // (line, point) pairs inside the cutoff and the job's window

  for (;;) {
    int q = 0, k = 0;
    if (lane == 0) {
      q = atomicAdd(&A.hdr->work_counter, 1);
      int lo_k = 0, hi_k = A.n_jobs - 1;           // first job with q_end > q
      while (lo_k < hi_k) {
        const int mid = (lo_k + hi_k) >> 1;
        if (A.q_end[mid] > q) hi_k = mid; else lo_k = mid + 1;
      }
      k = lo_k;
    }
    q = __shfl_sync(0xffffffffu, q, 0);
    k = __shfl_sync(0xffffffffu, k, 0);
    if (q >= A.n_queue) break;
    // queue entry -> the job's item and part (-1: the whole span, all parts in order)
    const RoxJobDev& J = A.job[k];
    const RoxListDev& Lst = A.list[J.list];
    const int item0 = k > 0 ? A.item_end[k - 1] : 0;
    const int whole = min(max(A.n_whole - item0, 0), J.n_spans);     // the job's whole items come first
    const int lq = q - (k > 0 ? A.q_end[k - 1] : 0), sq = lq - whole;
    const int local = sq < 0 ? lq : whole + sq / J.max_parts, part = sq < 0 ? -1 : sq % J.max_parts;
    const int cnt_i = item0 + local - A.n_whole;                     // split items: counter, first part slot
    const int slot0 = A.slot0[k] + (local - whole) * J.max_parts;
    const int span = J.span_first + J.n_spans - 1 - local;       // wide-line (high nu) spans first
    const int f16 = Lst.width_f16;
    // compensation weight of the part sums: 1 (ROX_KAHAN) keeps the Kahan correction term, 0
    // zeroes it, which leaves the plain sum (one branch-free form for both)
    const float kw = (J.flags & ROX_KAHAN) ? 1.0f : 0.0f;
    const float dnu_f = Lst.dnu_f;
    // offsets on a uniform grid round once more (X0 + 32 m dnu), hence the precision margin
    const float margin_cm = NU ? 0.0f : fast_margin(dnu_f);
    const int Aw = span * ROX_SPAN;
    const int Bw = Aw + ROX_SPAN - 1;
    const int Bg = (int)min((long long)Bw, Lst.n_lattice - 1);   // the span's last point on the grid
    if (*Lst.status != ROX_OK) continue;           // list not prepared from sorted lines
    float bh = 0.f, bl = 0.f, Ws = 0.f;             // span's first node; offset of its last node
    if constexpr (NU) {
#pragma unroll
      for (int m = 0; m < ROX_K; m++) Drow[32 * m + lane] = Lst.node_d[(long long)Aw + 32 * m + lane];
      const float2 b = Lst.span_base[span];
      bh = b.x;
      bl = b.y;
      __syncwarp();
      Ws = Drow[ROX_SPAN - 1].x;
    }
    const float half = NU ? 0.5f * Ws : 0.5f * (ROX_SPAN - 1) * dnu_f;
    const float tau = NU ? fmaf(cheb, half, half) : fmaf(cheb, 0.5f * (ROX_SPAN - 1), 0.5f * (ROX_SPAN - 1));
    const float inv_cut = rox_rcp(Lst.cutoff_f);
    float ntot = 0.f, ncmt = 0.f;   // whole items: this lane's Chebyshev point, over the parts
    const int lo = (int)max(Lst.span_lo[span], J.l0), hi = (int)min(Lst.span_hi[span], J.l1);   // at most 2e9 lines
    const int wlo = (int)max(J.first, (long long)Aw);              // evaluated points of this span
    const int whi = (int)min(J.first + J.n - 1, (long long)Bw);
    const double smax = __longlong_as_double((long long)*J.smax_bits);
    const int e = smax > 0.0 ? ilogb(smax) : 0;     // S32 holds S * 2^-e (FP32)
    if (part > 0 && part >= (max(hi - lo, 0) + 31) >> (5 + J.part_shift)) continue;   // more parts than batches
    const float* S_row = J.S32 - J.l0;              // indexed by line number
    const float4* rec = reinterpret_cast<const float4*>(J.S32);   // PRE: the job's constants of every line

    // Cells taken through their moments: left of the span [cl0, cl1), right of it [cr0, cr1), all of
    // whose lines cover the span, far enough for the expansion and for the lines' slow zones. Their
    // lines [xa, xb) and [xc, xd) leave the span's list, whose other lines are visited one by one.
    int cl0 = 0, cl1 = 0, cr0 = 0, cr1 = 0;
    bool runL = false, runR = false;   // the lines beyond the cells on that side run through the edge scan
    int xa = lo, xb = lo, xc = hi, xd = hi;
    if (!NU && J.n_cells > 0 && hi - lo >= ROX_CELL_LINES * min((2 * Lst.c_steps + ROX_SPAN) >> ROX_CELL_LOG2, J.n_cells) &&
        (!IDX || kept_fill_cells(Lst, J))) {
      const int c_end = J.c_first + J.n_cells;
      cl0 = max((Bw - Lst.c_steps + ROX_CELL - 1) >> ROX_CELL_LOG2, J.c_first);
      cr1 = min((Aw + Lst.c_steps) >> ROX_CELL_LOG2, c_end);
      float pm = 0.f, zm = 0.f;
      // over every cell that can hold a line of the span, edge cells included
      const int ca = max(cl0 - (ROX_CELLS_PER_SPAN + 2), J.c_first), cb = min(cr1 + ROX_CELLS_PER_SPAN + 2, c_end);
      for (int c = ca + lane; c < cb; c += 32) {
        const float4 v = A.mom[4 * (size_t)(J.mom_off + c - J.c_first) + 3];
        pm = fmaxf(pm, v.z);
        zm = fmaxf(zm, v.w);
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        pm = fmaxf(pm, __shfl_xor_sync(0xffffffffu, pm, o));
        zm = fmaxf(zm, __shfl_xor_sync(0xffffffffu, zm, o));
      }
      const float far = fmaxf(4.0f * fmaf(pm, Lst.inv_dnu_f, 0.5f * ROX_CELL), fmaf(zm, Lst.inv_dnu_f, 0.5f * ROX_CELL + 2.0f));
      // in cells from the span's centre, which lies half a step left of the start of cell cm
      const int dc = (int)ceilf((fminf(far, 1e7f) + 0.5f * ROX_SPAN) * (1.0f / ROX_CELL) - 0.5f);
      const int cm = (Aw + ROX_SPAN / 2) >> ROX_CELL_LOG2;
      cl1 = min(cm - dc, c_end);
      cr0 = max(cm + dc, J.c_first);
      if (cl1 > cl0) {
        xa = A.cstart[J.mom_off + cl0 - J.c_first];
        xb = A.cstart[J.mom_off + cl1 - J.c_first];
      } else {
        cl1 = cl0;
      }
      if (cr1 > cr0) {
        xc = A.cstart[J.mom_off + cr0 - J.c_first];
        xd = A.cstart[J.mom_off + cr1 - J.c_first];
      } else {
        cr1 = cr0;
      }
      // all of them no farther from their expansion centre than edge_batch allows, none with its zone
      // in the span
      const float dist = half + (ROX_CELL + 2) * dnu_f;
      const bool fits = dist + pm <= ROX_EDGE_R * (Lst.cutoff_f - half) && zm + dist + half < Lst.cutoff_f;
      runL = fits && cl1 > cl0 && cl0 - (ROX_CELLS_PER_SPAN + 2) >= J.c_first;
      runR = fits && cr1 > cr0 && cr1 + (ROX_CELLS_PER_SPAN + 2) <= c_end;
      if (part <= 0 && lane == 0) evals += (unsigned long long)((long long)(xb - xa) + (xd - xc)) * (unsigned)(whi - wlo + 1);
    }
    // without cells on the left the list is cut at the span's centre, so that the lines left of it
    // can run downwards (their window edges then come in order, see edge_batch); a few batches
    // seldom hold enough of them for a scan, and are left as they are
    const bool ordered = cl1 > cl0 || hi - lo > 4 * 32;
    if (cl1 <= cl0 && ordered) {
      const float mid = NU ? bh + half : (float)(Aw + ROX_SPAN / 2);
      int a = lo, len = hi - lo;
      while (len > 0) {
        const int step = (len + 31) >> 5, off = lane * step;
        const bool less = off < len && cell_k0(Lst, a + off) < mid;
        const int c = __popc(__ballot_sync(0xffffffffu, less));
        if (c == 0) break;
        const int na = a + (c - 1) * step + 1;
        len = min(step - 1, a + len - na);
        a = na;
      }
      xa = xb = min(a, xc);
    }
    const int n1 = xa - lo, n2 = n1 + (xc - xb), nn = n2 + max(hi - xd, 0);   // lines visited one by one
    auto line_at = [&](int q) { return q < n1 ? xa - 1 - q : (q < n2 ? xb + (q - n1) : xd + (q - n2)); };
    const int n_far = (cl1 - cl0) + (cr1 - cr0);

    const int nbat = (nn + 31) >> 5;
    const int np = min(J.max_parts, max(1, nbat >> J.part_shift));     // parts of this span
    if (part >= np) continue;
    const int p_first = part < 0 ? 0 : part, p_last = part < 0 ? np - 1 : part;
    for (int p = p_first; p <= p_last; p++) {
      const int plo = 32 * (int)((long long)nbat * p / np);
      const int phi = min(nn, 32 * (int)((long long)nbat * (p + 1) / np));
      // the part's total and its compensation: psum in shared memory (touched once in four batches), the
      // Chebyshev point's in nsum, ncmp
      int ekL = 0, ekR = 0;             // edge lines: first point without its final sum, per side
      bool edgeL = false, edgeR = false;
      carry[lane] = 0.f;                // both sides' 2 x ROX_CARRY floats
      float acc[ROX_K], nacc = 0.f, nsum = 0.f, ncmp = 0.f;
#pragma unroll
      for (int m = 0; m < ROX_K; m++) {
        acc[m] = 0.f;
        psum[32 * m] = make_float2(0.f, 0.f);
        zacc[32 * m + lane] = 0.f;
      }

      // the runs of edge lines beyond the cells: moments only, two 16-byte records a line, loaded one
      // batch ahead (per line about 7 warp instructions, where the general batch takes 20)
      if constexpr (!NU) {
        __syncwarp();
#pragma unroll 1
        for (int side = 0; side < 2; side++) {
          const bool left = side == 0;
          const int ea = left ? plo : max(plo, n2), eb = left ? min(phi, n1) : phi;
          if (!(left ? runL : runR) || ea >= eb) continue;
          if (left) edgeL = true; else edgeR = true;
          const float centre = left ? half - Lst.cutoff_f : half + Lst.cutoff_f;
          int kcur = 0;
          float4 g_n = make_float4(0.f, 0.f, 0.f, 0.f);
          LineK k_n = {1.f, 1.f, 0.f, 0.f, 1.f, 1.f, 0.f, 0.f, 3e38f, 0.f};
          auto fetch = [&](int q) {
            if (q >= eb) return;
            const int li = IDX ? Lst.idx[line_at(q)] : line_at(q);
            g_n = Lst.geo[li];
            if constexpr (PRE) {
              const float4 r0 = rec[3 * (long long)li];
              k_n.A = r0.x;
              k_n.B = r0.y;
              k_n.P = r0.z;
              k_n.Q = r0.w;
            } else {
              float ga, gb;
              load_widths<BRD>(J, Lst, f16, li, ga, gb);
              k_n = line_consts<BRD>(Lst.nu_min_f + fmaf(g_n.x, dnu_f, g_n.y), S_row[li], ga, gb, J, margin_cm);
            }
          };
          fetch(ea + lane);
          for (int b0 = ea; b0 < eb; b0 += 32) {
            const bool mine = b0 + lane < eb;
            const float4 g = g_n;
            const LineK k = k_n;
            fetch(b0 + 32 + lane);
            const int jlo = __float_as_int(g.z), jhi = __float_as_int(g.w);
            const int ov = min(jhi, whi) - max(jlo, wlo) + 1;
            if (mine && ov > 0) evals += (unsigned)ov;
            const int key = left ? (jhi < Bg ? Bw - jhi : 0) : max(jlo - Aw, 0);
            const float v = -fmaf((float)Aw - g.x, dnu_f, -g.y);
            edge_batch<NU>(BT.scan, carry + ROX_CARRY * side, left, mine, key, (v - centre) * inv_cut, k, kcur, lane, centre, inv_cut,
                           dnu_f, Drow, zacc);
          }
          if (left) ekL = kcur; else ekR = kcur;
        }
      }
      const int mlo = runL ? max(plo, n1) : plo, mhi = runR ? min(phi, n2) : phi;   // the rest, in general batches

      // stage a batch's lines, one a lane: batch 0 here, each next one as soon as the lanes have
      // turned the current one into constants; widths go through registers (with an index, the
      // positions' line numbers one batch further ahead)
      float gref = 0.f, nt = 0.f;
      int li_n = 0;   // IDX: line number of this lane's position in the next batch
      if (IDX && mlo + lane < mhi) li_n = Lst.idx[line_at(mlo + lane)];
      auto stage = [&](int q) {
        if (q < mhi) {
          const int li = IDX ? li_n : line_at(q);
          cp_async16(&geo_st[lane], &Lst.geo[li]);
          if constexpr (PRE) {
#pragma unroll
            for (int c = 0; c < 3; c++) cp_async16(&rec_st[lane][c], &rec[3 * (long long)li + c]);
          } else {
            cp_async4(&S_st[lane], &S_row[li]);
            load_widths<BRD>(J, Lst, f16, li, gref, nt);
          }
        }
        if (IDX && q + 32 < mhi) li_n = Lst.idx[line_at(q + 32)];
        cp_async_commit();
      };
      stage(mlo + lane);
      int nb = 0;
      for (int b0 = mlo; b0 < mhi; b0 += 32, nb++) {
        const int cnt = min(32, mhi - b0);
        cp_async_wait0();   // this lane's copies of the current batch have landed

        // ---- per-line constants (lane <-> line b0 + lane), written to the line's slot
        const bool live = lane < cnt;
        bool covers = false, zoned = false, smooth = false;
        float ax = 0.f, ay = 0.f, vA = 1.f, vB = 0.f, vP = 0.f, vQ = 0.f, tz = 0.f;
        float4 zl = make_float4(1.f, 0.f, 0.f, 0.f);
        LineK kk = {1.f, 1.f, 0.f, 0.f, 1.f, 1.f, 0.f, 0.f, 3e38f, 0.f};
        int jlo = 1, jhi = 0, zlo = 0, zhi = -1;
        if (live) {
          const float4 g = geo_st[lane];
          jlo = __float_as_int(g.z);
          jhi = __float_as_int(g.w);
          const int ov = min(jhi, whi) - max(jlo, wlo) + 1;
          if (ov > 0) evals += (unsigned)ov;
          covers = Aw >= jlo && Bg <= jhi;
          LineK kc;
          float dmin;
          if constexpr (PRE) {
            // uniform grid, constants from k_prep_scaled
            const float4 r0 = rec_st[lane][0], r1 = rec_st[lane][1], r2 = rec_st[lane][2];
            kc.A = r0.x;
            kc.B = r0.y;
            kc.P = r0.z;
            kc.Q = r0.w;
            kc.tz = r1.x;
            kc.iG = r1.y;
            kc.y = r1.z;
            kc.pc = r1.w;
            kc.zc = r2.x;
            if constexpr (NU) {
              // c = nu0 - (span's first node) as a double-float pair (the hi parts cancel exactly)
              const float ch = g.x - bh, cl = g.y - bl;
              ax = ch + cl;
              ay = cl - (ax - ch);
              kc.hz = r2.y;
              dmin = fmaf(ROX_SMOOTH_R, half, r2.w);
            } else {
              zlo = __float_as_int(r2.y);
              zhi = __float_as_int(r2.z);
              ax = (float)Aw - g.x;     // exact: both are integers below 2^24
              ay = -g.y;
              zoned = !(Bw < zlo || Aw > zhi);
              dmin = r2.w;
            }
          } else {
            const float Sp = S_st[lane];
            float nu0f;   // line centre; its offset state {E, F} (uniform grid) or {c hi, c lo} (nodes)
            if constexpr (NU) {
              // c = nu0 - (span's first node) as a double-float pair (the hi parts cancel exactly)
              nu0f = g.x;
              const float ch = g.x - bh, cl = g.y - bl;
              ax = ch + cl;
              ay = cl - (ax - ch);
            } else {
              nu0f = Lst.nu_min_f + fmaf(g.x, dnu_f, g.y);
              ax = (float)Aw - g.x;     // exact: both are integers below 2^24
              ay = -g.y;
            }
            kc = line_consts<BRD>(nu0f, Sp, gref, nt, J, margin_cm);
            if constexpr (!NU) {
              zone_bounds(g, kc.hz, Lst.inv_dnu_f, zlo, zhi);
              zoned = !(Bw < zlo || Aw > zhi);
            }
            dmin = smooth_dmin(kc.A, kc.B, half);
          }
          if constexpr (NU) {
            // the span's offsets run from -c to Ws - c
            const float hb = kc.hz * 1.001f + 1e-6f * (fabsf(ax) + Ws);
            zoned = -ax < hb && Ws - ax > -hb;
            if (zoned) {   // the span's nodes within the zone, by bisection on their offsets (widened a little)
              int q0 = 0, q1 = 0;
#pragma unroll
              for (int st = ROX_SPAN / 2; st > 0; st >>= 1) {
                if (Drow[q0 + st - 1].x - ax < -hb) q0 += st;
                if (Drow[q1 + st - 1].x - ax <= hb) q1 += st;
              }
              zlo = Aw + q0;
              zhi = Aw + q1;      // one past, at most: harmless, each point has its own test
            }
          }
          const float D = NU ? half - ax - ay : fmaf(ax + 0.5f * (ROX_SPAN - 1), dnu_f, ay);
          smooth = covers && !zoned && fabsf(D) >= dmin;
          vA = kc.A;
          vB = kc.B;
          vP = kc.P;
          vQ = kc.Q;
          tz = kc.tz;
          zl = make_float4(kc.iG, kc.y, kc.pc, kc.zc);
          kk = kc;
        }
        // ---- pass 2, all zoned lines of the batch at once where they lie close enough together: at
        // the points each zoned line has clamped in pass 1, the Faddeeva form
        int q0 = max(max(zlo, jlo) - Aw, 0), q1 = min(min(zhi, jhi) - Aw, ROX_SPAN - 1);
        zoned = zoned && live;
        const bool on = zoned && q0 <= q1;
        const int nz = __popc(__ballot_sync(0xffffffffu, on));
        bool batched = false;
        if (nz > 0) {
          const int qa = __reduce_min_sync(0xffffffffu, on ? q0 : ROX_SPAN), qb = __reduce_max_sync(0xffffffffu, on ? q1 : -1);
          batched = qb - qa + 1 <= ROX_ZONE_DENSE * nz;
          if (batched)       // (the tables of the batch before are no longer read: the loop ends in a __syncwarp)
            zone_batch<NU>(on, q0, q1, qa, qb, __any_sync(0xffffffffu, on && (jlo > zlo || jhi < zhi)), kk, ax, ay, dnu_f,
                           Drow, lane, reinterpret_cast<float*>(s_tab[w]), zacc);
        }
        // ---- window edges in order, where the lines are smooth on the span
        bool scanned = false;
        {
          const bool eL = live && !covers && !zoned && jlo <= Aw && jhi < Bg, eR = live && !covers && !zoned && jlo > Aw && jhi >= Bg;
          if (__any_sync(0xffffffffu, eL || eR)) {
            const float cL = half - Lst.cutoff_f, cR = half + Lst.cutoff_f;   // from the span's first point
            const float v = NU ? ax + ay : -fmaf(ax, dnu_f, ay);              // the line, from there
            const float bm = fabsf(kk.B) + 1e-30f, r2 = fabsf(kk.A) + bm * rox_rsqrt(bm) + 1e-30f;
            const float dL = v - cL, dR = v - cR, room = ROX_EDGE_R * (Lst.cutoff_f - half) - r2 * rox_rsqrt(r2);
            bool mL = eL && ordered && fabsf(dL) <= room, mR = eR && fabsf(dR) <= room;
            mL = __popc(__ballot_sync(0xffffffffu, mL)) >= ROX_EDGE_SCAN && mL;
            mR = __popc(__ballot_sync(0xffffffffu, mR)) >= ROX_EDGE_SCAN && mR;
            if (__any_sync(0xffffffffu, mL)) {
              edgeL = true;
              edge_batch<NU>(BT.scan, carry, true, mL, Bw - jhi, dL * inv_cut, kk, ekL, lane, cL, inv_cut, dnu_f, Drow, zacc);
            }
            if (__any_sync(0xffffffffu, mR)) {
              edgeR = true;
              edge_batch<NU>(BT.scan, carry + ROX_CARRY, false, mR, jlo - Aw, dR * inv_cut, kk, ekR, lane, cR, inv_cut, dnu_f, Drow, zacc);
            }
            scanned = mL || mR;
          }
        }
        const unsigned msm = __ballot_sync(0xffffffffu, live && smooth);
        const unsigned cov = __ballot_sync(0xffffffffu, live && covers && !smooth);
        const unsigned edge = __ballot_sync(0xffffffffu, live && !covers && !scanned);
        const int nsm = __popc(msm), ncov = nsm + __popc(cov), nslot = ncov + __popc(edge);
        const unsigned below = (1u << lane) - 1u;
        const int slot = !covers ? ncov + __popc(edge & below)
                         : smooth ? __popc(msm & below) : nsm + __popc(cov & below);
        const unsigned zslots = __reduce_or_sync(0xffffffffu, (on && !batched) ? (1u << slot) : 0u);
        // the line table serves the masked pairs (an odd covering line among them) and pass 2 line by line
        const bool lines_used = (edge != 0) | ((ncov & 1) != 0) | (zslots != 0);
        if (live && !scanned) {
          const int k = slot >> 1, h = slot & 1;
          float* ab = reinterpret_cast<float*>(&PT.ab[k]);
          float* pq = reinterpret_cast<float*>(&PT.pq[k]);
          float* ef = reinterpret_cast<float*>(&PT.ef[k]);
          ab[h] = vA;
          ab[2 + h] = vB;
          pq[h] = vP;
          pq[2 + h] = vQ;
          ef[h] = ax;
          ef[2 + h] = ay;
          reinterpret_cast<float*>(&PT.tz[k])[h] = tz;
          if (lines_used) {
            LT.W[slot] = make_int2(jlo, jhi);
            LT.Z[slot] = make_int2(zlo, zhi);
            LT.z[slot] = zl;
          }
        }
        if ((nslot & 1) && lane == 0) {    // an empty line completes the last pair
          const int k = nslot >> 1;
          float *ab = reinterpret_cast<float*>(&PT.ab[k]), *pq = reinterpret_cast<float*>(&PT.pq[k]);
          float* ef = reinterpret_cast<float*>(&PT.ef[k]);
          ab[1] = ab[3] = 1.f;
          pq[1] = pq[3] = ef[1] = ef[3] = 0.f;
          PT.tz[k].y = 1.f;
          LT.W[nslot] = make_int2(1 << 29, -(1 << 29));
        }
        stage(b0 + 32 + lane);
        __syncwarp();

        // ---- pass 1: smooth pairs at the Chebyshev points; covering pairs at every point of the span,
        // t clamped to the zone boundary (which a line without a slow zone there never meets: one
        // code for both, as the instruction caches are the scarcer resource); the rest (an odd
        // covering line, window-edge lines) in pairs with window masks. Fixed orders: the sum is
        // reproducible.
        const int ks = nsm >> 1, kz = ncov >> 1, ke = (nslot + 1) >> 1;
        for (int k = 0; k < ks; k++) nacc = smooth_pair<NU>(PT, k, tau, dnu_f, nacc);
        for (int k = ks; k < kz; k++) cover_pair<NU>(PT, k, lanef, dnu_f, D, acc);
        for (int k = kz; k < ke; k++) edge_pair<NU>(PT, LT, k, Aw, lane, lanef, dnu_f, D, zacc);
        // ---- pass 2 line by line otherwise
        for (unsigned z = zslots; z; z &= z - 1)
          zone_line<NU>(PT, LT, __ffs(z) - 1, Aw, lane, dnu_f, core_r, D, cbuf, zacc);
        __syncwarp();
        // the partial sums (acc, and zacc's masked pairs and zones) into the part's total every 4
        // batches: compensated (Kahan) with ROX_KAHAN, else plainly (kw = 0: the correction term stays 0)
        if ((nb & 3) == 3 || b0 + 32 >= mhi) {
#pragma unroll
          for (int m = 0; m < ROX_K; m++) {
            float2 v = psum[32 * m];
            sum_add(v.x, v.y, acc[m] + zacc[32 * m + lane], kw);
            psum[32 * m] = v;
            acc[m] = 0.f;
            zacc[32 * m + lane] = 0.f;
          }
          sum_add(nsum, ncmp, nacc, kw);
          nacc = 0.f;
        }
      }
      // edge lines: the points beyond the last edge have all of the part's lines of that side
      __syncwarp();
#pragma unroll 1
      for (int side = 0; side < 2; side++)
        if (side ? edgeR : edgeL)
          edge_points<NU>(reinterpret_cast<const EdgeRec*>(carry + ROX_CARRY * side), 1, side == 0, side ? ekR : ekL, ROX_SPAN, lane,
                          side ? half + Lst.cutoff_f : half - Lst.cutoff_f, inv_cut, dnu_f, Drow, zacc);
      __syncwarp();
      // this part's share of the far cells, at this lane's Chebyshev point, 16 of them to a compensated
      // addition (4e3 cells of 3e-8 each beside one of 1 lost 1.1e-4 in a plain sum)
      float ncell = 0.f;
      for (int c = n_far * p / np, c1 = n_far * (p + 1) / np; c < c1; c++) {
        const int cell = c < cl1 - cl0 ? cl0 + c : cr0 + (c - (cl1 - cl0));
        const float4* mo = A.mom + 4 * (size_t)(J.mom_off + cell - J.c_first);
        const float4 v0 = mo[0], v1 = mo[1], v2 = mo[2], v3 = mo[3];
        const float y = ((float)(Aw - ROX_CELL * cell) + (tau - 0.5f * ROX_CELL)) * (2.0f / ROX_CELL);
        const float z = rox_rcp(y);
        float f = fmaf(z, v3.y, v3.x);
        f = fmaf(z, fmaf(z, fmaf(z, fmaf(z, f, v2.w), v2.z), v2.y), v2.x);
        f = fmaf(z, fmaf(z, fmaf(z, fmaf(z, f, v1.w), v1.z), v1.y), v1.x);
        f = fmaf(z, fmaf(z, fmaf(z, fmaf(z, f, v0.w), v0.z), v0.y), v0.x);
        ncell = fmaf(z * z, f, ncell);
        if ((c & 15) == 15 || c + 1 == c1) {
          sum_add(nsum, ncmp, ncell, 1.0f);
          ncell = 0.f;
        }
      }
      nsum -= ncmp;
      // fold in what the last batches and the edges left in zacc
#pragma unroll
      for (int m = 0; m < ROX_K; m++) {
        psum[32 * m].x += zacc[32 * m + lane] - psum[32 * m].y;
      }
      if (part >= 0) {           // a split item: this part's sum goes to the tail scratch
        float* dst = A.tail_part + (size_t)(slot0 + p) * ROX_PART_FLOATS;
#pragma unroll
        for (int m = 0; m < ROX_K; m++) __stcg(&dst[32 * m + lane], psum[32 * m].x);
        __stcg(&dst[ROX_SPAN + lane], nsum);
      } else {
        sum_add(ntot, ncmt, nsum, kw);
#pragma unroll
        for (int m = 0; m < ROX_K; m++) {
          float v = p == 0 ? 0.f : stot[32 * m + lane], c = p == 0 ? 0.f : tot_cmp[32 * m];
          sum_add(v, c, psum[32 * m].x, kw);
          stot[32 * m + lane] = v;
          tot_cmp[32 * m] = c;
        }
      }
      __syncwarp();
    }   // parts

    if (part >= 0) {
      // the last part to finish adds the parts in order (the same sum as a whole item)
      __threadfence();
      __syncwarp();
      int done = 0;
      if (lane == 0) done = atomicAdd(&A.tail_cnt[cnt_i], 1);
      done = __shfl_sync(0xffffffffu, done, 0);
      if (done != np - 1) continue;
      __threadfence();
      const float* src = A.tail_part + (size_t)slot0 * ROX_PART_FLOATS + lane;
      float v[ROX_K], c[ROX_K];
#pragma unroll
      for (int m = 0; m < ROX_K; m++) v[m] = c[m] = 0.f;
#pragma unroll 2
      for (int pp = 0; pp < np; pp++) {
#pragma unroll
        for (int m = 0; m < ROX_K; m++) sum_add(v[m], c[m], __ldcg(&src[pp * ROX_PART_FLOATS + 32 * m]), kw);
        sum_add(ntot, ncmt, __ldcg(&src[pp * ROX_PART_FLOATS + ROX_SPAN]), kw);
      }
#pragma unroll
      for (int m = 0; m < ROX_K; m++) stot[32 * m + lane] = v[m];
    }
    // ---- the smooth lines' sum at the Chebyshev points, interpolated to the span's points
    if (__any_sync(0xffffffffu, ntot != 0.f)) interp_span<NU>(ntot, lane, D, half, stot);
    // ---- write the span once (its part inside the job's window); a value beyond the FP32
    // range is written as it is and flagged (rox_ws_status: ROX_EOVERFLOW)
    float* out = J.sigma - J.first;
    bool bad = false;
#pragma unroll
    for (int m = 0; m < ROX_K; m++) {
      const int j = Aw + 32 * m + lane;
      if (j >= wlo && j <= whi) {
        const float v = ldexpf(stot[32 * m + lane], e);
        const float o = (J.flags & ROX_ACCUMULATE) ? out[j] + v : v;
        bad |= !isfinite(o);
        out[j] = o;
      }
    }
    if (__any_sync(0xffffffffu, bad) && lane == 0) atomicOr(&A.hdr->overflow, 1);
    __syncwarp();
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) evals += __shfl_xor_sync(0xffffffffu, evals, o);
  if (lane == 0 && evals) atomicAdd(&A.hdr->evals_total, evals);
}

// Probe of the rate of evaluating lines point by point: cover_pair, the loop that k_voigt runs for lines
// that cover a span and are not smooth on it, alone, with W warps per CTA as k_voigt's launch, on synthetic
// far-wing constants held in each warp's pair table (offsets of 3-8 cm^-1, so no clamp applies).
// Each warp walks its 16 pairs `reps` times; no line set-up, staging, edges or slow
// zones. Not part of the cross-section method.
template <int W>
__global__ void __launch_bounds__(W * 32, 24 / W) k_pair_loop_probe(float* out, int reps, float dnu_f) {
  __shared__ PairTab s_pairs[W];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  PairTab& PT = s_pairs[w];
  if (lane < 16) {
    const float i0 = (float)(2 * lane), i1 = (float)(2 * lane + 1);
    PT.ab[lane] = make_float4(1.0e-4f * (1.0f + i0), 1.0e-4f * (1.0f + i1), 1.0e-8f * (1.0f + i0), 1.0e-8f * (1.0f + i1));
    PT.pq[lane] = make_float4(1.0e-3f, 1.1e-3f, 2.0e-7f, 2.1e-7f);
    PT.ef[lane] = make_float4(-300.0f - 17.0f * i0, -300.0f - 17.0f * i1, -0.0037f * (i0 + 1.0f), -0.0037f * (i1 + 1.0f));
    PT.tz[lane] = make_float2(0.0f, 0.0f);
  }
  __syncwarp();
  float acc[ROX_K];
#pragma unroll
  for (int m = 0; m < ROX_K; m++) acc[m] = 0.0f;
  const float lanef = (float)lane;
  for (int r = 0; r < reps; r++) {
#pragma unroll 1
    for (int k = 0; k < 16; k++) cover_pair<false>(PT, k, lanef, dnu_f, nullptr, acc);
  }
  float t = 0.0f;
#pragma unroll
  for (int m = 0; m < ROX_K; m++) t += acc[m];
  out[(size_t)blockIdx.x * blockDim.x + threadIdx.x] = t;
}

__global__ void k_faddeeva(const float* x, const float* y, float* out, long long n) {
  long long stride = (long long)gridDim.x * blockDim.x;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride)
    out[i] = rox_re_w(&rox_daw_taylor[0][0], x[i], y[i]);
}

}  // namespace

namespace {
// dynamic shared memory of an instantiation with W warps per CTA: the node rows (NU), then the
// staged per-line constants (ROX_VX_PRE)
template <bool NU, int X, int W>
constexpr size_t voigt_dyn_smem() {
  return (NU ? (size_t)W * ROX_SPAN * sizeof(float2) : (size_t)0) +
         ((X & ROX_VX_PRE) ? (size_t)W * 32 * 3 * sizeof(float4) : (size_t)0);
}
}  // namespace

namespace {

template <bool NU, int X, int W>
cudaError_t launch_k(const RoxVoigtArgs& A, int n_blocks, cudaStream_t s) {
  constexpr size_t dyn = voigt_dyn_smem<NU, X, W>();
  if (dyn) {   // static shared memory plus these exceed 48 KB: opt in (idempotent, per device)
    cudaError_t e = cudaFuncSetAttribute(k_voigt<NU, X, W>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dyn);
    if (e != cudaSuccess) return e;
  }
  k_voigt<NU, X, W><<<n_blocks, W * 32, dyn, s>>>(A);
  return cudaGetLastError();
}

template <bool NU, int X, int W>
cudaError_t blocks_k(int* nb) {
  constexpr size_t dyn = voigt_dyn_smem<NU, X, W>();
  if (dyn) {
    cudaError_t e = cudaFuncSetAttribute(k_voigt<NU, X, W>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dyn);
    if (e != cudaSuccess) return e;
  }
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(nb, k_voigt<NU, X, W>, W * 32, dyn);
}

template <int W>
cudaError_t launch_w(const RoxVoigtArgs& A, int n_blocks, bool nodes, int extras, cudaStream_t s) {
  if (nodes) {
    if (extras == ROX_VX_PRE) return launch_k<true, ROX_VX_PRE, W>(A, n_blocks, s);
    if (extras) return cudaErrorNotSupported;   // no caller combines nodes with a selection or broadening
    return launch_k<true, 0, W>(A, n_blocks, s);
  }
  switch (extras) {
    case 0: return launch_k<false, 0, W>(A, n_blocks, s);
    case ROX_VX_INDEX: return launch_k<false, ROX_VX_INDEX, W>(A, n_blocks, s);
    case ROX_VX_BROAD: return launch_k<false, ROX_VX_BROAD, W>(A, n_blocks, s);
    case ROX_VX_PRE: return launch_k<false, ROX_VX_PRE, W>(A, n_blocks, s);
    default: return cudaErrorNotSupported;   // no entry point combines these extras
  }
}

template <int W>
cudaError_t blocks_w(int* nb, bool nodes, bool pre) {
  if (pre) return nodes ? blocks_k<true, ROX_VX_PRE, W>(nb) : blocks_k<false, ROX_VX_PRE, W>(nb);
  if (nodes) return blocks_k<true, 0, W>(nb);
  return blocks_k<false, 0, W>(nb);
}

}  // namespace

// warps: warps per CTA of the launch (4 or 8; the launch configuration of rox_launch_config)
cudaError_t rox_launch_voigt(const RoxVoigtArgs& A, int n_blocks, bool nodes, int extras, int warps, cudaStream_t s) {
  if (warps == 4) return launch_w<4>(A, n_blocks, nodes, extras, s);
  if (warps == 8) return launch_w<8>(A, n_blocks, nodes, extras, s);
  return cudaErrorInvalidValue;
}

// moments of the cells of A's jobs (A.n_slots of them) ahead of the Voigt launch
cudaError_t rox_launch_moments(const RoxVoigtArgs& A, int extras, cudaStream_t s) {
  if (A.n_slots <= 0) return cudaSuccess;
  long long b = (A.n_slots / A.cells_task + 7) / 8;      // n_slots is a multiple of 4
  if (b > 152 * 16) b = 152 * 16;
  switch (extras) {
    case 0: k_moments<0><<<(int)b, 256, 0, s>>>(A); break;
    case ROX_VX_INDEX: k_moments<ROX_VX_INDEX><<<(int)b, 256, 0, s>>>(A); break;
    case ROX_VX_BROAD: k_moments<ROX_VX_BROAD><<<(int)b, 256, 0, s>>>(A); break;
    case ROX_VX_PRE: k_moments<ROX_VX_PRE><<<(int)b, 256, 0, s>>>(A); break;
    default: return cudaErrorNotSupported;
  }
  return cudaGetLastError();
}

cudaError_t rox_voigt_blocks_per_sm(int* nb, bool nodes, bool pre, int warps) {
  if (warps == 4) return blocks_w<4>(nb, nodes, pre);
  if (warps == 8) return blocks_w<8>(nb, nodes, pre);
  return cudaErrorInvalidValue;
}

// pair-loop probe: n_blocks CTAs of `warps` warps (4 or 8); out holds n_blocks * warps * 32 floats
cudaError_t rox_launch_pair_loop_probe(int n_blocks, int warps, int reps, float* out, cudaStream_t s) {
  if (warps == 4) k_pair_loop_probe<4><<<n_blocks, 4 * 32, 0, s>>>(out, reps, 0.01f);
  else if (warps == 8) k_pair_loop_probe<8><<<n_blocks, 8 * 32, 0, s>>>(out, reps, 0.01f);
  else return cudaErrorInvalidValue;
  return cudaGetLastError();
}

cudaError_t rox_launch_faddeeva(const float* x, const float* y, float* out, long long n, cudaStream_t s) {
  long long b = (n + 255) / 256;
  if (b > 152 * 8) b = 152 * 8;
  if (b < 1) b = 1;
  k_faddeeva<<<(int)b, 256, 0, s>>>(x, y, out, n);
  return cudaGetLastError();
}
