// Internal definitions shared by the librox translation units (CUDA path only).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>
#include "../../include/rox.h"

// Physical constants (CODATA 2018; c, h, k_B exact in SI).
#define ROX_C_CM 2.99792458e10          // speed of light, cm/s
#define ROX_C_M 2.99792458e8            // speed of light, m/s
#define ROX_KB 1.380649e-23             // Boltzmann constant, J/K
#define ROX_HPLANCK 6.62607015e-34      // Planck constant, J s
#define ROX_AMU 1.66053906660e-27       // atomic mass constant, kg
#define ROX_C2 (ROX_HPLANCK * ROX_C_CM / ROX_KB)  // second radiation constant, cm K
#define ROX_T_REF 296.0                 // K, reference temperature of S_ref and gamma_ref
#define ROX_P_REF 1.01325               // bar, 1 atm
#define ROX_PI 3.14159265358979323846

// Voigt work geometry: a warp owns one span of ROX_SPAN = 32*ROX_K consecutive grid points
// (each lane ROX_K points strided by 32) and is its own unit of scheduling; the warps of a CTA
// share nothing. Lines reach a warp in batches of 32.
#define ROX_K (ROX_SPAN / 32)           // ROX_SPAN (include/rox.h) = 256 grid points per span
#define ROX_TILE ROX_SPAN               // grid points per work item (per-item line ranges)

// The far formula (rox_re_w_far in physical units) is used only outside each line's slow
// zone, whose boundary |z|^2 goes with the line's y (rox_far_coefs). Its per-point offset is
// X_m = X_0 + 32 m dnu with X_0 the offset at the thread's first point, so X_m carries a
// rounding error of 6e-8 (|X_m| + span). What that does to the profile goes with the larger of |X|
// and gamma_L (the poles lie gamma_L off the axis), so the slow zone around each line reaches at least to
// X^2 + gamma_L^2 = (ROX_FAST_MARGIN * span)^2 (line_consts), which keeps the error below 2e-6 relative.
#define ROX_FAST_MARGIN 0.032

// Workspace header at the start of every xsec / prepared-list workspace.
struct RoxWsHeader {
  int32_t status;                  // ROX_OK / ROX_EUNSORTED / ROX_EGRID
  int32_t n_pt;
  unsigned long long evals_lines;  // (line, point) pairs inside the cutoff on the whole lattice
  unsigned long long evals_total;  // pairs evaluated by the last Voigt launch(es), all jobs
  int32_t work_counter;            // persistent-kernel work queue
  int32_t overflow;                // set by the Voigt kernel when it writes a non-finite sigma
  unsigned long long smax_bits[ROX_MAX_PT];  // per strength row: max S (double bits)
};
#define ROX_WS_HEADER_BYTES 8192

// Voigt launch: up to ROX_MAX_LISTS prepared line lists and ROX_MAX_JOBS jobs, each job one
// output window on its list's lattice at one (P,T) point; work items are (job, span) pairs.
#define ROX_MAX_JOBS 224
#define ROX_MAX_LISTS 8

struct RoxListDev {
  const int32_t* status;      // the list's preparation status (ROX_OK unless its nu0 was unsorted)
  const float4* geo;          // [n_lines] {k0 (float, exact), f*dnu, jlo (int bits), jhi (int bits)}
  const long long* span_lo;   // per lattice span of ROX_SPAN points: first line reaching it
  const long long* span_hi;   //   and one past the last
  const void* gamma_ref;
  const void* n_t;
  // broadened lists only (else NULL): per line and distinct temperature the broadeners' sum
  // sum_b vmr_b gamma_ref_b (296/T)^n_b, the job's row at gLT + t_row * gLT_stride; per line
  // the natural width (or NULL)
  const float* gLT;
  long long gLT_stride;
  const float* gN;
  // indexed lists only (else NULL): the list's lines as indices into the sorted line arrays, in
  // order (span ranges then count positions in this index)
  const int32_t* idx;
  // user-provided nodes only (NULL on a uniform grid): per node its offset from the first node
  // of its span, per span that first node, both as double-float pairs {hi, lo}; geo then holds
  // {nu0 hi, nu0 lo, jlo, jhi}
  const float2* node_d;
  const float2* span_base;
  long long n_lattice;
  float dnu_f;
  float nu_min_f;
  int32_t width_f16;
  float inv_dnu_f;            // 1/dnu (uniform grid; 0 on nodes)
  float cutoff_f;             // wing cutoff (cm^-1)
  int32_t c_steps;            // floor(cutoff / dnu) - 2: points every line's window surely reaches on each side
};

// Multipole cells (uniform grids): ROX_CELL grid steps of line centres, lines with k0 in
// [ROX_CELL c, ROX_CELL (c + 1)). Per job and cell 16 floats: ROX_MOMENTS coefficients of the sum
// of the cell's far forms in powers of 1/(offset from the cell's centre) (rox_voigt.cu, k_moments),
// the largest modulus of a pole and the largest slow-zone half-width of its lines (cm^-1).
#define ROX_CELL_LOG2 6
#define ROX_CELL (1 << ROX_CELL_LOG2)
#define ROX_MOMENTS 14
#define ROX_CELL_LINES 2           // lines a cell (of those within reach, at most the job's) from which a span
                                   // takes its cells: reading a cell takes 25 instructions, a line that
                                   // is smooth on the span about 20
#define ROX_CELL_EXT 512           // cells kept on each side of a job's spans (further lines: one by one)
#define ROX_MOM_JOBS 16            // jobs whose cells the workspace of a cross-section call holds at a time
#define ROX_CELL_BYTES 68          // 16 floats and the cell's first line (int32)
#define ROX_CELLS_PER_SPAN (ROX_SPAN / ROX_CELL)

// Lorentz-width description of rox_broadening in kernel parameter form
struct RoxBroadDev {
  int32_t n_b;
  int32_t natural;
  int32_t f16;                 // per-line columns stored as half
  int32_t pad;
  float vmr[ROX_MAX_BROADENERS];
  const void* gamma[ROX_MAX_BROADENERS];
  const void* n[ROX_MAX_BROADENERS];
  const float* tab_gamma[ROX_MAX_BROADENERS];
  const float* tab_n[ROX_MAX_BROADENERS];
  const int32_t* j_lower;
  long long tab_len;
};

// extras of a Voigt launch (kernel instantiations)
#define ROX_VX_INDEX 1    // lists are subsets of the sorted lines given by an index (RoxListDev::idx)
#define ROX_VX_BROAD 2    // widths from the broadening pass (RoxListDev::gLT, gN)
#define ROX_VX_PRE 4      // per-line constants precomputed for each (P,T) point (RoxJobDev::S32)
// (P,T) points up to which a call on user-provided nodes keeps them, 48 bytes of workspace per line and
// point (on a uniform grid: one, where most pairs need only the cells' moments). 3e6 lines, 3e6 nodes:
// kept 2.53, 4.61, 6.72, 8.85 ms for one to four points, per span 2.64, 4.86, 7.09, 9.33; 5% also on 1e6 lines,
// nothing on 3e4 (0.389 and 0.385 ms). The gain does not fall with the points; the workspace sets the limit.
#define ROX_PRE_POINTS 4
#define ROX_PRE_NODES_BYTES ((size_t)16 << 30)   // and up to 6% of the device's memory

struct RoxJobDev {
  // S * 2^-e of lines l0, l0+1, ... at this job's T. In a ROX_VX_PRE launch the job's per-line
  // constants instead, 3 float4 for each line of the list: {A, B, P, Q}, {t_z, 1/gamma_G, y,
  // S/(gamma_G sqrt(pi))}, {X^2 of the end of its own zone (LineTab::z), zlo, zhi (int bits),
  // smooth_dmin}; on user-provided nodes the last is {X^2, zone half-width, 0, smooth_dmin at width 0}
  const float* S32;
  float* sigma;                          // sigma[j - first] for lattice points j in [first, first + n)
  const unsigned long long* smax_bits;   // this job's largest strength (double bits)
  long long l0;
  long long l1;                          // lines [l0, l1) have strengths (others are skipped)
  long long first;
  long long n;
  int32_t list;
  int32_t span_first;
  int32_t n_spans;
  float p_fac;      // P / P_ref
  float gG_fac;     // sqrt(2 k T / (m amu)) / c  -> gamma_G = nu0 * gG_fac
  float l2_ratio;   // log2(T_ref / T)           -> (T_ref/T)^n_T = exp2(n_T * l2_ratio)
  uint32_t flags;   // ROX_ACCUMULATE, ROX_KAHAN
  int32_t t_row;    // broadened lists: the job's temperature row of the list's gLT
  int32_t mom_off;  // the job's first slot in RoxVoigtArgs::mom and cstart (a multiple of 4)
  int32_t c_first;  // the cell of that slot
  int32_t part_shift;  // a span's parts: its batches of lines >> part_shift, 1 .. max_parts
  int32_t max_parts;   // 1 .. rox_parts_cap(n_spans)
  int32_t n_cells;  // cells with moments (slot n_cells holds only the first line beyond them); 0: none
};

// Every span's lines are summed as up to rox_parts_cap consecutive parts (batch-aligned), each from
// zero, and the part sums are added in part order. How many is fixed by the job and the span: a job of
// many spans (three rounds of the GPU's warps or more) fills it with whole items and takes a part per 16
// batches (a part's fixed work, some 400 instructions and the wait for its first batch, is not worth
// less), a shorter one a part per 1 to 4 batches, in many spans at most about twice what they have on
// average (a split item has a queue entry per possible part; set_parts in rox_api.cu). Jobs of few spans may take more parts than 16, so
// that a narrow window on a dense list still fills the GPU (12 spans of 4e6 lines: 192 warps with 16
// parts, 1,536 with 128). A work item is normally a whole span; the
// last items of a launch are split into their parts, taken by different warps: each part stores
// its sum in the tail scratch and the last of them to finish adds the parts in the same order.
// The result is the same either way, so it depends neither on the split nor on the launch grid.
// How many items are split is chosen per launch so that the whole items fill complete rounds of
// the launch's warps and the split ones end the launch in pieces of a part (at most
// ROX_TAIL_ITEMS_MAX items and the part slots of the workspace's tail scratch).
#define ROX_PARTS 16
#define ROX_PARTS_MAX 128
#define ROX_JOB_PART_SLOTS 2048    // part slots that a job of few spans may use
static inline long long rox_parts_cap(long long n_spans) {
  const long long c = n_spans > 0 ? ROX_JOB_PART_SLOTS / n_spans : ROX_PARTS_MAX;
  return c > ROX_PARTS_MAX ? ROX_PARTS_MAX : (c < ROX_PARTS ? ROX_PARTS : c);
}
#define ROX_TAIL_ITEMS_MAX 8192
// A part's sum: its ROX_SPAN points, then its values at the span's ROX_NODES Chebyshev points
// (the lines that are smooth on the span, rox_voigt.cu)
#define ROX_NODES 32
#define ROX_PART_FLOATS (ROX_SPAN + ROX_NODES)

struct RoxVoigtArgs {
  RoxWsHeader* hdr;
  float* tail_part;                 // [part slots][ROX_PART_FLOATS] part sums
  int32_t* tail_cnt;                // [n_items - n_whole] parts finished (zeroed per launch)
  float4* mom;                      // [slots][4] moments of the jobs' cells
  int32_t* cstart;                  // [slots] first line (position) of each cell
  int32_t n_jobs;
  int32_t cells_task;               // cells a warp of k_moments takes at a time: 4, or 1 in small launches
  int32_t n_slots;                  // slots over all jobs (0: no moments in this launch)
  int32_t n_items;                  // items (spans over all jobs); the last n_items - n_whole split
  int32_t n_whole;
  int32_t n_queue;                  // queue entries: one per whole item, max_parts of its job per split item
  int32_t item_end[ROX_MAX_JOBS];   // item_end[k] = spans of jobs 0..k
  int32_t q_end[ROX_MAX_JOBS];      // queue entries of jobs 0..k
  int32_t slot0[ROX_MAX_JOBS];      // part slot of job k's first split item
  RoxListDev list[ROX_MAX_LISTS];
  RoxJobDev job[ROX_MAX_JOBS];
};
static_assert(sizeof(RoxVoigtArgs) < 32000, "kernel parameter space");

// Strengths of each job's line range at the job's temperature (rox_xsec_jobs).
struct RoxStrengthList {
  const double* nu0;
  const float* s_or_a;
  const float* g_up;
  const float* e_lower;
  int32_t convention;
  int32_t pad;
};
struct RoxStrengthJob {
  long long l0, count;     // lines [l0, l0 + count) of list `list`
  double* S64;             // [count]
  float* S32;              // [count], S * 2^-e of the job's maximum
  unsigned long long* smax_bits;
  double inv_T, q_ratio, c2_dT;
  int32_t list;
  int32_t pad;
};
struct RoxStrengthJobs {
  int32_t n_jobs;
  int32_t pad;
  RoxStrengthList list[ROX_MAX_LISTS];
  RoxStrengthJob job[ROX_MAX_JOBS];
};
static_assert(sizeof(RoxStrengthJobs) < 32000, "kernel parameter space");

static inline size_t rox_align256(size_t b) { return (b + 255) & ~(size_t)255; }
// moment slots of a job over n_spans spans, and the bytes of a number of slots
static inline long long rox_job_slots(long long n_spans) {
  return n_spans * ROX_CELLS_PER_SPAN + 2 * ROX_CELL_EXT + 4;
}
static inline size_t rox_mom_bytes(long long slots) {
  return rox_align256((size_t)slots * 64) + rox_align256((size_t)slots * 4);
}
// tail scratch of a workspace: part slots of ROX_PART_FLOATS floats (the items' counters lie next to the
// header)
static inline size_t rox_tail_part_bytes(long long slots) {
  return rox_align256((size_t)slots * ROX_PART_FLOATS * sizeof(float));
}
