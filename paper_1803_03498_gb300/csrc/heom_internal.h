// Internal declarations shared by the CUDA translation units of libheom (not part of the ABI).
#pragma once
#include <cuda_runtime.h>

#include <cstdint>
#include <string>
#include <vector>

#include "hierarchy.h"

namespace heom {

constexpr int kMaxStates = 24;
constexpr int kGenMaxStates = 32;  // states of general runs (element kernels only)

void set_error(const std::string &msg);

// Device error word of a run (StageCommon::err): bit 0 -- a bounded device-side wait gave up (the
// tensor-core kernel's, or the barrier of a launch of whole steps); bit 1 -- a bounds check of the debug build failed.  Every call that returns
// results of the run reports them as HEOM_E_TIMEOUT and HEOM_E_BOUNDS.
constexpr int kErrTimeout = 1;
constexpr int kErrBounds = 2;

// Debug build (compiled with -DHEOM_DEBUG): every neighbour index a link record names, its coupled
// state and every record range a stage kernel reads are checked before use; an index outside its
// range sets kErrBounds in the run's error word and the access is skipped.  Without HEOM_DEBUG the
// check is the constant true and costs nothing.
#ifdef HEOM_DEBUG
__device__ __forceinline__ bool heom_in_range(int *err, int64_t idx, int64_t lo, int64_t hi) {
  if (idx >= lo && idx < hi) return true;
  if (err) atomicOr(err, kErrBounds);
  return false;
}
#define HEOM_IN_RANGE(err, idx, lo, hi) heom_in_range((err), (int64_t)(idx), (int64_t)(lo), (int64_t)(hi))
#else
#define HEOM_IN_RANGE(err, idx, lo, hi) true
#endif

// A batch of nr link records starting at record lo, read from a region that holds records
// [rbase, limit): nr, or 0 (and kErrBounds) when the debug build finds the batch outside the region.
__device__ __forceinline__ int heom_rec_batch(int *err, int64_t lo, int nr, int64_t rbase, int64_t limit) {
#ifdef HEOM_DEBUG
  if (lo < rbase || nr < 0 || lo + nr > limit) {
    if (err) atomicOr(err, kErrBounds);
    return 0;
  }
#endif
  return nr;
}

// One link of an ADO u to a neighbour v = n(u) +- e_l through a mode l of state s.  Only row s and
// column s of v contribute to row s and column s of d sigma_u / dt: element (s, j != s) with
// coefficient R, element (i != s, s) with conj(R), element (s, s) with 2 Re R, where
//   up link (v = n + e_l):    R = i s+_l(n_l)            (s+ = sqrt((n_l + 1) |c_l|), or 1)
//   down link (v = n - e_l):  R = s-_l(n_l) (lamnu_l + i c_l)   (s- = sqrt(n_l / |c_l|), or n_l)
// (V^x contributes +1 on row s and -1 on column s, V^o +1 on both, 2 on the diagonal).
// The records of one ADO are ordered by s.  Field s holds the state in bits 0..7 and the owning
// ADO's index u mod 32 in bits 8..12, so that a warp working on ADOs u0 .. u0 + 31 finds the owner
// of a record as ((s >> 8) - u0) mod 32 without a search.
constexpr int kRecStateMask = 0xff;
template <typename T>
struct LinkRec;
template <>
struct alignas(16) LinkRec<float> {
  int v, s;
  float re, im;
};
template <>
struct alignas(16) LinkRec<double> {
  int v, s, pad0, pad1;
  double re, im;
};

// Hierarchy state storage of one RK4 copy: ADOs u < u_split ("head") as FP64 complex, ADOs
// u >= u_split ("body") as complex of the run's storage type.  Every ADO's N x N tile is contiguous
// and row-major: head[u * E + e], body[(u - u_split) * Ep + e] with E = N^2 and Ep = E rounded up so
// that a body tile is a multiple of 16 bytes.
struct StateView {
  double2 *head;
  void *body;
};

// Everything a stage launch needs besides H, passed by value in the kernel parameters.
struct StageCommon {
  StateView zin;        // state the RHS is evaluated on (own tile and neighbour gathers)
  StateView y;          // Horner base y (head == nullptr && body == nullptr: none)
  StateView out;        // result y + ch * L zin (or ch * L zin)
  const int64_t *link_off;  // [n_ado + 1] first link record of each ADO
  const void *recs_head;    // LinkRec<double> of ADOs u < u_split, indexed by link_off[u]
  const void *recs_body;    // LinkRec<body compute type> of ADOs u >= u_split, by link_off[u] - rec_split
  int64_t rec_split;        // link_off[u_split]
  const double *gsum;       // [n_ado] sum_l n_l gamma_l
  int E, Ep;                // N^2 and the body tile pitch (E rounded up to 16-byte tiles)
  int u_split, n_ado;
  int u_begin, u_end;   // ADO range of this launch
  int n;
  int cplx_h;           // H has an imaginary part
  int herm;             // every ADO is Hermitian: gather row s only, and s H = (H s)^dagger
  int *err;             // device error word (kErrTimeout, kErrBounds)
  int64_t n_recs;       // link records in all (link_off[n_ado]); the debug build checks ranges against it
  int occ_pct;          // schedule: grid sized for this percentage of the CTAs that fit on an SM
  int cpw;              // schedule: column-0 kernels' chunks per warp step (1, 2, 4)
};

// Nonzero while heom_propagate_static creates its run: the autotuner stays off there.
extern thread_local int g_tune_suppress;

// Chunks of floor(32 / n) ADOs that a column-0 warp step holds for a schedule's chunks per warp g:
// g, capped so that a step holds at most 32 ADOs (a link record names its ADO by u mod 32).
__host__ __device__ constexpr int vec_group(int n, int g) { return g < 32 / (32 / n) ? g : 32 / (32 / n); }

// CTAs per SM of the grid for a schedule's occupancy percentage (at least 1): up to 100 a persistent
// grid filling that share of each SM's CTA slots; above 100 that many percent of one resident wave,
// so that CTAs retire while the launch runs.
inline int sched_ctas(int per_sm, int occ_pct) {
  const int b = occ_pct <= 0 ? per_sm : per_sm * occ_pct / 100;
  return b < 1 ? 1 : b;
}

// Coherence-block (column-0) stage kernels (vec_stage_g{1,2,4}.cu, one unit per chunks-per-warp
// value): kind 0 FP64, 1 mixed body (FP32), 2 mixed head (FP64 compute, FP32 body neighbours).
// launch_stage_vec picks the unit from c.cpw.
int launch_stage_vec(int kind, const StageCommon &c, double ch, const double *term, const double *H, cudaStream_t st,
                     int sm_count);
#define HEOM_DECLARE_VEC(R)                                                                                 \
  int launch_stage_vec_g##R(int kind, const StageCommon &c, double ch, const double *term, const double *H, \
                            cudaStream_t st, int sm_count);
HEOM_DECLARE_VEC(1)
HEOM_DECLARE_VEC(2)
HEOM_DECLARE_VEC(4)
#undef HEOM_DECLARE_VEC

// Stage arguments of one run for the batched column-0 kernel; lives in the run's workspace.
struct VecRunDesc {
  StageCommon c;
  double ch;
  // row-major H, stride kMaxStates (shifted, rad/fs), then Delta per state: doubles, or floats for an FP32 body
  double H[kMaxStates * kMaxStates + kMaxStates];
};
constexpr int kBatchMaxRuns = 1024;   // runs per batched launch (kernel-parameter space)
struct VecBatchArgs {
  const VecRunDesc *d[kBatchMaxRuns];
  int64_t chunk0[kBatchMaxRuns + 1];  // prefix sums of the runs' warp-step counts (for cpw)
  int nruns;
  int occ_pct, cpw;                   // schedule of the launch (the runs' own schedules do not apply)
};
// One launch of the batched column-0 kernel for runs of n states (kind as launch_stage_vec).
int launch_stage_vec_batch(int kind, int n, const VecBatchArgs &a, cudaStream_t st, int sm_count);
int launch_stage_vec_batch_g1(int kind, int n, const VecBatchArgs &a, cudaStream_t st, int sm_count);
int launch_stage_vec_batch_g2(int kind, int n, const VecBatchArgs &a, cudaStream_t st, int sm_count);
int launch_stage_vec_batch_g4(int kind, int n, const VecBatchArgs &a, cudaStream_t st, int sm_count);

// Tensor-core (split-TF32) form of the FP32 body stage: Hermitian runs with real H and N <= 16.
// Returns 1 when it does not cover n_states.
int launch_stage_tc_a(const StageCommon &c, double ch, const double *term, const double *H, cudaStream_t st,
                      int sm_count);
int launch_stage_tc_b(const StageCommon &c, double ch, const double *term, const double *H, cudaStream_t st,
                      int sm_count);

template <typename CT>
struct StageArgs {
  StageCommon c;
  CT ch;                      // Horner coefficient times h (1 for a bare RHS evaluation)
  CT term[kMaxStates];        // terminator Delta per state (0 if none)
  alignas(16) CT H[kMaxStates * kMaxStates];   // Re H - h0 I, row stride kMaxStates, rad/fs (pairs load as 8 bytes)
  CT Hi[kMaxStates * kMaxStates];  // Im H
};

// Stage launchers, one per storage combination and range of n (stage_*.cu); each returns 0 on
// success, 1 if n is not compiled in that unit, negative on error.
#define HEOM_DECLARE_LAUNCH(NAME)                                                                      \
  int NAME(const StageCommon &c, double ch, const double *term, const double *H, const double *Hi, \
           cudaStream_t st, int sm_count);
HEOM_DECLARE_LAUNCH(launch_stage_fp32_a)
HEOM_DECLARE_LAUNCH(launch_stage_fp32_b)
HEOM_DECLARE_LAUNCH(launch_stage_fp32_c)
HEOM_DECLARE_LAUNCH(launch_stage_fp32_d)
#undef HEOM_DECLARE_LAUNCH


// Column-form FP64 stage kernel (stage_col.cuh) for Hermitian runs with a real H and 8 <= n <= 16:
// every lane of a warp owns one column of one part of an ADO's result, so all 32 lanes do FP64 work.
// Returns 1 when it does not cover n.
constexpr bool col_covers(int n) { return n >= 8 && n <= 16; }
constexpr int col_gcd(int a, int b) { return b == 0 ? a : col_gcd(b, a % b); }
constexpr int col_passes(int n) { return 2 * n / col_gcd(2 * n, 32); }  // of 32 columns per warp chunk
int launch_stage_col(const StageCommon &c, double ch, const double *term, const double *H, cudaStream_t st,
                     int sm_count);

// Element kernels (resident.cuh).  Constants of a matrix-layout run, in its workspace, [n][n] row-major
// and FP64: Re H - h0, Im H, the terminator rate T_ij of element (i, j), and the terminator Delta_i per state; mup: the
// laser field's M+ of this launch (NULL: no field).
struct ElConsts {
  const double *H, *Hi, *T, *mup, *term;
};
// M+ by value: a captured launch keeps its field when the run's field changes.
template <bool SET>
struct ElMup {};
template <>
struct ElMup<true> {
  double v[kGenMaxStates * kGenMaxStates];
};
// One stage over [c.u_begin, c.u_end): out = y + c1 L zin, and out2 = y2 + c2 L zin if out2 is set;
// gr + i gi is the laser field's g(t).
struct ElStageArgs {
  StageCommon c;
  ElConsts k;
  StateView y2, out2;
  double c1, c2, gr, gi;
  int apu, splits;  // ADOs per unit, or (apu = 1) units per ADO (set by the launcher)
  bool general;     // couplings with several states per bath, a laser field or more than 24 states
};
// kind as launch_stage_vec (the FP32 body only for general runs); mup: [n][n] M+ on the host, or NULL.
int launch_el_stage(int kind, const ElStageArgs &a, const double *mup, cudaStream_t st, int sm_count);

// One run of an el_run_kernel launch, in the run's workspace.
struct ElRunDesc {
  StageCommon c;
  StateView st[3];  // y, zA, zB
  ElConsts k;
  unsigned *bar;    // [2] barrier counters, zero between launches
  const double *w;
  double *records;
  int64_t *rec_count;
  int64_t max_records;
  int fp64, pad;
};
struct ElEntry {
  const ElRunDesc *d;
  int cta0;                  // first CTA of the run
  int hcta;                  // CTAs of the FP64 part
  int apu64, split64, apu32;  // units of the FP64 part and of an FP32 body taken by elements
  int row_bytes;             // shared memory per warp of an FP32 body taken by rows
  int steps;
  int stride, first_rec;     // a record every stride steps, the first after first_rec steps (0: none)
};
// el_run_kernel for a mixed run of n states with a Hermitian state (nullptr: not compiled in the unit)
const void *mixed_run_kernel_a(int n);
const void *mixed_run_kernel_b(int n);
const void *mixed_run_kernel_c(int n);
constexpr int kElMaxRuns = 256;  // runs per launch (kernel parameters: about 10 KB)
struct ElList {
  ElEntry e[kElMaxRuns];
  double ch[4];  // the stages' Horner coefficients times h
  int nruns;
};

// Work-list launches (stage_list.cuh): one launch covers the same stage of the FP32 bodies of many runs of
// equal n_states (real H).  A run's stage arguments for such launches live in its workspace.
struct alignas(16) GroupArgs {
  StageCommon c;
  float ch;                           // Horner coefficient times h
  float term[kMaxStates];             // terminator Delta per state
  alignas(16) float H[kMaxStates * kMaxStates];   // Re H - h0 I, row stride kMaxStates, rad/fs
};
constexpr int kListMaxRuns = 64;  // runs per work-list launch (kernel parameters: about 0.8 KB)
struct ListLaunch {
  const GroupArgs *args[kListMaxRuns];  // arguments of run i for this stage (device)
  int item0[kListMaxRuns + 1];     // run i owns items [item0[i], item0[i + 1]) of cpi chunks each
  int nruns;
  int cpi;
};
// One work-list launch of runs of n states.  Returns 1 when n is not compiled in the unit.
int launch_stage_list(int n, const ListLaunch &L, cudaStream_t st, int sm_count);
int launch_stage_list_a(int n, const ListLaunch &L, cudaStream_t st, int sm_count);
int launch_stage_list_b(int n, const ListLaunch &L, cudaStream_t st, int sm_count);
int launch_stage_list_c(int n, const ListLaunch &L, cudaStream_t st, int sm_count);

// The FP64 heads of the same runs (resident.cuh): CTAs [cta0[i], cta0[i + 1]) take run i's units of apu ADOs, or (apu = 1)
// `splits` units of one ADO.
struct HeadList {
  const ElRunDesc *d[kListMaxRuns];
  int cta0[kListMaxRuns + 1];
  int nruns, n, herm, apu, splits;
  int stage;   // 0..3
  double ch;
};
int launch_head_list(const HeadList &L, cudaStream_t st);

// The FP32 body of a mixed run on the row kernels (stage_kernel.cuh).
int launch_stage(const StageCommon &c, double ch, const double *term, const double *H,
                 const double *Hi, cudaStream_t st, int sm_count);

}  // namespace heom
