// Launchers of the element kernels (resident.cuh): single stages, and whole RK4 steps of one or many runs.
#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstring>
#include <string>

#include "../../include/heom.h"
#include "heom_internal.h"
#include "heom_run.h"
#include "resident.cuh"
#include "column_run.cuh"

namespace heom {

namespace {

// Shared memory of a CTA of el_run_kernel: two CTAs per SM (228 KB less 1 KB per CTA and the static part).
constexpr size_t kElSmemMax = 110u << 10;
// Steps per launch: long enough that the launch (about 10 us with the drain of the one before) is noise, short
// enough that work on other streams gets the SMs again within about kElLaunchMs.
constexpr int kElSteps = 64;
constexpr double kElLaunchMs = 2.0;

int max_smem(const void *f, const char *what) {
  const cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kElSmemMax);
  if (e == cudaSuccess) return 0;
  set_error(std::string(what) + ": shared memory attribute: " + cudaGetErrorString(e));
  return -4;
}

// ADOs of tile pitch `pitch` whose tiles and link ranges fit beside the constants in `budget` bytes, at
// most 32 (a record names its ADO by u mod 32).
int fit_ados(int n, int pitch, int pairs, size_t real_bytes, bool general, size_t budget) {
  int k = 32;
  while (k > 1 && el_smem_bytes(n, k, pitch, pairs, real_bytes, general) > budget) --k;
  return k;
}

template <typename CT, typename BT, int FORM, bool CPLX>
int launch_stage_kind(const ElStageArgs &a, const double *mup, cudaStream_t st, int sm_count) {
  const auto kern = el_stage_kernel<CT, BT, FORM, CPLX>;
  static std::atomic<bool> ready{false};
  if (!ready) {
    const int rc = max_smem((const void *)kern, "element stage kernel");
    if (rc) return rc;
    ready = true;
  }
  const StageCommon &c = a.c;
  const bool own_head = sizeof(CT) == 8 && sizeof(BT) == 4;
  const int P = el_pairs(c.n, c.herm), pitch = own_head ? c.E : c.Ep;
  const size_t smem = el_smem_bytes(c.n, a.apu, pitch, P, sizeof(CT), true);
  const int64_t units = ((int64_t)(c.u_end - c.u_begin) + a.apu - 1) / a.apu * a.splits;
  static std::atomic<int> by_regs{0};  // CTAs per SM that the registers allow; shared memory below
  cudaError_t e = cudaSuccess;
  if (by_regs == 0) {
    int ps = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&ps, kern, kElThreads, 0);
    if (e != cudaSuccess || ps < 1) {
      set_error(std::string("element stage kernel: occupancy query failed or zero blocks: ") + cudaGetErrorString(e));
      return -4;
    }
    by_regs = ps;
  }
  const int per_sm = std::max(1, std::min((int)by_regs, (int)((227u << 10) / (smem + 1024))));
  const int grid = (int)std::max<int64_t>(1, std::min<int64_t>(units, (int64_t)sched_ctas(per_sm, c.occ_pct) * sm_count));
  ElMup<CPLX> m{};
  if constexpr (CPLX)
    if (mup) std::copy(mup, mup + (size_t)c.n * c.n, m.v);
  kern<<<grid, kElThreads, smem, st>>>(a, m, mup != nullptr);
  e = cudaGetLastError();
  if (e == cudaSuccess) return 0;
  set_error(std::string("element stage kernel launch: ") + cudaGetErrorString(e));
  return -4;
}

}  // namespace

// Hermitian runs with a real H and one state per bath, up to kLeanMaxStates states.
bool lean_covers(int n, int herm, int cplx, bool general) { return herm && !cplx && !general && n <= kLeanMaxStates; }

namespace {
template <typename BT, bool FIXED>
int launch_lean(const ElStageArgs &a, cudaStream_t st, int sm_count) {
  static std::atomic<int> by_regs{0};
  cudaError_t e = cudaSuccess;
  if (by_regs == 0) {
    int ps = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&ps, lean_stage_kernel<BT, FIXED>, kLeanThreads, 0);
    if (e != cudaSuccess || ps < 1) {
      set_error(std::string("pair stage kernel: occupancy query failed or zero blocks: ") + cudaGetErrorString(e));
      return -4;
    }
    by_regs = ps;
  }
  const int n_ado = a.c.u_end - a.c.u_begin;
  ElStageArgs x = a;
  // fewer ADOs per CTA where there are not enough for every CTA slot
  x.apu = std::max(1, std::min(lean_ados(a.c.n, kLeanThreads), n_ado / (2 * sm_count)));
  const int chunks = (n_ado + x.apu - 1) / x.apu;
  const size_t smem = lean_smem_bytes(a.c.n, x.apu, 0);  // below 48 KB
  const int grid = std::max(1, std::min(chunks, sched_ctas(by_regs, a.c.occ_pct) * sm_count));
  lean_stage_kernel<BT, FIXED><<<grid, kLeanThreads, smem, st>>>(x);
  e = cudaGetLastError();
  if (e == cudaSuccess) return 0;
  set_error(std::string("pair stage kernel launch: ") + cudaGetErrorString(e));
  return -4;
}
}  // namespace

int launch_el_stage(int kind, const ElStageArgs &in, const double *mup, cudaStream_t st, int sm_count) {
  ElStageArgs a = in;
  const StageCommon &c = a.c;
  const int n_ado = c.u_end - c.u_begin;
  if (n_ado <= 0) return 0;
  if (kind != 1 && lean_covers(c.n, c.herm, c.cplx_h, a.general)) {
    // the part of the run, not of the launch, decides (see lean_fixed)
    const bool fixed = kind == 0 ? lean_fixed(c.n, c.n_ado) : lean_head_fixed(c.n);
    if (kind == 0) return fixed ? launch_lean<double, true>(a, st, sm_count) : launch_lean<double, false>(a, st, sm_count);
    return fixed ? launch_lean<float, true>(a, st, sm_count) : launch_lean<float, false>(a, st, sm_count);
  }
  const size_t rb = kind == 1 ? 4 : 8;
  const int P = el_pairs(c.n, c.herm), pitch = kind == 2 ? c.E : c.Ep;
  // units of about two rounds of the CTA's threads; fewer ADOs than CTA slots (2 per SM) take smaller units, and
  // fewer ADOs than SMs split each ADO's elements, so that the FP64 pipes of all SMs take part
  a.splits = 1;
  a.apu = std::max(1, std::min(2 * kElThreads / P, fit_ados(c.n, pitch, P, rb, true, kElSmemMax / 2)));
  a.apu = std::max(1, std::min(a.apu, n_ado / (2 * sm_count)));
  if (n_ado < 2 * sm_count) a.splits = std::max(1, std::min(2 * sm_count / n_ado, P / 64));
  const bool cplx = c.cplx_h || mup;
  // Up to 4 states 4 n (8 n) FMAs are as fast as the splitting, whose steps follow each other (general runs of 4 states, 15 ADOs
  // 38 us per step against 47; heads of complex mixed runs of 2 states 33.5 against 37).  Only runs that never
  // take whole steps, so that both forms of launch of the others give the same bits.
  const bool chain = c.n < 5 && (a.general || (kind == 2 && c.cplx_h));
  auto go = [&](auto CT, auto BT, auto FORM) {
    using C = decltype(CT);
    using B = decltype(BT);
    return cplx ? launch_stage_kind<C, B, FORM.value, true>(a, mup, st, sm_count) : launch_stage_kind<C, B, FORM.value, false>(a, mup, st, sm_count);
  };
  const std::integral_constant<int, kElFixed> fixed;
  const std::integral_constant<int, kElGeneral> fma;
  switch (kind) {
    case 0: return chain ? go(0.0, 0.0, fma) : go(0.0, 0.0, fixed);
    case 1: return go(0.f, 0.f, fma);
    default: return chain ? go(0.0, 0.f, fma) : go(0.0, 0.f, fixed);
  }
}

int launch_head_list(const HeadList &L, cudaStream_t st) {
  const bool lean = lean_covers(L.n, L.herm, 0, false);
  const int ctas = L.cta0[L.nruns];
  if (ctas <= 0) return 0;
  const size_t smem = lean ? lean_smem_bytes(L.n, L.apu, 0)
                           : el_smem_bytes(L.n, L.apu, L.n * L.n, el_pairs(L.n, L.herm), 8, true);
  if (lean) {
    if (lean_head_fixed(L.n)) head_list_kernel<true, true><<<ctas, kElThreads, smem, st>>>(L);
    else head_list_kernel<true, false><<<ctas, kElThreads, smem, st>>>(L);
  } else {
    static std::atomic<bool> ready{false};
    if (!ready) {
      const int rc = max_smem((const void *)head_list_kernel<false, true>, "head list kernel");
      if (rc) return rc;
      ready = true;
    }
    head_list_kernel<false, true><<<ctas, kElThreads, smem, st>>>(L);
  }
  const cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess) return 0;
  set_error(std::string("head list kernel launch: ") + cudaGetErrorString(e));
  return -4;
}

// ---- constants and descriptor of a run, in its workspace -----------------------------------------------

static const char kElTag = 0;  // desc_owner of runs whose descriptor area holds an ElRunDesc

static size_t desc_bytes(int n) { return 512 + ((size_t)3 * n * n + n) * sizeof(double); }
// The work-list arguments of the four stages follow (grouped runs: at most kMaxStates states).
constexpr size_t kGroupArgsAt = (512 + (3 * kMaxStates * kMaxStates + kMaxStates) * sizeof(double) + 15) & ~(size_t)15;
static_assert(kGroupArgsAt + 4 * sizeof(GroupArgs) <= 8 * sizeof(VecRunDesc), "the descriptor area holds them");
static_assert(sizeof(ElRunDesc) <= 512, "descriptor header");
static_assert(512 + (3 * kGenMaxStates * kGenMaxStates + kGenMaxStates) * sizeof(double) <= 8 * sizeof(VecRunDesc),
              "the descriptor area holds the element kernels' constants");

ElConsts el_consts_of(const heom_run *r) {
  const double *k = reinterpret_cast<const double *>(reinterpret_cast<const char *>(r->desc_dev) + 512);
  const size_t E = (size_t)r->n * r->n;
  return ElConsts{k, k + E, k + 2 * E, nullptr, k + 3 * E};
}

// The run's constants and descriptor (matrix layout), enqueued on the run's stream; the host data is pageable and
// small, so it is consumed when the copy returns.
int el_upload(heom_run *r) {
  const size_t E = (size_t)r->n * r->n;
  std::vector<char> buf(desc_bytes(r->n), 0);
  ElRunDesc d{};
  const StateView none{nullptr, nullptr};
  d.c = common_for(r, none, none, none);
  d.st[0] = r->y;
  d.st[1] = r->zA;
  d.st[2] = r->zB;
  d.k = el_consts_of(r);
  d.bar = r->bar_dev;
  d.w = r->w_dev;
  d.records = r->records;
  d.rec_count = r->rec_count;
  d.max_records = r->max_records;
  d.fp64 = r->precision == HEOM_FP64;
  std::memcpy(buf.data(), &d, sizeof(d));
  double *k = reinterpret_cast<double *>(buf.data() + 512);
  std::copy(r->H.begin(), r->H.end(), k);
  std::copy(r->Hi.begin(), r->Hi.end(), k + E);
  for (int i = 0; i < r->n; ++i)
    for (int j = 0; j < r->n; ++j)
      k[2 * E + (size_t)i * r->n + j] = r->gen ? r->T[(size_t)i * r->n + j] : i != j ? r->term[i] + r->term[j] : 0.0;
  std::copy(r->term.begin(), r->term.end(), k + 3 * E);
  const cudaError_t e = cudaMemcpyAsync(r->desc_dev, buf.data(), buf.size(), cudaMemcpyHostToDevice, r->stream);
  if (e != cudaSuccess) return cuda_fail("stage constants upload", e);
  r->desc_owner = &kElTag;
  r->group_dt = 0;  // the area may have held something else
  return HEOM_OK;
}

static bool run_lean(const heom_run *r) { return lean_covers(r->n, r->herm, r->cplx_h, r->gen); }

const GroupArgs *group_args_of(const heom_run *r) {
  return reinterpret_cast<const GroupArgs *>(reinterpret_cast<const char *>(r->desc_dev) + kGroupArgsAt);
}

// The run's work-list arguments for time step h, written on stream s unless they are there already.
int el_group_args(heom_run *r, double h, cudaStream_t s) {
  if (r->group_dt == h && r->group_herm == r->herm) return HEOM_OK;
  std::vector<GroupArgs> g(4);
  std::memset(static_cast<void *>(g.data()), 0, 4 * sizeof(GroupArgs));
  const StateView st[3] = {r->y, r->zA, r->zB};
  for (int q = 0; q < 4; ++q) {
    g[q].c = common_for(r, st[q == 0 ? 0 : q == 2 ? 2 : 1], r->y, st[q == 3 ? 0 : q == 1 ? 2 : 1]);
    g[q].c.u_begin = r->u_split;
    g[q].c.u_end = (int)r->n_ado;
    g[q].c.occ_pct = r->sched[0].occupancy_pct;
    g[q].c.cpw = r->sched[0].chunks_per_warp;
    g[q].ch = (float)horner_c(q, h);
    for (int i = 0; i < r->n; ++i) g[q].term[i] = (float)r->term[i];
    for (int i = 0; i < r->n; ++i)
      for (int j = 0; j < r->n; ++j) g[q].H[i * kMaxStates + j] = (float)r->H[(size_t)i * r->n + j];
  }
  const cudaError_t e = cudaMemcpyAsync(const_cast<GroupArgs *>(group_args_of(r)), g.data(), 4 * sizeof(GroupArgs),
                                        cudaMemcpyHostToDevice, s);
  if (e != cudaSuccess) return cuda_fail("heom_group_propagate: stage arguments", e);
  r->group_dt = h;
  r->group_herm = r->herm;
  return HEOM_OK;
}

// ADOs per CTA and parts per ADO of a head of u_split ADOs in a list launch, and its CTAs: a head has few ADOs, so
// each CTA takes as few as fill its SM partitions.
void head_plan(const heom_run *r, int *apu, int *splits, int *ctas) {
  const int P = el_pairs(r->n, r->herm);
  *apu = std::max(1, std::min(128 / P, 32));
  *splits = 1;
  if (!run_lean(r) && P > 256) *splits = P / 128;
  *ctas = (r->u_split + *apu - 1) / *apu * *splits;
}

// ---- whole steps -------------------------------------------------------------------------------------

namespace {

// Rough cycles of one stage of a run on one SM: the FP64 part (fixed-point commutator, then about 18 FP64
// instructions per 32 elements at 18.7 cycles) and the FP32 body (rows: cycles per chunk as the row kernel
// measures them, 1250 for one ADO of 19 states; elements otherwise).
double cost64(const heom_run *r) {
  const double ados = r->precision == HEOM_FP64 ? (double)r->n_ado : (double)r->u_split;
  return ados * el_pairs(r->n, r->herm) * ((r->cplx_h ? 0.7 : 0.35) * r->n + 12.0);
}
double cost32(const heom_run *r) {
  if (r->precision == HEOM_FP64) return 0;
  const double ados = (double)(r->n_ado - r->u_split);
  if (!r->herm) return ados * r->n * r->n * (0.3 * r->n + 4.0);
  const int a = 32 / r->n < 32 ? 32 / r->n : 31;
  return std::ceil(ados / a) * (200.0 + 2.6 * r->n * r->n * a);
}
int row_bytes(int n) {
  int b = 0;
  row_dispatch<1, kMaxStates>(n, [&](auto N) { b = RowSmem<N.value>::total; });
  return b;
}

// A CTA's share of one stage below which another CTA costs more (barrier, tile traffic) than it takes off.
constexpr double kElGrain = 1500.0;

// Whether one CTA takes a whole run: its barrier is then a __syncthreads.  The head and the body of a mixed run follow each
// other there, so only the smallest stay in one (us per step in one CTA and in two: 2 states, 70 ADOs 31.7 and 25.5;
// 3 states, 56 ADOs 26.2 and 21.7, from a coherence 48.2 and 39.5; 2 states, 6 ADOs 20.8 and 18.1).
bool one_cta(const heom_run *r) {
  const double cost = cost64(r) + cost32(r);
  return cost <= (cost32(r) > 0 ? 0.3 : 2.0) * kElGrain;
}

struct ElShare {
  int n64, n32;  // CTAs of the FP64 part and of the body (1, 1: one CTA for both)
};

// CTAs for a run out of at most `cap` (at least 1).
ElShare share_of(const heom_run *r, int cap) {
  const double a = cost64(r), b = cost32(r);
  const int64_t n64 = r->precision == HEOM_FP64 ? r->n_ado : r->u_split, nb = r->n_ado - n64;
  const int P = el_pairs(r->n, r->herm);
  if (cap <= 1 || one_cta(r)) return ElShare{1, nb > 0 ? 1 : 0};
  // the most CTAs each part can use: an element kernel splits an FP64 ADO down to 64 pairs
  const double max64 = (double)n64 * (run_lean(r) ? 1 : std::max(1, P / 64)), max32 = (double)nb;
  double w64 = std::min(std::max(1.0, a / kElGrain), max64), w32 = nb > 0 ? std::min(std::max(1.0, b / kElGrain), max32) : 0.0;
  // a body taken by elements: a unit of 32 ADOs (the most that its records tell apart) for each CTA at the least, for a CTA builds
  // the link ranges of every further unit again in every stage (2 states, 126 ADOs in one CTA 66 us per step, in four 32)
  if (nb > 0 && !r->herm) w32 = std::max(w32, std::ceil((double)nb / 32));
  if (w64 + w32 > cap) {
    // a head keeps the CTAs that it can use, up to a quarter: an ADO of 17 to 22 states takes one about 10 us, so
    // two after each other in a CTA hold the body's CTAs at the barrier
    const double f = cap / (a + b);
    w64 = std::max(1.0, nb > 0 ? std::min(w64, std::max(a * f, 0.25 * cap)) : std::min(max64, a * f));
    if (nb > 0) w32 = std::max(1.0, std::min(max32, cap - std::floor(w64)));
    w64 = std::min(max64, cap - std::floor(w32));
  }
  return ElShare{(int)w64, (int)w32};
}

}  // namespace

// Small hierarchies: their work of one stage, spread over the GPU, takes at most a few tens of microseconds.
// FP64 runs of this size take the element kernels in every form of launch (the others the column kernel, where
// it covers them); FP32 bodies get the same bits from the element and the row kernels.
// Where the column kernel covers a run, it takes less per ADO but P passes for a warp's first chunk (P = 1 for 8 and 16 states,
// 3 for 12, 7 for 14, 11 for 11), each about 1.1 us per state: the line is kElColPass P N.  Measured on both sides, us per step
// whole / column: 8 states, 1287 ADOs 29 / 51, 12870 195 / 165; 10, 8008 192 / 264, 19448 436 / 345; 11, 12376 370 / 578, 31824
// 1014 / 795; 12, 6188 201 / 216, 18564 614 / 487; 14, 11628 572 / 586, 38760 1955 / 1304; 16, 969 107 / 100, 4845 409 / 238.
// Elsewhere stage launches of the same kernels come level at kElMaxCost64: 7 states, 19448 ADOs 218 / 228,
// 31824 345 / 345; 18 states, 1330 ADOs 159 / 171, 7315 774 / 763.
// Mixed runs, whole steps / stage launches: up to kElMaxCost32 (about 6400 ADOs of 7 or 8 states, 3600 of 12) 7 states, 6435 ADOs
// 33 / 42; 8, 6435 34 / 37; 10, 3003 32 / 42; 13, 2380 36 / 50; from a coherence 7, 3432 57 / 66, 6435 87 / 66.  From 16 states on the row
// form spills at this kernel's 128 registers, and the lines lie lower: 16 states, 153 ADOs 35 / 42, 969 52 / 46; 17, 171 37 / 45,
// 630 52 / 51 (a third of the limit); 19, 210 50 / 49; 22, 276 62 / 50 (from 19 on only heads without a body).
bool el_small(const heom_run *r) {
  if (r->vec || r->gen) return false;
  if (r->precision == HEOM_FP64) return cost64(r) <= (r->herm && !r->cplx_h && col_covers(r->n) ? kElColPass * col_passes(r->n) * r->n : kElMaxCost64);
  if (r->precision != HEOM_FP32_MIXED || r->cplx_h || r->u_split <= 0) return false;
  if (r->n_ado == r->u_split || !r->herm) return cost32(r) <= kElMaxCost32;
  return r->n <= kElMaxRows && cost32(r) <= (r->n >= 16 ? kElMaxCost32 / 3 : kElMaxCost32);
}

// A cooperative launch that this context cannot hold at once (fewer SMs than the device has): it was not enqueued, and the
// caller takes the steps that the runs' counters still lack stage by stage.
static bool no_room(cudaError_t e) {
  if (e != cudaErrorCooperativeLaunchTooLarge && e != cudaErrorNotSupported) return false;
  cudaGetLastError();
  return true;
}

// CTAs that an FP64 run needs to be kept (kRunKept).
static int kept_ctas(const heom_run *r) {
  const int a = lean_ados(r->n, kLeanRunThreads);
  return (int)((r->n_ado + a - 1) / a);
}

// ADOs per unit, at most `fit`, of a part of `ados` ADOs on `ctas` CTAs: every CTA gets the same number of units, none nearly
// empty.  (Units as large as fit: 11628 non-Hermitian ADOs of 7 states were 364 units on 304 CTAs, two rounds for work of
// little more than one; 467 us per step against 356 stage by stage before.)
static int even_units(int64_t ados, int ctas, int fit) {
  const int64_t per = (ados + ctas - 1) / ctas, rounds = (per + fit - 1) / fit;
  return (int)((per + rounds - 1) / rounds);
}

// The forms of el_run_kernel (kind, fixed, states of the row form) and their kernels.
// 0..3: kept, chunks; 5: mixed without a body; 8 + n: mixed of n states
constexpr int kFormOther = 4, kFormHead = 5, kFormMixed = 8, kForms = kFormMixed + kElMaxRows + 1;
static int form_of(const heom_run *r, bool kept) {
  if (!run_lean(r)) return kFormOther;
  if (r->precision != HEOM_FP64) return r->n <= kElMaxRows ? kFormMixed + r->n : kFormHead;
  return (kept ? 0 : 2) + (lean_fixed(r->n, r->n_ado) ? 1 : 0);
}
static const void *form_kernel(int form) {
  switch (form) {
    case 0: return (const void *)el_run_kernel<kRunKept, false, 0>;
    case 1: return (const void *)el_run_kernel<kRunKept, true, 0>;
    case 2: return (const void *)el_run_kernel<kRunChunks, false, 0>;
    case 3: return (const void *)el_run_kernel<kRunChunks, true, 0>;
    case kFormOther: return (const void *)el_run_kernel<kRunOther, true, 0>;
    case kFormHead: return (const void *)el_run_kernel<kRunMixed, true, 0>;
  }
  const int n = form - kFormMixed;
  const void *k = mixed_run_kernel_a(n);
  if (!k) k = mixed_run_kernel_b(n);
  if (!k) k = mixed_run_kernel_c(n);
  return k;
}

// Every run of g by its number of steps on stream s, in as few launches as possible; the runs' counters
// (steps_done, t_fs, records_host, launches) advance, also where it stops with kElNoRoom.
int el_propagate(const ElShared &g, double h, int64_t stride, cudaStream_t s) {
  const int form = g.form, n_runs = (int)g.runs.size(), cap = g.cap;
  heom_run *const *runs = g.runs.data();
  const int64_t *steps = g.steps.data();
  static std::atomic<bool> ready[kForms];
  const void *kernel = form_kernel(form);
  if (!kernel) {
    set_error("element run kernel: n_states not compiled");
    return HEOM_E_CUDA;
  }
  if (!ready[form]) {
    const int rc = max_smem(kernel, "element run kernel");
    if (rc) return HEOM_E_CUDA;
    ready[form] = true;
  }
  const bool kept_form = form < 2;
  const int threads = kept_form ? kLeanRunThreads : kElThreads;
  int64_t most = 0;
  for (int i = 0; i < n_runs; ++i) most = std::max(most, steps[i]);
  const int per_launch = std::min(kElMaxRuns, cap);  // a CTA for each run
  for (int b0 = 0; b0 < n_runs; b0 += per_launch) {
    const int b1 = std::min(n_runs, b0 + per_launch);
    int64_t k = 0;
    for (int64_t at = 0; at < most; at += k) {
      ElList L;
      for (int q = 0; q < 4; ++q) L.ch[q] = horner_c(q, h);
      L.nruns = 0;
      std::vector<int> in;
      double total = 0;
      int want = 0, kept = 0;
      for (int i = b0; i < b1; ++i)
        if (steps[i] > at) {
          in.push_back(i);
          total += cost64(runs[i]) + cost32(runs[i]);
          if (kept_form) kept += kept_ctas(runs[i]);
          const ElShare w = share_of(runs[i], cap);
          want += one_cta(runs[i]) ? 1 : w.n64 + w.n32;
        }
      if (in.empty()) break;
      size_t smem = 0;
      int cta = 0;
      double longest = 0;  // the longest CTA's cycles in one stage
      for (size_t q = 0; q < in.size(); ++q) {
        heom_run *r = runs[in[q]];
        const double cost = cost64(r) + cost32(r);
        // everything each run can use, or its share of the CTAs by cost, one at least for each that follows
        int mine = cap;
        if (kept_form) {
          mine = kept_ctas(r) + (int)(cost / total * (cap - kept));
        } else if (want > cap) {
          const int left = cap - cta - (int)(in.size() - q - 1);
          mine = std::max(1, std::min(left, (int)(cost / total * (cap - (int)in.size())) + 1));
        }
        const ElShare w = share_of(r, mine);
        const bool fp64 = r->precision == HEOM_FP64;
        const int64_t n64 = fp64 ? r->n_ado : r->u_split, nb = r->n_ado - n64;
        const int P = el_pairs(r->n, r->herm), pitch64 = fp64 ? r->Ep : r->E;
        // a kept run spreads until its CTAs have a warp for each partition of their SM (FP64 instructions of
        // one warp follow each other 64 clocks apart, whatever the other partitions do)
        const int64_t kept_h = std::min<int64_t>(r->n_ado, std::max<int64_t>(kept_ctas(r), std::min<int64_t>(mine, (r->n_ado * P + 127) / 128)));
        const bool one = kept_form ? kept_h == 1 : mine <= 1 || one_cta(r);
        const int h64 = kept_form ? (int)kept_h : one ? 1 : w.n64, h32 = one ? 1 : w.n32;
        ElEntry &e = L.e[L.nruns++];
        e.d = reinterpret_cast<const ElRunDesc *>(r->desc_dev);
        e.cta0 = cta;
        e.hcta = h64;
        const size_t room = one && !fp64 ? kElSmemMax / 6 : kElSmemMax;
        e.apu64 = even_units(n64, h64, run_lean(r) ? lean_ados(r->n, threads) : fit_ados(r->n, pitch64, P, 8, true, room));
        e.split64 = n64 < h64 ? std::max(1, std::min(h64 / (int)n64, P / 64)) : 1;
        e.apu32 = nb > 0 ? even_units(nb, h32, fit_ados(r->n, r->Ep, P, 4, false, room)) : 1;
        longest = std::max(longest, one ? cost : std::max(cost64(r) / h64, cost32(r) / std::max(1, h32)));
        e.row_bytes = nb > 0 && r->herm ? row_bytes(r->n) : 0;
        const size_t m64 = run_lean(r) ? lean_smem_bytes(r->n, e.apu64, kept_form ? threads : 0)
                                       : el_smem_bytes(r->n, e.apu64, pitch64, P, 8, true);
        const size_t m32 = nb <= 0 ? 0 : r->herm ? sizeof(RowConsts) + (size_t)e.row_bytes * (kElThreads / 32)
                                               : el_smem_bytes(r->n, e.apu32, r->Ep, P, 4, false);
        smem = std::max(smem, one ? m64 + m32 : std::max(m64, m32));
        cta += one ? 1 : h64 + (nb > 0 ? h32 : 0);
      }
      const double step_ms = 4 * (2.5e-3 + longest / 1.9e6);
      k = std::max<int64_t>(1, std::min<int64_t>(kElSteps, (int64_t)(kElLaunchMs / step_ms)));
      for (size_t q = 0; q < in.size(); ++q) {
        ElEntry &e = L.e[q];
        e.steps = (int)std::min<int64_t>(k, steps[in[q]] - at);
        e.stride = (int)std::min<int64_t>(stride, 1 << 30);
        e.first_rec = 0;
        if (stride > 0) {
          const int64_t first = stride - runs[in[q]]->steps_done % stride;
          e.first_rec = first <= e.steps ? (int)first : 0;
        }
      }
      void *args[] = {&L};
      cudaError_t ce = cudaLaunchCooperativeKernel(kernel, dim3(cta), dim3(threads), args, smem, s);
      if (ce == cudaSuccess) ce = cudaGetLastError();
      if (no_room(ce)) return kElNoRoom;
      if (ce != cudaSuccess) return cuda_fail("element run kernel launch", ce);
      for (size_t q = 0; q < in.size(); ++q) {
        heom_run *r = runs[in[q]];
        const int64_t m = L.e[q].steps;
        if (stride > 0) r->records_host += (r->steps_done + m) / stride - r->steps_done / stride;
        r->steps_done += m;
        for (int64_t x = 0; x < m; ++x) r->t_fs += h;
        ++r->launches;
      }
    }
  }
  return HEOM_OK;
}

int64_t el_ctas(const heom_run *r) { return run_lean(r) ? kept_ctas(r) : 1 + (int64_t)(cost64(r) / (4 * kElGrain)); }

// The runs by their form of launch, each with a share by cost of `cap` CTAs (at most 2 per SM: launch bounds and
// kElSmemMax), so that launches on streams of their own fit the GPU beside each other.
std::vector<ElShared> el_split(heom_run *const *runs, int n_runs, const int64_t *steps, int cap) {
  std::vector<ElShared> out;
  auto add = [&](int form, int i) {
    for (ElShared &g : out)
      if (g.form == form) {
        g.runs.push_back(runs[i]);
        g.steps.push_back(steps[i]);
        return;
      }
    out.push_back(ElShared{form, 0, {runs[i]}, {steps[i]}});
  };
  for (int i = 0; i < n_runs; ++i) add(form_of(runs[i], true), i);
  double total = 0;
  for (int i = 0; i < n_runs; ++i) total += cost64(runs[i]) + cost32(runs[i]);
  for (ElShared &g : out) {
    double cost = 0;
    int need = 0;  // CTAs that keep the runs
    for (const heom_run *r : g.runs) {
      cost += cost64(r) + cost32(r);
      if (g.form < 2) need += kept_ctas(r);
    }
    g.cap = std::max(1, std::min(cap, (int)(cap * cost / total + 0.5)));
    if (g.form < 2 && need > g.cap) g.form += 2;
  }
  return out;
}

// ---- column-0 runs --------------------------------------------------------------------------------------

// CTAs and ADOs per CTA of a part of `ados` ADOs: an element per thread.
static void col_part(int n, int64_t ados, int *ctas, int *apu) {
  *apu = std::max(1, kColThreads / n);
  *ctas = (int)((ados + *apu - 1) / *apu);
}

// Column-0 runs whose elements have a thread each on the GPU (two CTAs of 256 per SM): up to 77,824 elements, e.g. 9,700
// ADOs of 8 states.  FP64 parts are held to four warps per SM, where their pipe is no bound yet.
bool col_small(const heom_run *r) {
  if (!r->vec) return false;
  const int64_t n64 = r->precision == HEOM_FP64 ? r->n_ado : r->u_split;
  int c64, c32, apu;
  col_part(r->n, n64, &c64, &apu);
  col_part(r->n, r->n_ado - n64, &c32, &apu);
  return (int64_t)c64 + c32 <= 2 * (int64_t)r->sm_count && n64 * r->n <= 128 * (int64_t)r->sm_count;
}

int col_propagate(heom_run *r, double h, int64_t steps, int64_t stride, cudaStream_t s) {
  ColRunArgs a{};
  const StateView none{nullptr, nullptr};
  ElRunDesc &d = a.d;
  d.c = common_for(r, none, none, none);
  d.st[0] = r->y;
  d.st[1] = r->zA;
  d.st[2] = r->zB;
  d.bar = r->bar_dev;
  d.w = r->w_dev;
  d.records = r->records;
  d.rec_count = r->rec_count;
  d.max_records = r->max_records;
  d.fp64 = r->precision == HEOM_FP64;
  for (int q = 0; q < 4; ++q) a.ch[q] = horner_c(q, h);
  for (int i = 0; i < r->n; ++i) {
    a.term[i] = r->term[i];
    for (int j = 0; j < r->n; ++j) a.H[i * kMaxStates + j] = r->H[(size_t)i * r->n + j];
  }
  const int64_t n64 = d.fp64 ? r->n_ado : r->u_split;
  int c32;
  col_part(r->n, n64, &a.hcta, &a.apu64);
  col_part(r->n, r->n_ado - n64, &c32, &a.apu32);
  // a short FP64 part spreads further: its warps wait for their SM partition's pipe
  if (!d.fp64) {
    const int spread = std::max(1, 2 * r->sm_count - c32), per = std::max<int>(1, (int)((n64 + spread - 1) / spread));
    a.apu64 = std::min(a.apu64, std::max(per, std::max(1, 128 / r->n)));
    a.hcta = (int)((n64 + a.apu64 - 1) / a.apu64);
  }
  const size_t smem = std::max(col_smem_bytes(r->n, a.apu64, 8), col_smem_bytes(r->n, a.apu32, 4));  // below 48 KB
  for (int64_t at = 0; at < steps;) {
    a.steps = (int)std::min<int64_t>(kElSteps * 2, steps - at);  // about a millisecond
    a.stride = (int)std::min<int64_t>(stride, 1 << 30);
    a.first_rec = 0;
    if (stride > 0) {
      const int64_t first = stride - r->steps_done % stride;
      a.first_rec = first <= a.steps ? (int)first : 0;
    }
    void *args[] = {&a};
    cudaError_t e = cudaLaunchCooperativeKernel((const void *)col_run_kernel, dim3(a.hcta + c32), dim3(kColThreads), args, smem, s);
    if (e == cudaSuccess) e = cudaGetLastError();
    if (no_room(e)) return kElNoRoom;
    if (e != cudaSuccess) return cuda_fail("column run kernel launch", e);
    if (stride > 0) r->records_host += (r->steps_done + a.steps) / stride - r->steps_done / stride;
    r->steps_done += a.steps;
    for (int x = 0; x < a.steps; ++x) r->t_fs += h;
    ++r->launches;
    at += a.steps;
  }
  return HEOM_OK;
}

}  // namespace heom
