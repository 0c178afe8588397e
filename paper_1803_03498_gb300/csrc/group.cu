// C ABI of libheom, part 5: heom_group_propagate -- many runs advanced together, the RK4 stages of
// small mixed-precision runs of equal n_states sharing work-list launches (stage_list.cuh).
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <cstring>
#include <map>
#include <string>
#include <vector>

#include "../../include/heom.h"
#include "heom_internal.h"
#include "heom_run.h"

using namespace heom;

namespace {

// Runs above this many body ADOs keep launches of their own: the work-list kernel reads H from
// shared memory instead of the constant bank, which costs at the sizes where one run fills the GPU.
constexpr int64_t kListRunMaxAdos = 200000;
// Chunks per work item: one per warp of the 4-warp FP32 body kernel, so that a small run spreads over as many
// CTAs as it has chunks -- at these sizes a launch is latency-bound.
constexpr int kListCpiBody = 4;

// The Horner stages of one RK4 step: input, base, output (horner_c: the coefficient).
struct HornerStage {
  int zin, y, out;  // 0 = y, 1 = zA, 2 = zB
};
constexpr HornerStage kHorner[4] = {{0, 0, 1}, {1, 0, 2}, {2, 0, 1}, {1, 0, 0}};

StateView view_of(const heom_run *r, int k) { return k == 0 ? r->y : (k == 1 ? r->zA : r->zB); }

bool list_eligible(const heom_run *r) {
  return r->precision == HEOM_FP32_MIXED && !r->vec && !r->gen && !r->has_field && !r->cplx_h && r->u_split > 0 &&
         r->n_ado - r->u_split <= kListRunMaxAdos;
}

}  // namespace

extern "C" int heom_group_propagate(heom_run *const *runs, int n_runs, double dt_fs, const int64_t *n_steps,
                                    int64_t obs_stride, void *cuda_stream) {
  if (!runs || n_runs < 0 || (n_runs > 0 && !n_steps) || !(dt_fs > 0) || obs_stride < 0) {
    set_error("heom_group_propagate: need runs, n_runs >= 0, n_steps, dt_fs > 0, obs_stride >= 0");
    return HEOM_E_ARG;
  }
  const double h = dt_fs;
  std::vector<heom_run *> rv(runs, runs + n_runs);
  {
    std::vector<heom_run *> sorted(rv);
    std::sort(sorted.begin(), sorted.end());
    if (std::adjacent_find(sorted.begin(), sorted.end()) != sorted.end()) {
      set_error("heom_group_propagate: a run is listed twice");
      return HEOM_E_ARG;
    }
  }
  int64_t max_steps = 0;
  for (int i = 0; i < n_runs; ++i) {
    heom_run *r = rv[i];
    if (!r || n_steps[i] < 0) {
      set_error("heom_group_propagate: NULL run or negative step count");
      return HEOM_E_ARG;
    }
    if (h * r->max_rate > 2.5) {
      set_error("heom_group_propagate: dt_fs * depth * max gamma > 2.5 for a run (RK4 unstable; the paper asks "
                "dt << 1/gamma_k)");
      return HEOM_E_ARG;
    }
    if (r->has_field) {
      set_error("heom_group_propagate: a run has a laser field (use heom_propagate)");
      return HEOM_E_STATE;
    }
    if (r->timing) {
      set_error("heom_group_propagate: a run has kernel timing on");
      return HEOM_E_STATE;
    }
    if (obs_stride > 0) {
      const int64_t first = obs_stride - (r->steps_done % obs_stride);
      const int64_t need = (n_steps[i] >= first) ? 1 + (n_steps[i] - first) / obs_stride : 0;
      if (r->records_host + need > r->max_records) {
        set_error("heom_group_propagate: observable records of a run would exceed its max_records");
        return HEOM_E_NOMEM;
      }
    }
    max_steps = std::max(max_steps, n_steps[i]);
  }
  if (n_runs == 0 || max_steps == 0) return HEOM_OK;
  cudaStream_t gs = reinterpret_cast<cudaStream_t>(cuda_stream);

  // order after the work already enqueued on every run's stream
  std::vector<cudaStream_t> streams;
  for (heom_run *r : rv)
    if (std::find(streams.begin(), streams.end(), r->stream) == streams.end()) streams.push_back(r->stream);
  std::vector<cudaEvent_t> evs(streams.size() + 1, nullptr);
  auto cleanup = [&]() {
    for (cudaEvent_t e : evs)
      if (e) cudaEventDestroy(e);
  };
  cudaError_t e = cudaSuccess;
  for (size_t k = 0; k < evs.size() && e == cudaSuccess; ++k) e = cudaEventCreateWithFlags(&evs[k], cudaEventDisableTiming);
  for (size_t k = 0; k < streams.size() && e == cudaSuccess; ++k) {
    if (streams[k] == gs) continue;
    e = cudaEventRecord(evs[k], streams[k]);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(gs, evs[k], 0);
  }
  if (e != cudaSuccess) {
    cleanup();
    return cuda_fail("heom_group_propagate: stream order", e);
  }

  // work-list arguments of the eligible runs
  std::vector<bool> listed(n_runs);
  for (int i = 0; i < n_runs; ++i) {
    listed[i] = list_eligible(rv[i]) && n_steps[i] > 0;
    if (listed[i]) {
      const int rc = el_group_args(rv[i], h, gs);
      if (rc != HEOM_OK) {
        cleanup();
        return rc;
      }
    }
  }

  int rc = HEOM_OK;
  // small FP64 runs: whole steps in shared launches (resident.cuh)
  std::vector<int64_t> left(n_steps, n_steps + n_runs);
  std::vector<ElShared> shared;
  if (!capturing(gs)) {
    std::vector<heom_run *> small;
    std::vector<int64_t> small_steps;
    bool others = false;
    int sm_count = 1;
    int64_t ctas = 0;
    for (int i = 0; i < n_runs; ++i) {
      if (n_steps[i] == 0) continue;
      if (listed[i] || rv[i]->precision != HEOM_FP64 || !el_small(rv[i])) {
        others = true;
        continue;
      }
      ctas += el_ctas(rv[i]);
      small.push_back(rv[i]);
      small_steps.push_back(n_steps[i]);
      left[i] = 0;
      sm_count = rv[i]->sm_count;
    }
    // Beside other runs, small ones that are content with a CTA on every other SM stay there: on all slots they kept
    // the others' stages waiting (680 ADOs of 7 states beside a mixed run of 11628: 7.1 ms for 60 steps, so 5.8,
    // one after the other 7.1).  Larger ones take all slots: held to a quarter of them, 3060 ADOs beside four mixed runs
    // took up to 14 ms against 11.
    const int cap = others && ctas <= sm_count / 2 ? sm_count / 2 : 2 * sm_count;
    if (!small.empty()) shared = el_split(small.data(), (int)small.size(), small_steps.data(), cap);
  }
  // Each size class and each kind of shared launches gets a stream of its own for the whole call (forked from and joined
  // back into the caller's stream): their launch chains run side by side, while the stages of one class
  // follow each other.  A run keeps its class, so its launches stay in order.
  std::vector<cudaStream_t> cls(kMaxStates + 1, nullptr), shs(shared.size(), nullptr);
  std::vector<cudaEvent_t> cls_ev;
  // one size class or kind and nothing else: its launches go straight to the caller's stream
  bool any = false, single = shared.size() <= 1;
  int n0 = -1;
  for (int i = 0; i < n_runs && single; ++i) {
    if (left[i] == 0) continue;
    any = true;
    if (n0 < 0) n0 = rv[i]->n;
    single = listed[i] && rv[i]->n == n0;
  }
  if (any && !shared.empty()) single = false;
  // a stream forked from the caller's in *out (the caller's, which may be the NULL stream, when the call
  // needs only one)
  auto fork_stream = [&](cudaStream_t *slot, cudaStream_t *out) -> int {
    *out = gs;
    if (single) return HEOM_OK;
    if (!*slot) {
      // the forked streams take the caller's priority, so that a high-priority caller's ticks stay ahead
      // of other streams' launches when SM slots free up
      cudaEvent_t fe = nullptr;
      int prio = 0;
      cudaError_t ce = cudaStreamGetPriority(gs, &prio);
      if (ce == cudaSuccess) ce = cudaStreamCreateWithPriority(slot, cudaStreamNonBlocking, prio);
      if (ce == cudaSuccess) ce = cudaEventCreateWithFlags(&fe, cudaEventDisableTiming);
      if (ce == cudaSuccess) cls_ev.push_back(fe);
      if (ce == cudaSuccess) ce = cudaEventRecord(fe, gs);
      if (ce == cudaSuccess) ce = cudaStreamWaitEvent(*slot, fe, 0);
      if (ce != cudaSuccess) return cuda_fail("heom_group_propagate: class stream", ce);
    }
    *out = *slot;
    return HEOM_OK;
  };
  // the caller's stream waits for what is on st so far
  auto join_stream = [&](cudaStream_t st) -> int {
    cudaEvent_t je = nullptr;
    cudaError_t ce = cudaEventCreateWithFlags(&je, cudaEventDisableTiming);
    if (ce == cudaSuccess) ce = cudaEventRecord(je, st);
    if (ce == cudaSuccess) ce = cudaStreamWaitEvent(gs, je, 0);
    if (je) cudaEventDestroy(je);
    return ce == cudaSuccess ? HEOM_OK : cuda_fail("heom_group_propagate: class stream join", ce);
  };
  for (size_t k = 0; k < shared.size() && rc == HEOM_OK; ++k) {
    ElShared &g = shared[k];
    std::vector<int64_t> goal;
    for (size_t q = 0; q < g.runs.size(); ++q) goal.push_back(g.runs[q]->steps_done + g.steps[q]);
    cudaStream_t st = gs;
    if ((rc = fork_stream(&shs[k], &st)) == HEOM_OK) rc = el_propagate(g, h, obs_stride, st);
    if (rc != kElNoRoom) continue;
    // a context too small for the launch: the steps that are left go with the others', after those enqueued
    rc = st == gs ? HEOM_OK : join_stream(st);
    for (size_t q = 0; q < g.runs.size(); ++q)
      left[std::find(rv.begin(), rv.end(), g.runs[q]) - rv.begin()] = goal[q] - g.runs[q]->steps_done;
  }
  // the work-list launches of one step, rebuilt only when a run's steps end: per class of equal
  // n_states and per batch of at most kListMaxRuns runs, the head and body launch of each stage
  struct Prepared {
    int n, sm_count;
    bool head;
    cudaStream_t stream;
    ListLaunch L[4];
    HeadList H;
    std::vector<heom_run *> members;
  };
  std::vector<Prepared> prep;
  int64_t rebuilt_at = -1;
  max_steps = *std::max_element(left.begin(), left.end());
  for (int64_t s = 0; s < max_steps && rc == HEOM_OK; ++s) {
    bool change = rebuilt_at < 0;
    for (int i = 0; i < n_runs && !change; ++i) change = listed[i] && left[i] == s;
    if (change) {
      std::map<int, std::vector<int>> classes;  // n_states -> listed runs still stepping
      for (int i = 0; i < n_runs; ++i)
        if (listed[i] && left[i] > s) classes[rv[i]->n].push_back(i);
      prep.clear();
      for (const auto &cl : classes) {
        cudaStream_t cs = gs;
        if ((rc = fork_stream(&cls[cl.first], &cs)) != HEOM_OK) break;
        // FP64 heads: Hermitian runs and others take different kernels
        for (int herm = 0; herm < 2; ++herm) {
          std::vector<heom_run *> hr;
          for (int i : cl.second)
            if ((rv[i]->herm ? 1 : 0) == herm) hr.push_back(rv[i]);
          for (size_t b0 = 0; b0 < hr.size(); b0 += kListMaxRuns) {
            Prepared p;
            p.n = cl.first;
            p.head = true;
            p.sm_count = hr[0]->sm_count;
            p.stream = cs;
            p.members.assign(hr.begin() + b0, hr.begin() + std::min(hr.size(), b0 + (size_t)kListMaxRuns));
            HeadList &L = p.H;
            L.nruns = (int)p.members.size();
            L.n = cl.first;
            L.herm = herm;
            L.cta0[0] = 0;
            for (int q = 0; q < L.nruns; ++q) {
              int ctas = 0;
              head_plan(p.members[q], &L.apu, &L.splits, &ctas);
              L.d[q] = reinterpret_cast<const ElRunDesc *>(p.members[q]->desc_dev);
              L.cta0[q + 1] = L.cta0[q] + ctas;
            }
            prep.push_back(std::move(p));
          }
        }
        for (size_t b0 = 0; b0 < cl.second.size(); b0 += kListMaxRuns) {
          const size_t b1 = std::min(cl.second.size(), b0 + (size_t)kListMaxRuns);
          Prepared p;
          p.n = cl.first;
          p.head = false;
          p.sm_count = rv[cl.second[b0]]->sm_count;
          p.stream = cs;
          for (int st = 0; st < 4; ++st) {
            ListLaunch &L = p.L[st];
            L.nruns = (int)(b1 - b0);
            L.cpi = kListCpiBody;
            L.item0[0] = 0;
            for (size_t q = b0; q < b1; ++q) {
              const heom_run *r = rv[cl.second[q]];
              const int A = 32 / r->n < 32 ? 32 / r->n : 31;
              const int64_t chunks = (r->n_ado - r->u_split + A - 1) / A;
              L.args[q - b0] = group_args_of(r) + st;
              L.item0[q - b0 + 1] = L.item0[q - b0] + (int)((chunks + L.cpi - 1) / L.cpi);
            }
          }
          for (size_t q = b0; q < b1; ++q) p.members.push_back(rv[cl.second[q]]);
          prep.push_back(std::move(p));
        }
      }
      rebuilt_at = s;
    }
    for (int st = 0; st < 4 && rc == HEOM_OK; ++st) {
      for (Prepared &p : prep) {
        if (p.head) {
          p.H.stage = st;
          p.H.ch = horner_c(st, h);
        }
        if (p.head ? launch_head_list(p.H, p.stream) : launch_stage_list(p.n, p.L[st], p.stream, p.sm_count)) {
          rc = HEOM_E_CUDA;
          break;
        }
        for (heom_run *r : p.members) ++r->launches;  // one work-list launch counts for each of its runs
      }
      // runs outside the work lists: their own launches, on the caller's stream
      for (int i = 0; i < n_runs && rc == HEOM_OK; ++i) {
        if (listed[i] || left[i] <= s) continue;
        heom_run *r = rv[i];
        const HornerStage &hs = kHorner[st];
        cudaStream_t own = r->stream;
        r->stream = gs;
        rc = run_stage(r, view_of(r, hs.zin), view_of(r, hs.y), view_of(r, hs.out), horner_c(st, h));
        r->stream = own;
      }
    }
    for (int i = 0; i < n_runs && rc == HEOM_OK; ++i) {  // step counters and observable records
      if (left[i] <= s) continue;
      heom_run *r = rv[i];
      ++r->steps_done;
      r->t_fs += h;
      if (obs_stride > 0 && r->steps_done % obs_stride == 0) {
        cudaStream_t own = r->stream;
        r->stream = (listed[i] && !single) ? cls[r->n] : gs;  // after the run's own stage launches
        rc = enqueue_record(r);
        r->stream = own;
      }
    }
  }
  // join the forked streams back into the caller's stream
  cls.insert(cls.end(), shs.begin(), shs.end());
  for (cudaStream_t st : cls) {
    if (!st) continue;
    const int jr = join_stream(st);
    if (rc == HEOM_OK) rc = jr;
    cudaStreamDestroy(st);  // released once its work is done
  }
  for (cudaEvent_t fe : cls_ev) cudaEventDestroy(fe);

  // later work on every run's stream is ordered after this call's launches
  e = cudaEventRecord(evs.back(), gs);
  for (size_t k = 0; k < streams.size() && e == cudaSuccess; ++k)
    if (streams[k] != gs) e = cudaStreamWaitEvent(streams[k], evs.back(), 0);
  cleanup();
  if (rc != HEOM_OK) return rc;
  return e == cudaSuccess ? HEOM_OK : cuda_fail("heom_group_propagate: stream order", e);
}
