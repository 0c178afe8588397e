// Whole RK4 steps of one small column-0 run in one cooperative launch (sm_103a).
//
// A linear-absorption run stores column 0 of every ADO (vec_kernel.cuh states its right-hand side).  At a few thousand
// ADOs a stage is all latency: launched stage by stage it took 9 us (FP64 head and FP32 body launches, fork and join)
// for work of well under one.  Here every element (ADO u, state a) belongs to one thread for the whole launch:
// x, y, its decay and the first records of its state stay in registers, H and the columns of the CTA's ADOs in
// shared memory, and a stage is one round trip to L2 for the neighbour elements and one barrier of the CTAs (see
// el_barrier).  CTAs [0, hcta) take the FP64 part (the head of a mixed run, or every ADO), the others the FP32 body.  Each
// sum has the terms and the order of vec_step, so the results equal its launches' bit for bit.
#pragma once
#include "vec_kernel.cuh"

namespace heom {

constexpr int kColThreads = 256;
constexpr int kColSlots = 4;

struct ColRunArgs {
  ElRunDesc d;
  double ch[4];                        // the stages' Horner coefficients times h
  int hcta, apu64, apu32;              // CTAs of the FP64 part; ADOs per CTA of either part
  int steps, stride, first_rec;        // as ElEntry
  double term[kMaxStates];
  double H[kMaxStates * kMaxStates];   // stride kMaxStates
};

// Element s of ADO v's column, past the L1 cache.
template <typename CT, typename BT>
__device__ __forceinline__ typename VCplx<CT>::type col_fetch(const StateView &s, int n, int u_split, int v, int e) {
  typename VCplx<CT>::type r;
  if (v < u_split) {
    const double2 d = __ldcg(s.head + (int64_t)v * n + e);
    r.x = (CT)d.x;
    r.y = (CT)d.y;
  } else {
    const auto b = __ldcg(reinterpret_cast<const typename VCplx<BT>::type *>(s.body) + (int64_t)(v - u_split) * n + e);
    r.x = (CT)b.x;
    r.y = (CT)b.y;
  }
  return r;
}

// Shared memory of a CTA: H by columns, the CTA's columns twice (stages alternate), record ranges.
__host__ __device__ inline size_t col_smem_bytes(int n, int ados, size_t real) {
  return ((((size_t)n * n * real + 15) & ~(size_t)15) + 4 * (size_t)ados * n * real + 4 * (size_t)ados * n + 15) & ~(size_t)15;
}

// One part of the run (CT, BT as vec_step) for all steps; first: the CTA's first ADO, cnt of them.
template <typename CT, typename BT>
__device__ __forceinline__ void col_run_part(const ColRunArgs &a, unsigned char *sm, int apu, int first, int cnt, int rank,
                                             int ncta) {
  using C2 = typename VCplx<CT>::type;
  constexpr bool kOwnHead = sizeof(CT) == 8 && sizeof(BT) == 4;
  const StageCommon &c = a.d.c;
  const int n = c.n, t = threadIdx.x;
  CT *H = reinterpret_cast<CT *>(sm);  // H[b n + i] = H_ib
  C2 *xs = reinterpret_cast<C2 *>(sm + (((size_t)n * n * sizeof(CT) + 15) & ~(size_t)15));
  uint32_t *rng = reinterpret_cast<uint32_t *>(xs + 2 * apu * n);
  for (int e = t; e < n * n; e += kColThreads) H[e] = (CT)a.H[(e % n) * kMaxStates + e / n];
  for (int e = t; e < apu * n; e += kColThreads) rng[e] = 0;
  __syncthreads();
  const int64_t rbase = kOwnHead ? 0 : c.rec_split;
  const LinkRec<CT> *recs0 = reinterpret_cast<const LinkRec<CT> *>(kOwnHead ? c.recs_head : c.recs_body);
  for (int la = t >> 5; la < cnt; la += kColThreads / 32) {  // record ranges, a warp for each ADO
    const int64_t lo = c.link_off[first + la];
    const int nrec = heom_rec_batch(c.err, lo, (int)(c.link_off[first + la + 1] - lo), rbase, kOwnHead ? c.rec_split : c.n_recs);
    const LinkRec<CT> *r = recs0 + (lo - rbase);
    uint16_t *half = reinterpret_cast<uint16_t *>(rng);
    for (int k = t & 31; k < nrec; k += 32) {
      const int s = r[k].s & kRecStateMask;
      if (!HEOM_IN_RANGE(c.err, s, 0, n)) continue;
      if (k == 0 || (r[k - 1].s & kRecStateMask) != s) half[2 * (la * n + s)] = (uint16_t)k;
      if (k + 1 == nrec || (r[k + 1].s & kRecStateMask) != s) half[2 * (la * n + s) + 1] = (uint16_t)(k + 1);
    }
  }
  __syncthreads();
  const int la = t / n, li = t - la * n, u = first + la;
  const bool have = la < cnt;
  const CT h00 = (CT)a.H[0];
  C2 x, y;
  x.x = x.y = y.x = y.y = 0;
  CT f = 0;
  int nq = 0;
  const LinkRec<CT> *r = recs0;
  LinkRec<CT> rec[kColSlots];
  if (have) {
    x = col_fetch<CT, BT>(a.d.st[0], n, c.u_split, u, li);
    f = (CT)c.gsum[u] + (CT)a.term[li];
    const uint32_t q = rng[la * n + li];
    nq = (int)(q >> 16) - (int)(q & 0xffff);
    r = recs0 + (c.link_off[u] - rbase) + (q & 0xffff);
#pragma unroll
    for (int k = 0; k < kColSlots; ++k)
      if (k < nq) {
        rec[k] = r[k];
        if (!HEOM_IN_RANGE(c.err, rec[k].v, 0, c.n_ado)) rec[k].v = 0;
      }
  }
  unsigned target = 0;
  int due = a.first_rec;
  C2 *cur = xs;
  for (int step = 0; step < a.steps; ++step) {
#pragma unroll 1
    for (int q = 0; q < 4; ++q) {
      const StateView zin = a.d.st[q == 0 ? 0 : q == 2 ? 2 : 1], out = a.d.st[q == 3 ? 0 : q == 1 ? 2 : 1];
      const CT ch = (CT)a.ch[q];
      C2 v[kColSlots];
      if (have) {
#pragma unroll
        for (int k = 0; k < kColSlots; ++k)
          if (k < nq) v[k] = col_fetch<CT, BT>(zin, n, c.u_split, rec[k].v, li);
        if (q == 0) y = x;
        cur[t] = x;
      }
      __syncthreads();
      if (have) {
        CT rr = -h00 * x.y, ri = h00 * x.x;
        const C2 *col = cur + la * n;
        const CT *h = H + li;
#pragma unroll 4
        for (int b = 0; b < n; ++b) {
          const C2 xb = col[b];
          rr = fma(h[b * n], xb.y, rr);
          ri = fma(-h[b * n], xb.x, ri);
        }
        rr = fma(-f, x.x, rr);
        ri = fma(-f, x.y, ri);
        auto link = [&](const LinkRec<CT> &k, const C2 &w) {
          const CT cr = fma(k.re, w.x, -k.im * w.y), ci = fma(k.re, w.y, k.im * w.x);
          rr += cr;
          ri += ci;
        };
#pragma unroll
        for (int k = 0; k < kColSlots; ++k)
          if (k < nq) link(rec[k], v[k]);
        for (int k = kColSlots; k < nq; ++k) {
          const LinkRec<CT> m = r[k];
          if (HEOM_IN_RANGE(c.err, m.v, 0, c.n_ado)) link(m, col_fetch<CT, BT>(zin, n, c.u_split, m.v, li));
        }
        x.x = fma(ch, rr, y.x);
        x.y = fma(ch, ri, y.y);
        if constexpr (kOwnHead) __stcg(out.head + (int64_t)u * n + li, make_double2(x.x, x.y));
        else __stcg(reinterpret_cast<C2 *>(out.body) + (int64_t)(u - c.u_split) * n + li, x);
      }
      cur = cur == xs ? xs + apu * n : xs;
      target += ncta;
      if (!el_barrier(a.d.bar, target, c.err)) return;
    }
    if (due > 0 && --due == 0) {  // sigma_0 stays as it is until the last stage of the next step
      if (rank == ncta - 1 && t < 32)
        record_warp(a.d.st[0], c.u_split, !a.d.fp64, 1, n, a.d.w, a.d.records, a.d.rec_count, a.d.max_records);
      due = a.stride;
    }
  }
  __syncthreads();
  if (t == 0) {  // the last CTA to leave clears the counters for the next launch
    __threadfence();
    if (atomicAdd(a.d.bar + 1, 1u) == (unsigned)ncta - 1) {
      a.d.bar[0] = 0;
      a.d.bar[1] = 0;
      __threadfence();
    }
  }
}

__global__ void __launch_bounds__(kColThreads, 2) col_run_kernel(const __grid_constant__ ColRunArgs a) {
  extern __shared__ __align__(16) unsigned char el_sm[];
  // an earlier launch of this run gave up: the whole CTA leaves, whatever each of its threads reads
  if (__syncthreads_or(*(volatile int *)a.d.c.err & kErrTimeout)) return;
  const int rank = blockIdx.x, ncta = gridDim.x, n64 = a.d.fp64 ? a.d.c.n_ado : a.d.c.u_split;
  if (rank < a.hcta) {
    const int first = rank * a.apu64, cnt = max(0, min(a.apu64, n64 - first));
    if (a.d.fp64) col_run_part<double, double>(a, el_sm, a.apu64, first, cnt, rank, ncta);
    else col_run_part<double, float>(a, el_sm, a.apu64, first, cnt, rank, ncta);
  } else {
    const int first = a.d.c.u_split + (rank - a.hcta) * a.apu32, cnt = max(0, min(a.apu32, a.d.c.n_ado - first));
    col_run_part<float, float>(a, el_sm, a.apu32, first, cnt, rank, ncta);
  }
}

}  // namespace heom
