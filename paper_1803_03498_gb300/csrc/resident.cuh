// Element kernels (sm_103a): every thread owns element pairs of ADOs, and a small hierarchy keeps its
// threads for many RK4 steps.
//
// The right-hand side of Eq. HEOM (arXiv 1803.03498, section "HEOM formalism", with the ADO rescaling;
// hbar = 1, energies in rad/fs) is local in the element index except for the commutator: element (i, j)
// of ADO u needs row i and column j of its own tile, and of every linked neighbour v only the same
// element v_ij, with coefficient R for a link through a mode of state i and conj(R) for one of state j
// (both: 2 Re R; see LinkRec).  So a thread computes one element -- for a Hermitian run one pair
// (i <= j), whose mirror element it also writes, half the work and exactly Hermitian results -- with
// its neighbour loads independent of each other: no chain from link to link, which is what bound the
// FP64 row kernels once used at these sizes (one warp-synchronised step per link; 24 us per launch for 3060 ADOs
// of 7 x 7, 18.7 us for 680, 58 us for the 20 FP64 head ADOs of a 19-state run).  Pairs of consecutive
// ADOs are numbered through, so every lane has work for every n_states, and the pairs of one ADO can be
// split over CTAs on different SMs: GB300's FP64 pipe (18.7 clocks per warp FMA and SM) bounds these kernels, and
// the few FP64 head ADOs of a mixed run (1 + M of them) then use the pipes of all SMs.
//
// Two forms of launch run the same code, so results do not depend on the form:
//  - el_stage_kernel: one stage (zin, base, out, coefficient) of a range of ADOs; also the two-output form
//    of classic RK4 with a time-dependent H(t), and couplings with several states per bath;
//  - el_run_kernel: whole RK4 steps of one or many runs in one cooperative launch.  Each run has CTAs
//    of its own that keep their ADOs, constants and link ranges in shared memory; a barrier of the
//    run's CTAs (a counter in the run's workspace) follows every stage.  A stage then costs one barrier
//    and one round trip to L2 instead of a kernel launch or two.
// Arithmetic forms (FORM): kElFixed -- FP64 runs and heads, the commutator in fixed point (fixed_point.cuh);
// kElGeneral -- FP32 runs of the general kind; kElRowOrder -- FP32 non-Hermitian runs in el_run_kernel, every
// sum in the order of stage_kernel's shared-memory path, so that the results equal that kernel's bit for
// bit (FP32 Hermitian bodies there run the row kernel's own code, row_body).
//
#pragma once
#include <cuda_runtime.h>

#include <cstdint>
#include <type_traits>

#include "fixed_point.cuh"
#include "heom_internal.h"
#include "record.cuh"
#include "stage_kernel.cuh"

namespace heom {

constexpr int kElGeneral = 0, kElFixed = 1, kElRowOrder = 2;

template <typename T>
struct ECplx;
template <>
struct ECplx<float> {
  using type = float2;
};
template <>
struct ECplx<double> {
  using type = double2;
};

__device__ __forceinline__ void el_cp16(void *smem, const void *gmem) {
  const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(s), "l"(gmem) : "memory");
}
__device__ __forceinline__ void el_cp_wait() {
  asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;\n" ::: "memory");
}

// Element e of ADO v, past the L1 cache (other CTAs of the same launch wrote it).
template <typename CT, typename BT>
__device__ __forceinline__ typename ECplx<CT>::type el_fetch(const StateView &s, const StageCommon &c, int v, int e) {
  typename ECplx<CT>::type r;
  if (v < c.u_split) {
    const double2 d = __ldcg(s.head + (int64_t)v * c.E + e);
    r.x = (CT)d.x;
    r.y = (CT)d.y;
  } else {
    const auto b = __ldcg(reinterpret_cast<const typename ECplx<BT>::type *>(s.body) + (int64_t)(v - c.u_split) * c.Ep + e);
    r.x = (CT)b.x;
    r.y = (CT)b.y;
  }
  return r;
}

template <typename CT>
struct ElRec {  // a link record without its padding
  int v;
  CT re, im;
};
template <typename CT>
__device__ __forceinline__ ElRec<CT> el_rec(const LinkRec<CT> *p);
template <>
__device__ __forceinline__ ElRec<float> el_rec<float>(const LinkRec<float> *p) {
  const int4 w = __ldg(reinterpret_cast<const int4 *>(p));
  return ElRec<float>{w.x, __int_as_float(w.z), __int_as_float(w.w)};
}
template <>
__device__ __forceinline__ ElRec<double> el_rec<double>(const LinkRec<double> *p) {
  const double2 w = __ldg(reinterpret_cast<const double2 *>(p) + 1);
  return ElRec<double>{__ldg(&p->v), w.x, w.y};
}

// Shared memory of one part (FP64 or FP32) of a CTA: constants, pair table, link ranges, tiles.
template <typename CT>
struct ElSmem {
  using C2 = typename ECplx<CT>::type;
  CT *H, *Hi, *T, *term;
  C2 *tile;
  uint32_t *rng;     // [cnt][n] records of (ADO, state): begin | end << 16, relative to the chunk's first
  int2 *rest;        // [cnt][pitch] the tiles' third limbs, Re and Im (fixed point)
  int2 *hrest;       // [n][n] those of H and Im H
  double2 *hd;       // [n][n] H and Im H in FP64, for the FMA chain
  int *key;          // [cnt][2] largest |Re|, |Im| of an ADO's tile: FP64 high word (fixed point)
  int *hkey;         // the same of H
  uint16_t *pair;    // element p of an ADO: i << 8 | j
  unsigned char *end;
};

// Bytes of ElSmem for `cnt` ADOs of tile pitch `pitch`; general: with Im H and the T matrix.
__host__ __device__ inline size_t el_smem_bytes(int n, int cnt, int pitch, int pairs, size_t real_bytes, bool general) {
  size_t b = 0;
  b += ((general ? 3 : 1) * (size_t)n * n + n) * real_bytes;
  b = (b + 15) & ~(size_t)15;
  b += (size_t)cnt * pitch * 2 * real_bytes;
  b = (b + 15) & ~(size_t)15;
  if (real_bytes == 8) b += ((((size_t)cnt * pitch + (size_t)n * n) * 8 + 15) & ~(size_t)15) + (size_t)n * n * 16;  // third limbs, hd
  b += (size_t)cnt * n * 4 + (size_t)cnt * 8 + 16 + (size_t)pairs * 2;
  return (b + 15) & ~(size_t)15;
}

template <typename CT>
__device__ __forceinline__ ElSmem<CT> el_carve(unsigned char *p, int n, int cnt, int pitch, int pairs, bool general) {
  using C2 = typename ECplx<CT>::type;
  ElSmem<CT> s;
  CT *q = reinterpret_cast<CT *>(p);
  s.H = q;
  q += n * n;
  s.Hi = s.T = q;
  if (general) {
    s.T = q + n * n;
    q += 2 * n * n;
  }
  s.term = q;
  q += n;
  uintptr_t a = (reinterpret_cast<uintptr_t>(q) + 15) & ~(uintptr_t)15;
  s.tile = reinterpret_cast<C2 *>(a);
  a = (a + (size_t)cnt * pitch * sizeof(C2) + 15) & ~(uintptr_t)15;
  s.rest = reinterpret_cast<int2 *>(a);
  s.hrest = s.rest + (size_t)cnt * pitch;
  if (sizeof(CT) == 8) a = (a + ((size_t)cnt * pitch + (size_t)n * n) * 8 + 15) & ~(uintptr_t)15;
  s.hd = reinterpret_cast<double2 *>(a);
  if (sizeof(CT) == 8) a += (size_t)n * n * 16;
  s.rng = reinterpret_cast<uint32_t *>(a);
  s.key = reinterpret_cast<int *>(s.rng + cnt * n);  // then the key of H
  s.pair = reinterpret_cast<uint16_t *>(s.key + 2 * cnt + 4);
  a = (reinterpret_cast<uintptr_t>(s.pair + pairs) + 15) & ~(uintptr_t)15;
  s.end = reinterpret_cast<unsigned char *>(a);
  s.hkey = s.key + 2 * cnt;
  return s;
}

__host__ __device__ inline int el_pairs(int n, int herm) { return herm ? n * (n + 1) / 2 : n * n; }

// Constants and the pair table into shared memory (followed by a __syncthreads of the caller).
// gr, gi: the laser field's g(t) (0 without a field): H(t) = H - g M+ - conj(g) (M+)^T.
template <typename CT>
__device__ __forceinline__ void el_consts(const ElSmem<CT> &s, const ElConsts &k, int n, int herm, bool general,
                                          double gr, double gi) {
  for (int e = threadIdx.x; e < n * n; e += blockDim.x) {
    double h = k.H[e];
    if (general) {
      double hi = k.Hi[e];
      if (k.mup) {
        const int i = e / n, j = e - i * n;
        const double a = k.mup[e], b = k.mup[j * n + i];
        h = h - gr * (a + b);
        hi = hi - gi * a + gi * b;
      }
      s.Hi[e] = (CT)hi;
      s.T[e] = (CT)k.T[e];
    }
    s.H[e] = (CT)h;
  }
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    s.term[i] = (CT)k.term[i];
    // row i of the pair table: (i, j) for j >= i (Hermitian) or every j
    const int j0 = herm ? i : 0, first = herm ? i * n - i * (i - 1) / 2 : i * n;
    for (int j = j0; j < n; ++j) s.pair[first + j - j0] = (uint16_t)(i << 8 | j);
  }
}

// H (and Im H) from FP64 to limbs, in place, after el_consts and a __syncthreads; followed by another.
template <bool CPLX>
__device__ __forceinline__ void el_fix_consts(const ElSmem<double> &s, int n) {
  if (threadIdx.x == 0) *s.hkey = 0;
  __syncthreads();
  int key = 0;
  for (int e = threadIdx.x; e < n * n; e += blockDim.x) {
    key = max(key, fx_key(s.H[e]));
    if (CPLX) key = max(key, fx_key(s.Hi[e]));
  }
  key = __reduce_max_sync(0xffffffffu, key);
  if ((threadIdx.x & 31) == 0) atomicMax(s.hkey, key);
  __syncthreads();
  const int ex = fx_exp(*s.hkey);
  for (int e = threadIdx.x; e < n * n; e += blockDim.x) {
    int2 rest = make_int2(0, 0);
    s.hd[e] = make_double2(s.H[e], CPLX ? s.Hi[e] : 0.0);
    reinterpret_cast<int2 *>(s.H)[e] = fx_split(s.H[e], ex, rest.x);
    if (CPLX) reinterpret_cast<int2 *>(s.Hi)[e] = fx_split(s.Hi[e], ex, rest.y);
    s.hrest[e] = rest;
  }
}

// The tiles of a chunk from FP64 to limbs, in place (element: Re hi, Re lo, Im hi, Im lo), with the key of each part.
template <bool CPLX>
__device__ __forceinline__ void el_fix_tiles(const ElSmem<double> &s, int n, int cnt, int pitch) {
  for (int t = threadIdx.x; t < 2 * cnt; t += blockDim.x) s.key[t] = 0;
  __syncthreads();
  const int total = cnt * pitch;
  for (int e0 = 0; e0 < total; e0 += blockDim.x) {
    const int e = e0 + threadIdx.x;
    const bool ok = e < total;
    const double2 z = ok ? s.tile[e] : make_double2(0, 0);
    const int la = ok ? e / pitch : -1;
    int kx = fx_key(z.x), ky = fx_key(z.y);
    if (CPLX) kx = ky = max(kx, ky);  // Re and Im mix: one scale
    const int first = __shfl_sync(0xffffffffu, la, 0);
    if (__all_sync(0xffffffffu, la == first)) {
      kx = __reduce_max_sync(0xffffffffu, kx);
      ky = __reduce_max_sync(0xffffffffu, ky);
      if ((threadIdx.x & 31) == 0 && first >= 0) {
        atomicMax(&s.key[2 * first], kx);
        atomicMax(&s.key[2 * first + 1], ky);
      }
    } else if (ok) {
      atomicMax(&s.key[2 * la], kx);
      atomicMax(&s.key[2 * la + 1], ky);
    }
  }
  __syncthreads();
  for (int e = threadIdx.x; e < total; e += blockDim.x) {
    const int la = e / pitch;
    const double2 z = s.tile[e];
    int2 rest;
    const int2 a = fx_split(z.x, fx_exp(s.key[2 * la]), rest.x), b = fx_split(z.y, fx_exp(s.key[2 * la + 1]), rest.y);
    reinterpret_cast<int4 *>(s.tile)[e] = make_int4(a.x, a.y, b.x, b.y);
    s.rest[e] = rest;
  }
  __syncthreads();
}

// C = H z - z H of element (i, j) of ADO u from the limbs; bits 0 and 1 of the result: Re C, Im C is weak (fx_weak).
template <bool CPLX>
__device__ __forceinline__ int el_fix_comm(const ElSmem<double> &s, int n, int la, int pitch, int i, int j, double &cr,
                                           double &ci) {
  FxSum r, m;
  const int4 *z = reinterpret_cast<const int4 *>(s.tile) + la * pitch;
  const int4 *zi = z + i * n, *zj = z + j;
  const int2 *wi = s.rest + la * pitch + i * n, *wj = s.rest + la * pitch + j;
  const int2 *hi_ = reinterpret_cast<const int2 *>(s.H) + i * n, *hj = reinterpret_cast<const int2 *>(s.H) + j;
  const int2 *gi_ = reinterpret_cast<const int2 *>(s.Hi) + i * n, *gj = reinterpret_cast<const int2 *>(s.Hi) + j;
  const int2 *vi = s.hrest + i * n, *vj = s.hrest + j;
#pragma unroll 2
  for (int k = 0; k < n; ++k) {
    const int4 a = zj[k * n], b = zi[k];
    const int2 ar = wj[k * n], br = wi[k];
    const int2 h1 = hi_[k], h2 = hj[k * n], r1 = vi[k], r2 = vj[k * n];
    r.add(h1.x, h1.y, r1.x, a.x, a.y, ar.x);
    m.add(h1.x, h1.y, r1.x, a.z, a.w, ar.y);
    const int nx = -h2.x, ny = -h2.y, nr = -r2.x;
    r.add(nx, ny, nr, b.x, b.y, br.x);
    m.add(nx, ny, nr, b.z, b.w, br.y);
    if constexpr (CPLX) {
      const int2 g1 = gi_[k], g2 = gj[k * n];
      r.add(-g1.x, -g1.y, -r1.y, a.z, a.w, ar.y);
      m.add(g1.x, g1.y, r1.y, a.x, a.y, ar.x);
      r.add(g2.x, g2.y, r2.y, b.z, b.w, br.y);
      m.add(-g2.x, -g2.y, -r2.y, b.x, b.y, br.x);
    }
  }
  return fx_finish(r, m, *s.hkey, s.key[2 * la], s.key[2 * la + 1], cr, ci);
}

// C = H z - z H of element (i, j) by FP64 FMAs; h: H and Im H in shared memory, z: the ADO's tile in global memory.  (With
// H read from global memory and H(t) put together in every term the first steps of a pulse, where many sums are
// weak, took a third longer.)
template <bool CPLX>
__device__ __noinline__ double2 el_fma_comm(const double2 *h, const double2 *z, int n, int i, int j) {
  double ar = 0, ai = 0, br = 0, bi = 0;
#pragma unroll 4
  for (int k = 0; k < n; ++k) {
    const double2 a = __ldcg(z + k * n + j), b = __ldcg(z + i * n + k);
    const double2 h1 = h[i * n + k], h2 = h[k * n + j];
    ar = fma(h1.x, a.x, ar);
    ai = fma(h1.x, a.y, ai);
    br = fma(b.x, h2.x, br);
    bi = fma(b.y, h2.x, bi);
    if (CPLX) {
      ar = fma(-h1.y, a.y, ar);
      ai = fma(h1.y, a.x, ai);
      br = fma(-b.y, h2.y, br);
      bi = fma(b.x, h2.y, bi);
    }
  }
  return make_double2(ar - br, ai - bi);
}

// Link ranges of the chunk [u0, u0 + cnt), cnt <= 32, records [lo, hi) at recs (already offset): a record
// names its ADO (u mod 32) and state, and the records of an ADO are ordered by state.
template <typename CT>
__device__ __forceinline__ void el_ranges(const ElSmem<CT> &s, const StageCommon &c, const LinkRec<CT> *recs, int nrec,
                                          int u0, int cnt) {
  for (int t = threadIdx.x; t < cnt * c.n; t += blockDim.x) s.rng[t] = 0;
  __syncthreads();
  uint16_t *half = reinterpret_cast<uint16_t *>(s.rng);  // little endian: begin first
  for (int t = threadIdx.x; t < nrec; t += blockDim.x) {
    const int sw = __ldg(&recs[t].s);
    const int o = (((sw >> 8) - u0) & 31) * c.n + (sw & kRecStateMask);
    if (!HEOM_IN_RANGE(c.err, sw & kRecStateMask, 0, c.n) || !HEOM_IN_RANGE(c.err, o, 0, cnt * c.n)) continue;
    if (t == 0 || __ldg(&recs[t - 1].s) != sw) half[2 * o] = (uint16_t)t;
    if (t + 1 == nrec || __ldg(&recs[t + 1].s) != sw) half[2 * o + 1] = (uint16_t)(t + 1);
  }
}

// Where a stage reads and writes.
struct ElStage {
  StateView zin, y, out, y2, out2;  // y / y2: base (none: null); out2: second output (null: none)
  double c1, c2;
};

__device__ __forceinline__ bool el_set(const StateView &v) { return v.head != nullptr || v.body != nullptr; }

template <typename CT, typename BT, bool OWN_HEAD>
__device__ __forceinline__ typename ECplx<CT>::type *el_own(const StateView &s, const StageCommon &c, int u) {
  using C2 = typename ECplx<CT>::type;
  if constexpr (OWN_HEAD) return reinterpret_cast<C2 *>(s.head) + (int64_t)u * c.E;
  else return reinterpret_cast<C2 *>(s.body) + (int64_t)(u - c.u_split) * c.Ep;
}

// Elements [p0, p1) (numbered through the ADOs) of the chunk [u0, u0 + cnt) of one stage, by the whole CTA.
// build: the link ranges are not in shared memory yet.  CPLX: H has an imaginary part.  TWO: a second output.
template <typename CT, typename BT, int FORM, bool CPLX, bool TWO>
__device__ __forceinline__ void el_unit(const ElSmem<CT> &s, const StageCommon &c, const ElStage &g, int u0, int cnt,
                                        int p0, int p1, bool build) {
  using C2 = typename ECplx<CT>::type;
  constexpr bool OWN_HEAD = sizeof(CT) == 8 && sizeof(BT) == 4;
  constexpr int PF = 4;  // neighbour elements loaded ahead of the commutator
  const int n = c.n, pitch = OWN_HEAD ? c.E : c.Ep;
  const bool herm = c.herm != 0;
  const int P = el_pairs(n, herm);
  const int64_t rbase = OWN_HEAD ? 0 : c.rec_split;
  const int64_t lo = c.link_off[u0];
  const LinkRec<CT> *recs = reinterpret_cast<const LinkRec<CT> *>(OWN_HEAD ? c.recs_head : c.recs_body) + (lo - rbase);
  {  // own tiles, one contiguous block
    const char *src = reinterpret_cast<const char *>(el_own<CT, BT, OWN_HEAD>(g.zin, c, u0));
    char *dst = reinterpret_cast<char *>(s.tile);
    const int bytes = cnt * pitch * (int)sizeof(C2);
    for (int o = threadIdx.x * 16; o < bytes; o += blockDim.x * 16) el_cp16(dst + o, src + o);
  }
  if (build) {
    const int nrec = heom_rec_batch(c.err, lo, (int)(c.link_off[u0 + cnt] - lo), rbase,
                                    OWN_HEAD ? c.rec_split : c.n_recs);
    el_ranges<CT>(s, c, recs, nrec, u0, cnt);
    __syncthreads();
  }
  const bool has_y = el_set(g.y), has2 = TWO && el_set(g.out2), has_y2 = TWO && el_set(g.y2);
  const CT c1 = (CT)g.c1, c2 = (CT)g.c2;
  bool landed = false;
  for (int t0 = p0; t0 < p1; t0 += blockDim.x) {
    const int t = t0 + (int)threadIdx.x;
    const bool have = t < p1;
    int la = 0, i = 0, j = 0;
    ElRec<CT> rec[PF];
    C2 v[PF];
    // the element's records: those of state i (coefficient R), then those of state j (conj R); slot q
    // of the nq in all
    int ib = 0, ni = 0, jb = 0, nq = 0;
    C2 yv, y2v, zij;
    yv.x = yv.y = y2v.x = y2v.y = zij.x = zij.y = 0;
    if (have) {
      la = t / P;
      const int pr = s.pair[t - la * P];
      i = pr >> 8;
      j = pr & 255;
      const uint32_t qi = s.rng[la * n + i], qj = s.rng[la * n + j];
      ib = qi & 0xffff;
      ni = (int)(qi >> 16) - ib;
      nq = ni + (int)(qj >> 16) - (int)(qj & 0xffff);
      jb = (int)(qj & 0xffff) - ni;
      if constexpr (FORM != kElRowOrder) {
#pragma unroll
        for (int q = 0; q < PF; ++q)
          if (q < nq) rec[q] = el_rec<CT>(recs + (q < ni ? ib : jb) + q);
#pragma unroll
        for (int q = 0; q < PF; ++q) {
          v[q].x = v[q].y = 0;
          if (q < nq && HEOM_IN_RANGE(c.err, rec[q].v, 0, c.n_ado)) v[q] = el_fetch<CT, BT>(g.zin, c, rec[q].v, i * n + j);
        }
      }
      const int e = i * n + j;
      zij = __ldcg(el_own<CT, BT, OWN_HEAD>(g.zin, c, u0 + la) + e);
      if (has_y) yv = __ldcg(el_own<CT, BT, OWN_HEAD>(g.y, c, u0 + la) + e);
      if (has_y2) y2v = __ldcg(el_own<CT, BT, OWN_HEAD>(g.y2, c, u0 + la) + e);
    }
    if (!landed) {  // the tiles
      el_cp_wait();
      __syncthreads();
      if constexpr (FORM == kElFixed) el_fix_tiles<CPLX>(s, n, cnt, pitch);
      landed = true;
    }
    if (!have) continue;
    const C2 *z = s.tile + la * pitch;
    const CT gs = (CT)__ldg(c.gsum + u0 + la);
    CT rr, ri;
    if constexpr (FORM != kElRowOrder) {
      CT cr = 0, ci = 0;  // C = H z - z H
      if constexpr (FORM == kElFixed) {
        int chain = 3;
        if (fx_ok(*s.hkey, s.key[2 * la]) && fx_ok(*s.hkey, s.key[2 * la + 1]))
          chain = el_fix_comm<CPLX>(s, n, la, pitch, i, j, cr, ci);
        if (herm && i == j) chain &= 2;  // Re C = 0 there and is not used
        if (chain) {
          const double2 x = el_fma_comm<CPLX>(s.hd, el_own<CT, BT, OWN_HEAD>(g.zin, c, u0 + la), n, i, j);
          if (chain & 1) cr = x.x;
          if (chain & 2) ci = x.y;
        }
      } else {
        CT ar = 0, ai = 0, br = 0, bi = 0;
        const CT *hi_ = s.H + i * n, *hj = s.H + j;
        const C2 *zi = z + i * n, *zj = z + j;
        const CT *gi_ = s.Hi + i * n, *gj = s.Hi + j;
#pragma unroll 2
        for (int k = 0; k < n; ++k) {
          const C2 a = zj[k * n], b = zi[k];
          const CT h1 = hi_[k], h2 = hj[k * n];
          ar = fma(h1, a.x, ar);
          ai = fma(h1, a.y, ai);
          br = fma(b.x, h2, br);
          bi = fma(b.y, h2, bi);
          if constexpr (CPLX) {
            const CT g1 = gi_[k], g2 = gj[k * n];
            ar = fma(-g1, a.y, ar);
            ai = fma(g1, a.x, ai);
            br = fma(-b.y, g2, br);
            bi = fma(b.x, g2, bi);
          }
        }
        cr = ar - br;
        ci = ai - bi;
      }
      const CT f = gs + s.T[i * n + j];
      rr = fma(-f, zij.x, ci);  // -i C
      ri = fma(-f, zij.y, -cr);
      auto link = [&](const ElRec<CT> &r, const C2 &x, bool row) {  // R v_ij or conj(R) v_ij
        const CT im = row ? r.im : -r.im;
        rr = fma(r.re, x.x, fma(-im, x.y, rr));
        ri = fma(r.re, x.y, fma(im, x.x, ri));
      };
#pragma unroll
      for (int q = 0; q < PF; ++q)
        if (q < nq) link(rec[q], v[q], q < ni);
      for (int q = PF; q < nq; ++q) {
        const ElRec<CT> r = el_rec<CT>(recs + (q < ni ? ib : jb) + q);
        if (HEOM_IN_RANGE(c.err, r.v, 0, c.n_ado)) link(r, el_fetch<CT, BT>(g.zin, c, r.v, i * n + j), q < ni);
      }
      if (herm && i == j) ri = 0;  // exactly Hermitian, as the state is
    } else {
      // stage_kernel's order for non-Hermitian runs: -i (H z), + i (z H), decay, then the links by state
      CT ar = 0, ai = 0;
      const CT *hi_ = s.H + i * n, *hj = s.H + j;
      const C2 *zi = z + i * n, *zj = z + j;
#pragma unroll 4
      for (int k = 0; k < n; ++k) {
        const C2 a = zj[k * n];
        ar = fma(hi_[k], a.y, ar);
        ai = fma(-hi_[k], a.x, ai);
      }
#pragma unroll 4
      for (int k = 0; k < n; ++k) {
        const C2 b = zi[k];
        ar = fma(-b.y, hj[k * n], ar);
        ai = fma(b.x, hj[k * n], ai);
      }
      const CT f = gs + (i != j ? s.term[i] + s.term[j] : (CT)0);
      rr = fma(-f, zij.x, ar);
      ri = fma(-f, zij.y, ai);
      // slots in record order: the lower state's records first
      const bool i_first = i <= j;
      const int nj = nq - ni, n0 = i_first ? ni : nj;
      for (int q = 0; q < (i == j ? ni : nq); ++q) {
        const bool row = (q < n0) == i_first;
        const int at = row ? ib + (i_first ? q : q - nj) : jb + ni + (i_first ? q - ni : q);
        const ElRec<CT> r = el_rec<CT>(recs + at);
        if (!HEOM_IN_RANGE(c.err, r.v, 0, c.n_ado)) continue;
        const C2 x = el_fetch<CT, BT>(g.zin, c, r.v, i * n + j);
        if (i == j) {
          rr = fma(2 * r.re, x.x, rr);
          ri = fma(2 * r.re, x.y, ri);
        } else {
          const CT im = row ? r.im : -r.im;
          rr = fma(r.re, x.x, fma(-im, x.y, rr));
          ri = fma(r.re, x.y, fma(im, x.x, ri));
        }
      }
    }
    // outputs; a pair's mirror element is the conjugate
    auto put = [&](const StateView &o, CT cc, bool base, const C2 &b) {
      C2 w;
      w.x = base ? fma(cc, rr, b.x) : cc * rr;
      w.y = base ? fma(cc, ri, b.y) : cc * ri;
      C2 *d = el_own<CT, BT, OWN_HEAD>(o, c, u0 + la);
      __stcg(d + i * n + j, w);
      if (herm && i != j) {
        w.y = -w.y;
        __stcg(d + j * n + i, w);
      }
    };
    put(g.out, c1, has_y, yv);
    if (has2) put(g.out2, c2, has_y2, y2v);
  }
  if (!landed) el_cp_wait();
}

// How a launch cuts [u_begin, u_end) into units: apu ADOs each, or (apu = 1) `splits` parts of one ADO.
struct ElPlan {
  int apu, splits;
};

template <typename CT, typename BT, int FORM, bool CPLX, bool TWO>
__device__ __forceinline__ void el_units(const ElSmem<CT> &s, const StageCommon &c, const ElStage &g, const ElPlan &pl,
                                         int first, int stride, bool &built) {
  const int P = el_pairs(c.n, c.herm);
  const int units = (c.u_end - c.u_begin + pl.apu - 1) / pl.apu * pl.splits;
  const bool one = units <= stride;  // this CTA never has a second unit: its link ranges stay
  for (int w = first; w < units; w += stride) {
    const int ch = w / pl.splits, part = w - ch * pl.splits;
    const int u0 = c.u_begin + ch * pl.apu, cnt = min(pl.apu, c.u_end - u0);
    const int per = (cnt * P + pl.splits - 1) / pl.splits;
    if (w != first) __syncthreads();  // the tile buffer is reused
    el_unit<CT, BT, FORM, CPLX, TWO>(s, c, g, u0, cnt, part * per, min(cnt * P, part * per + per), !(one && built));
    built = true;
  }
}

// The same out of line: el_run_kernel holds one call per form, each with the registers to itself.
template <typename CT, typename BT, int FORM, bool CPLX>
__device__ __noinline__ bool el_stage_of(const ElSmem<CT> &s, const StageCommon &c, const ElStage &g, const ElPlan &pl,
                                         int first, int stride, bool built) {
  el_units<CT, BT, FORM, CPLX, false>(s, c, g, pl, first, stride, built);
  return built;
}

}  // namespace heom

#include "lean.cuh"

namespace heom {

constexpr int kElThreads = 256;
static_assert(kElThreads == kLeanThreads, "el_run_kernel runs both");

// FP32 body of a Hermitian run with a real H: chunks of floor(32 / N) ADOs per warp, lane (a, i) owning row i of
// ADO a as in stage_kernel, with its operations in its order (see there).  One buffer per warp: a warp of
// el_run_kernel has few chunks per stage, and the other warps of the SM cover its loads.
template <int N>
struct RowSmem {
  using S = StageShape<N>;
  static constexpr int tile = 0;
  static constexpr int rec = (S::A * S::Ep * 8 + 15) & ~15;
  static constexpr int gbuf = rec + 2 * S::RC * 16;
  static constexpr int tb = gbuf + ((S::RC * 2 * N * 8 + 15) & ~15);
  static constexpr int total = tb + 64;
};
struct RowConsts {
  alignas(16) float H[kMaxStates * kMaxStates];
  float term[kMaxStates];
};

// k_at, w_at: offsets of the RowConsts and of the warp's buffers in the dynamic shared memory (an address that the
// compiler can see to be shared: through generic pointers the same code ran 3.5 times slower).
template <int N>
__device__ __forceinline__ void row_body(int k_at, int w_at, const StageCommon &cr, float ch, int first, int nwarps) {
  using S = StageShape<N>;
  using W = RowSmem<N>;
  constexpr int A = S::A, EPO = S::Ep;
  extern __shared__ __align__(16) unsigned char el_sm[];
  const RowConsts &k = *reinterpret_cast<const RowConsts *>(el_sm + k_at);
  unsigned char *wb = el_sm + w_at;
  const StageCommon c = cr;
  const int lane = threadIdx.x & 31, la = lane / N, li = lane - la * N;
  const bool lane_ok = la < A;
  float2 *zt_all = reinterpret_cast<float2 *>(wb + W::tile);
  LinkRec<float> *rec = reinterpret_cast<LinkRec<float> *>(wb + W::rec);
  float2 *gbuf = reinterpret_cast<float2 *>(wb + W::gbuf);
  const float2 *zin = reinterpret_cast<const float2 *>(c.zin.body), *y = reinterpret_cast<const float2 *>(c.y.body);
  const LinkRec<float> *recs = reinterpret_cast<const LinkRec<float> *>(c.recs_body);
  const float term_i = lane_ok ? k.term[li] : 0.f;
  constexpr int cap = 2 * S::RC;
  const int n_chunks = (c.u_end - c.u_begin + A - 1) / A;
  for (int chn = first; chn < n_chunks; chn += nwarps) {
    const int u0 = c.u_begin + chn * A, cnt = min(A, c.u_end - u0);
    const int64_t off = lane <= cnt ? __ldg(c.link_off + u0 + lane) : (int64_t)0;
    const int64_t lo = __shfl_sync(0xffffffffu, off, 0), hi = __shfl_sync(0xffffffffu, off, cnt);
    const int nrec = heom_rec_batch(c.err, lo, (int)min(hi - lo, (int64_t)cap), c.rec_split, c.n_recs);
    const float gsv = lane_ok && la < cnt ? (float)__ldg(c.gsum + u0 + la) : 0.f;
    warp_copy16(rec, recs + (lo - c.rec_split), nrec * 16, lane);
    warp_copy16(zt_all, zin + (int64_t)(u0 - c.u_split) * EPO, cnt * EPO * 8, lane);
    cp_async_commit();
    cp_async_wait<0>();
    __syncwarp();
    issue_gathers<N>(c, rec, nrec, gbuf, lane);
    const bool active = lane_ok && la < cnt;
    float rr[N], ri[N];
    if (active) {
      float2 zr[N];
#pragma unroll
      for (int j = 0; j < N; ++j) {
        rr[j] = ri[j] = 0;
        zr[j] = zt_all[la * EPO + li * N + j];
      }
      if constexpr (N % 2 == 0) {
        uint64_t pr[N / 2], pi[N / 2];
#pragma unroll
        for (int jp = 0; jp < N / 2; ++jp) pr[jp] = pi[jp] = 0;
#pragma unroll
        for (int q = 0; q < N; ++q) {
          const uint64_t sy = pack2(-zr[q].y, -zr[q].y), sx = pack2(zr[q].x, zr[q].x);
#pragma unroll
          for (int jp = 0; jp < N / 2; ++jp) {
            const uint64_t hp = *reinterpret_cast<const uint64_t *>(&k.H[q * kMaxStates + 2 * jp]);
            pr[jp] = ffma2(sy, hp, pr[jp]);
            pi[jp] = ffma2(sx, hp, pi[jp]);
          }
        }
#pragma unroll
        for (int jp = 0; jp < N / 2; ++jp) {
          unpack2(pr[jp], rr[2 * jp], rr[2 * jp + 1]);
          unpack2(pi[jp], ri[2 * jp], ri[2 * jp + 1]);
        }
      } else {
#pragma unroll
        for (int q = 0; q < N; ++q) {
#pragma unroll
          for (int j = 0; j < N; ++j) {
            const float h = k.H[q * kMaxStates + j];
            rr[j] = fmaf(-zr[q].y, h, rr[j]);
            ri[j] = fmaf(zr[q].x, h, ri[j]);
          }
        }
      }
#pragma unroll
      for (int j = 0; j < N; ++j) {
        float f = gsv + ((j != li) ? (term_i + k.term[j]) : 0.f);
        f *= 0.5f;
        rr[j] = fmaf(-f, zr[j].x, rr[j]);
        ri[j] = fmaf(-f, zr[j].y, ri[j]);
      }
    }
    cp_async_wait<0>();
    __syncwarp();
    owner_apply<N>(c, recs, c.rec_split, rec, gbuf, wb + W::tb, lo, hi, nrec, cap, u0, lane, rr, ri);
    owner_combine<N>(active, la, li, zt_all, rr, ri);
    __syncwarp();
    // out = y + ch R, 16 bytes per access
    const int64_t at = (int64_t)(u0 - c.u_split) * EPO;
    const float4 *o4 = reinterpret_cast<const float4 *>(zt_all), *y4 = reinterpret_cast<const float4 *>(y + at);
    float4 *d4 = reinterpret_cast<float4 *>(reinterpret_cast<float2 *>(c.out.body) + at);
#pragma unroll 4
    for (int t = lane; t < cnt * EPO / 2; t += 32) {
      float4 w = o4[t];
      const float4 yv = __ldcg(y4 + t);
      w.x = fmaf(ch, w.x, yv.x);
      w.y = fmaf(ch, w.y, yv.y);
      w.z = fmaf(ch, w.z, yv.z);
      w.w = fmaf(ch, w.w, yv.w);
      __stcg(d4 + t, w);
    }
    __syncwarp();
  }
}

// f(std::integral_constant<int, N>) for N = n in LO..HI.
template <int LO, int HI, typename F>
inline void row_dispatch(int n, F f) {
  if (n == LO) f(std::integral_constant<int, LO>{});
  else if constexpr (LO < HI) row_dispatch<LO + 1, HI>(n, f);
}

template <typename CT, typename BT, int FORM, bool CPLX>
__global__ void __launch_bounds__(kElThreads, 2) el_stage_kernel(const __grid_constant__ ElStageArgs a,
                                                                 const __grid_constant__ ElMup<CPLX> m, int field) {
  extern __shared__ __align__(16) unsigned char el_sm[];
  constexpr bool OWN_HEAD = sizeof(CT) == 8 && sizeof(BT) == 4;
  const StageCommon &c = a.c;
  const ElSmem<CT> s = el_carve<CT>(el_sm, c.n, a.apu, OWN_HEAD ? c.E : c.Ep, el_pairs(c.n, c.herm), true);
  ElConsts k = a.k;
  if constexpr (CPLX) k.mup = field ? m.v : nullptr;
  el_consts<CT>(s, k, c.n, c.herm, true, a.gr, a.gi);
  __syncthreads();
  if constexpr (FORM == kElFixed) {
    el_fix_consts<CPLX>(s, c.n);
    __syncthreads();
  }
  const ElStage g{c.zin, c.y, c.out, a.y2, a.out2, a.c1, a.c2};
  bool built = false;
  el_units<CT, BT, FORM, CPLX, true>(s, c, g, ElPlan{a.apu, a.splits}, blockIdx.x, gridDim.x, built);
}

// The FP64 heads of many runs of equal n_states and equal form in one launch: every CTA takes the units of its run's
// head that fall to it.
template <bool LEAN, bool FIXED>
__global__ void __launch_bounds__(kElThreads, 2) head_list_kernel(const __grid_constant__ HeadList L) {
  extern __shared__ __align__(16) unsigned char el_sm[];
  __shared__ StageCommon c;
  int lo = 0, hi = L.nruns;
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (L.cta0[mid] <= (int)blockIdx.x) lo = mid;
    else hi = mid;
  }
  const ElRunDesc *d = L.d[lo];
  if (threadIdx.x == 0) {
    const int q = L.stage;
    c = d->c;
    c.zin = d->st[q == 0 ? 0 : q == 2 ? 2 : 1];
    c.y = d->st[0];
    c.out = d->st[q == 3 ? 0 : q == 1 ? 2 : 1];
    c.u_begin = 0;
    c.u_end = c.u_split;
  }
  __syncthreads();
  const ElConsts k = d->k;
  const int rank = blockIdx.x - L.cta0[lo], ncta = L.cta0[lo + 1] - L.cta0[lo];
  if constexpr (LEAN) {
    const LeanSmem s = lean_carve(el_sm, L.n, L.apu, 0);
    lean_consts<FIXED>(s, k, L.n);
    lean_chunks<float, FIXED>(s, lean_pair(L.n), c, L.ch, k, rank, ncta);
  } else {
    const ElSmem<double> s = el_carve<double>(el_sm, L.n, L.apu, c.E, el_pairs(L.n, L.herm), true);
    el_consts<double>(s, k, L.n, L.herm, true, 0.0, 0.0);
    __syncthreads();
    el_fix_consts<false>(s, L.n);
    __syncthreads();
    const StateView none{nullptr, nullptr};
    const ElStage g{c.zin, c.y, c.out, none, none, L.ch, 0.0};
    bool built = false;
    el_units<double, float, kElFixed, false, false>(s, c, g, ElPlan{L.apu, L.splits}, rank, ncta, built);
  }
}

// ---- whole steps in one launch ---------------------------------------------------------------------

// The barrier of a run's CTAs: bar[0] counts arrivals of this launch, which every CTA waits to reach
// `target`.  The wait gives up after kElWaitClocks (the run's error word then says kErrTimeout and every
// CTA of the run leaves).  Returns false when it gave up.
constexpr long long kElWaitClocks = 4000000000ll;  // about 2 s
__device__ __forceinline__ bool el_barrier(unsigned *bar, unsigned target, int *err) {
  __shared__ int ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    atomicAdd(bar, 1u);
    const long long t0 = clock64();
    int good = 1;
    unsigned v;
    while (true) {
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(bar) : "memory");
      if (v >= target) break;
      if (clock64() - t0 > kElWaitClocks) {
        atomicOr(err, kErrTimeout);
        good = 0;
        break;
      }
    }
    __threadfence();
    ok = good;
  }
  __syncthreads();
  return ok != 0;
}

// The kinds of el_run_kernel, one per set of code that its CTAs hold (FIXED: with the pair kernels' commutator in fixed
// point; as a branch it cost the runs without it 10 % in registers; ROWS: the states of a Hermitian FP32 body in row form, or
// 0): FP64 runs that the pair kernels cover, with every ADO kept by a CTA or in chunks; mixed runs whose head they
// cover; and all others.  A kernel for each number of states, with its code in line: the row form as functions called
// from one kernel had a stack of 2.6 KB a thread to save registers in, 0.47 GB of device memory that the
// runtime takes at the first such launch.
constexpr int kRunKept = 0, kRunMixed = 1, kRunOther = 2, kRunChunks = 3;

template <int KIND, bool FIXED, int ROWS>
__global__ void __launch_bounds__(KIND == kRunKept ? kLeanRunThreads : kElThreads, 2) el_run_kernel(const __grid_constant__ ElList L) {
  extern __shared__ __align__(16) unsigned char el_sm[];
  __shared__ ElRunDesc d;
  __shared__ StageCommon cs[2][4];  // [FP64 part, FP32 body][stage]
  int lo = 0, hi = L.nruns;         // the run of this CTA
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (L.e[mid].cta0 <= (int)blockIdx.x) lo = mid;
    else hi = mid;
  }
  const ElEntry &en = L.e[lo];
  {
    const int *src = reinterpret_cast<const int *>(en.d);
    int *dst = reinterpret_cast<int *>(&d);
    for (int t = threadIdx.x; t < (int)(sizeof(ElRunDesc) / 4); t += blockDim.x) dst[t] = src[t];
  }
  __syncthreads();
  const int rank = blockIdx.x - en.cta0, ncta = (lo + 1 < L.nruns ? L.e[lo + 1].cta0 : (int)gridDim.x) - en.cta0;
  // an earlier launch of this run gave up: the whole CTA leaves, whatever each of its threads reads
  if (__syncthreads_or(*(volatile int *)d.c.err & kErrTimeout)) return;
  // part 0: FP64 (every ADO of an FP64 run, the head of a mixed one); part 1: the FP32 body
  if (threadIdx.x < 8) {
    const int part = threadIdx.x >> 2, q = threadIdx.x & 3;
    StageCommon &c = cs[part][q];
    c = d.c;
    c.zin = d.st[q == 0 ? 0 : q == 2 ? 2 : 1];
    c.y = d.st[0];
    c.out = d.st[q == 3 ? 0 : q == 1 ? 2 : 1];
    c.u_begin = part ? d.c.u_split : 0;
    c.u_end = part || d.fp64 ? d.c.n_ado : d.c.u_split;
  }
  __syncthreads();
  const int n = d.c.n;
  // CTAs [0, hcta) take the FP64 part, the others the FP32 part; a single CTA takes both
  const bool both = ncta == 1;
  const bool do64 = both || rank < en.hcta;
  const bool do32 = KIND != kRunKept && KIND != kRunChunks && !d.fp64 && d.c.n_ado > d.c.u_split && (both || rank >= en.hcta);
  const int n64 = both ? 1 : en.hcta, n32 = both ? 1 : ncta - en.hcta, r32 = both ? 0 : rank - en.hcta;
  unsigned char *top = el_sm;
  LeanSmem sl{};
  LeanPair lp{};
  LeanState ls{};
  ElSmem<double> s64{};
  ElSmem<float> s32{};
  int k_at = 0, w_at = 0;  // the FP32 body's constants and this warp's buffers in el_sm
  if (do64) {
    if constexpr (KIND != kRunOther) {
      sl = lean_carve(top, n, en.apu64, KIND == kRunKept ? kLeanRunThreads : 0);
      top = sl.end;
      lean_consts<FIXED>(sl, d.k, n);
      lp = lean_pair(n);
      if constexpr (KIND == kRunKept) lean_begin<double, FIXED>(ls, sl, lp, cs[0][0], rank, n64);
    } else {
      const int P = el_pairs(n, d.c.herm);
      s64 = el_carve<double>(top, n, en.apu64, d.fp64 ? d.c.Ep : d.c.E, P, true);
      top = s64.end;
      el_consts<double>(s64, d.k, n, d.c.herm, true, 0.0, 0.0);
      __syncthreads();
      if (d.c.cplx_h) el_fix_consts<true>(s64, n);
      else el_fix_consts<false>(s64, n);
    }
  }
  if (do32) {
    if constexpr (ROWS > 0) {
      RowConsts *rk = reinterpret_cast<RowConsts *>(top);
      k_at = (int)(top - el_sm);
      w_at = k_at + (int)sizeof(RowConsts) + (threadIdx.x >> 5) * en.row_bytes;
      for (int e = threadIdx.x; e < kMaxStates * kMaxStates; e += blockDim.x) {
        const int i = e / kMaxStates, j = e - i * kMaxStates;
        rk->H[e] = i < n && j < n ? (float)d.k.H[i * n + j] : 0.f;
      }
      for (int i = threadIdx.x; i < kMaxStates; i += blockDim.x) rk->term[i] = i < n ? (float)d.k.term[i] : 0.f;
    } else if constexpr (KIND == kRunOther) {
      s32 = el_carve<float>(top, n, en.apu32, d.c.Ep, el_pairs(n, 0), false);
      el_consts<float>(s32, d.k, n, 0, false, 0.0, 0.0);
    }
  }
  __syncthreads();
  bool built64 = false, built32 = false;
  unsigned target = 0;
  int due = en.first_rec;  // steps until the next record (0: none in this launch)
  for (int step = 0; step < en.steps; ++step) {
#pragma unroll 1
    for (int q = 0; q < 4; ++q) {
      const double ch = L.ch[q];
      ElStage g{};
      if constexpr (KIND == kRunOther) {
        g.zin = cs[0][q].zin;
        g.y = cs[0][q].y;
        g.out = cs[0][q].out;
        g.y2 = g.out2 = StateView{nullptr, nullptr};
        g.c1 = ch;
        g.c2 = 0;
      }
      if (do64) {
        const StageCommon &c = cs[0][q];
        if constexpr (KIND == kRunKept) {
          lean_step<double, FIXED>(ls, sl, lp, c, ch, d.k, q == 0);
        } else if constexpr (KIND == kRunChunks) {
          lean_chunks<double, FIXED>(sl, lp, c, ch, d.k, rank, n64);
        } else if constexpr (KIND == kRunMixed) {
          lean_chunks<float, FIXED>(sl, lp, c, ch, d.k, rank, n64);
        } else {
          const ElPlan pl{en.apu64, en.split64};
          if (d.fp64) {
            if (c.cplx_h) built64 = el_stage_of<double, double, kElFixed, true>(s64, c, g, pl, rank, n64, built64);
            else built64 = el_stage_of<double, double, kElFixed, false>(s64, c, g, pl, rank, n64, built64);
          } else {
            built64 = el_stage_of<double, float, kElFixed, false>(s64, c, g, pl, rank, n64, built64);
          }
        }
      }
      if (do32) {
        const StageCommon &c = cs[1][q];
        if constexpr (ROWS > 0) {
          row_body<ROWS>(k_at, w_at, c, (float)ch, (threadIdx.x >> 5) * n32 + r32, n32 * (kElThreads / 32));
        } else if constexpr (KIND == kRunOther) {
          built32 = el_stage_of<float, float, kElRowOrder, false>(s32, c, g, ElPlan{en.apu32, 1}, r32, n32, built32);
        }
      }
      target += ncta;
      if (both) {
        __threadfence_block();
        __syncthreads();
      } else if (!el_barrier(d.bar, target, d.c.err)) {
        return;
      }
    }
    if (due > 0 && --due == 0) {
      // sigma_0 stays as it is until the last stage of the next step
      if (rank == ncta - 1 && threadIdx.x < 32)
        record_warp(d.st[0], d.c.u_split, !d.fp64, 0, n, d.w, d.records, d.rec_count, d.max_records);
      due = en.stride;
    }
  }
  if (!both) {  // the last CTA to leave clears the counters for the next launch
    __syncthreads();
    if (threadIdx.x == 0) {
      __threadfence();
      if (atomicAdd(d.bar + 1, 1u) == (unsigned)ncta - 1) {
        d.bar[0] = 0;
        d.bar[1] = 0;
        __threadfence();
      }
    }
  }
}

}  // namespace heom
