// FP64 stages of Hermitian runs with a real H (every ADO of an FP64 run, the head of a mixed one), one thread
// per element pair (i <= j) of an ADO (sm_103a).  Included by resident.cuh, which states the element form of
// Eq. HEOM and the fixed-point commutator that these kernels use.
//
// A CTA of kLeanThreads threads takes floor(kLeanThreads / P) consecutive ADOs of P = n (n + 1) / 2 pairs, so a
// thread's pair, its shared-memory addresses and its element offsets never change.  Per chunk a thread loads its
// own element of the input (the upper triangle only: the lower one is its conjugate), the CTA agrees on the
// tiles' scales, every thread writes its element and its mirror as limbs to shared memory, and while
// the neighbour elements of up to four links are on their way it forms the commutator there.  FP64 instructions
// (18.7 clocks per warp and SM) remain for decay, links and the RK4 combination: about 4 + 4 per link slot.
// Measured, FP64 runs, us per step (row kernels before): 1716 ADOs of 7 x 7 69.5 -> 27.0, 330 of them 65.8 -> 19.1, 680 of
// 14 x 14 393 -> 38.9, 3003 of 10 x 10 230 -> 84.
#pragma once

namespace heom {

constexpr int kLeanMaxStates = 22;  // 253 pairs: one ADO fits a CTA of 256 threads
constexpr int kLeanThreads = 256;   // stage kernel, and CTAs of mixed runs
// CTAs that keep FP64 runs: more ADOs in each than with 256 threads, so that larger runs still fit (680 ADOs of 14 states
// 38.9 us per step against 65.9, 2002 of 9 37 against 59), and more warps for the smallest (120 of 3 states 14.5 / 17.7)
constexpr int kLeanRunThreads = 320;
constexpr int kLeanSlots = 4;       // link slots in registers (stages); more are read in a loop
constexpr int kLeanKept = 6;        // the same of CTAs that keep their ADOs

// The most ADOs of n states that a CTA takes at once.
__host__ __device__ inline int lean_ados(int n, int threads) {
  const int a = threads / (n * (n + 1) / 2);
  return a < 32 ? a : 32;
}

// Whether the commutator of a part of `ados` ADOs runs in fixed point.  An FP64 FMA holds its SM partition for 64
// clocks whether one warp or many wait, so with few warps per SM 4 n of them per pair are as fast as the integer path,
// and only the pipe's throughput counts from about 200 pairs per SM on or where one ADO fills it.  Measured, us per
// step, FMAs / fixed point: 6 states, 19404 pairs 18.3 / 19.2, 36036 27.7 / 24.1; 7, 9240 19.0 / 19.8, 48048 33.4 / 27.0; 8, 17820
// 19.6 / 21.0, 46332 33.2 / 27.1; 9, 2475 20.1 / 21.0, 32175 30.9 / 25.5; 12, 7098 21.7 / 23.4, 35490 34.4 / 28.2; 14, 1575
// 25.7 / 23.6; 4 states, 12870 21.4 / 23.2.  A property of the run: every form of launch decides alike.
__host__ __device__ inline bool lean_fixed(int n, int64_t ados) {
  return n >= 9 || (n >= 5 && ados * (n * (n + 1) / 2) >= 32768);
}
// The same for the head of a mixed run: its 1 + n_modes ADOs (at most 256) never reach the second line.  Of one step, 8 states, 165
// ADOs 27.7 / 28.0; 9, 715 32.6 / 32.3; 10, 1001 33.8 / 31.6; 12, 455 31.0 / 32.5, 1820 41.7 / 37.2.
__host__ __device__ constexpr bool lean_head_fixed(int n) { return n >= 9; }

// Shared memory: limbs of H and of the tiles, T, scale keys (two sets), link ranges; and for resident CTAs the
// coefficients of each thread's slots.
struct LeanSmem {
  int4 *tile;      // [ados][n][n] Re hi, Re lo, Im hi, Im lo (fixed point) or the FP64 elements
  int2 *rest;      // [ados][n][n] third limbs, Re and Im
  double2 *coef;   // [kLeanKept][threads] R (resident)
  double *T;       // [n][n]
  int2 *H;         // [n][n] limbs or FP64
  int *hrest;      // [n][n] third limbs
  int *key;        // [2][2 ados]
  int *hkey;
  uint32_t *rng;   // [ados][n] begin | end << 16, relative to the ADO's first record
  unsigned char *end;
  int ados;        // ADOs per chunk
};
__host__ __device__ inline size_t lean_smem_bytes(int n, int a, int kept_threads) {
  const size_t E = (size_t)n * n;
  const size_t b = a * E * 24 + (size_t)kLeanKept * kept_threads * 16 + E * 20 + 16 * (size_t)a + 16 + 4 * (size_t)a * n;
  return (b + 15) & ~(size_t)15;
}
__device__ __forceinline__ LeanSmem lean_carve(unsigned char *p, int n, int a, int kept_threads) {
  const int E = n * n;
  LeanSmem s;
  s.tile = reinterpret_cast<int4 *>(p);
  s.coef = reinterpret_cast<double2 *>(s.tile + a * E);
  s.rest = reinterpret_cast<int2 *>(s.coef + kLeanKept * kept_threads);
  s.T = reinterpret_cast<double *>(s.rest + a * E);
  s.H = reinterpret_cast<int2 *>(s.T + E);
  s.hrest = reinterpret_cast<int *>(s.H + E);
  s.key = s.hrest + E;
  s.hkey = s.key + 4 * a;
  s.rng = reinterpret_cast<uint32_t *>(s.hkey + 4);
  s.end = p + lean_smem_bytes(n, a, kept_threads);
  s.ados = a;
  return s;
}

// A thread's pair.
struct LeanPair {
  int la, i, j;        // ADO in the chunk, element (i <= j)
  int e, em;           // i n + j, j n + i
  bool whole;          // every lane of the warp has the same ADO
};
__device__ __forceinline__ LeanPair lean_pair(int n) {
  LeanPair p;
  const int P = n * (n + 1) / 2, t = threadIdx.x;
  p.la = t / P;
  int r = t - p.la * P, i = 0;
  while (r >= n - i) {
    r -= n - i;
    ++i;
  }
  p.i = i;
  p.j = i + r;
  p.e = p.i * n + p.j;
  p.em = p.j * n + p.i;
  p.whole = __all_sync(0xffffffffu, p.la == __shfl_sync(0xffffffffu, p.la, 0));
  return p;
}

// H as limbs, T; synchronises the CTA.  FIXED: the commutator in fixed point (lean_fixed).
template <bool FIXED>
__device__ __forceinline__ void lean_consts(const LeanSmem &s, const ElConsts &k, int n) {
  if (threadIdx.x == 0) *s.hkey = 0;
  __syncthreads();
  int key = 0;
  for (int e = threadIdx.x; e < n * n; e += blockDim.x) {
    key = max(key, fx_key(k.H[e]));
    s.T[e] = k.T[e];
  }
  key = __reduce_max_sync(0xffffffffu, key);
  if ((threadIdx.x & 31) == 0) atomicMax(s.hkey, key);
  __syncthreads();
  const int ex = fx_exp(*s.hkey);
  for (int e = threadIdx.x; e < n * n; e += blockDim.x) {
    if (FIXED) s.H[e] = fx_split(k.H[e], ex, s.hrest[e]);
    else reinterpret_cast<double *>(s.H)[e] = k.H[e];
  }
  __syncthreads();
}

// Called by every thread of the CTA (z = 0 where a thread has no element).
template <bool FIXED>
__device__ __forceinline__ void lean_key(const LeanSmem &s, const LeanPair &p, int *key, double2 z) {
  if (!FIXED) return;
  int kx = fx_key(z.x), ky = fx_key(z.y);
  if (p.whole) {
    kx = __reduce_max_sync(0xffffffffu, kx);
    ky = __reduce_max_sync(0xffffffffu, ky);
    if ((threadIdx.x & 31) != 0) return;
  }
  if (p.la >= s.ados) return;
  atomicMax(&key[2 * p.la], kx);
  atomicMax(&key[2 * p.la + 1], ky);
}

// The element and its mirror (conjugate) as limbs.
template <bool FIXED>
__device__ __forceinline__ void lean_limbs(const LeanSmem &s, const LeanPair &p, int n, const int *key, double2 z) {
  if constexpr (!FIXED) {
    double2 *t = reinterpret_cast<double2 *>(s.tile) + p.la * n * n;
    t[p.e] = z;
    if (p.i != p.j) t[p.em] = make_double2(z.x, -z.y);
  } else {
    int2 w;
    const int2 a = fx_split(z.x, fx_exp(key[2 * p.la]), w.x), b = fx_split(z.y, fx_exp(key[2 * p.la + 1]), w.y);
    int4 *t = s.tile + p.la * n * n;
    int2 *tw = s.rest + p.la * n * n;
    t[p.e] = make_int4(a.x, a.y, b.x, b.y);
    tw[p.e] = w;
    if (p.i != p.j) {
      t[p.em] = make_int4(a.x, a.y, -b.x, -b.y);
      tw[p.em] = make_int2(w.x, -w.y);
    }
  }
}

// C = H z - z H of element (i, j) by FP64 FMAs, H and the ADO's tile z in global memory.
static __device__ __noinline__ double2 lean_fma_comm(const double *H, const double2 *z, int n, int i, int j) {
  double ar = 0, ai = 0, br = 0, bi = 0;
#pragma unroll 4
  for (int k = 0; k < n; ++k) {
    const double2 a = __ldcg(z + k * n + j), b = __ldcg(z + i * n + k);
    const double h1 = H[i * n + k], h2 = H[k * n + j];
    ar = fma(h1, a.x, ar);
    ai = fma(h1, a.y, ai);
    br = fma(b.x, h2, br);
    bi = fma(b.y, h2, bi);
  }
  return make_double2(ar - br, ai - bi);
}

// -i (H z - z H)_ij - f z_ij; zin: the ADO's tile in global memory (read only where the FMA chain takes over).
template <bool FIXED>
__device__ __forceinline__ double2 lean_comm(const LeanSmem &s, const LeanPair &p, int n, const int *key, double2 z, double f,
                                             const double2 *zin, const ElConsts &kc) {
  double cr = 0, ci = 0;
  if constexpr (!FIXED) {
    double ar = 0, ai = 0, br = 0, bi = 0;
    const double2 *zi = reinterpret_cast<const double2 *>(s.tile) + (p.la * n + p.i) * n;
    const double2 *zj = reinterpret_cast<const double2 *>(s.tile) + p.la * n * n + p.j;
    const double *hi_ = reinterpret_cast<const double *>(s.H) + p.i * n, *hj = reinterpret_cast<const double *>(s.H) + p.j;
    for (int k = 0; k < n; ++k) {
      const double2 a = *zj, b = zi[k];
      const double h1 = hi_[k], h2 = *hj;
      zj += n;
      hj += n;
      ar = fma(h1, a.x, ar);
      ai = fma(h1, a.y, ai);
      br = fma(b.x, h2, br);
      bi = fma(b.y, h2, bi);
    }
    cr = ar - br;
    ci = ai - bi;
  } else {
    const int kx = key[2 * p.la], ky = key[2 * p.la + 1], hk = *s.hkey;
    int chain = 3;  // bits: Re C, Im C by FMAs
    if (fx_ok(hk, kx) && fx_ok(hk, ky)) {
      FxSum r, m;
      const int4 *zi = s.tile + (p.la * n + p.i) * n, *zj = s.tile + p.la * n * n + p.j;
      const int2 *wi = s.rest + (p.la * n + p.i) * n, *wj = s.rest + p.la * n * n + p.j;
      const int2 *hi_ = s.H + p.i * n, *hj = s.H + p.j;
      const int *vi = s.hrest + p.i * n, *vj = s.hrest + p.j;
#pragma unroll 2
      for (int k = 0; k < n; ++k) {
        const int4 a = *zj, b = zi[k];
        const int2 ar = *wj, br = wi[k], h1 = hi_[k], h2 = *hj;
        const int r1 = vi[k], nx = -h2.x, ny = -h2.y, nr = -*vj;
        zj += n;
        wj += n;
        hj += n;
        vj += n;
        r.add(h1.x, h1.y, r1, a.x, a.y, ar.x);
        m.add(h1.x, h1.y, r1, a.z, a.w, ar.y);
        r.add(nx, ny, nr, b.x, b.y, br.x);
        m.add(nx, ny, nr, b.z, b.w, br.y);
      }
      chain = fx_finish(r, m, hk, kx, ky, cr, ci);
    }
    if (p.i == p.j) chain &= 2;  // Re C = 0 there and is not used
    if (chain) {
      const double2 x = lean_fma_comm(kc.H, zin, n, p.i, p.j);
      if (chain & 1) cr = x.x;
      if (chain & 2) ci = x.y;
    }
  }
  return make_double2(fma(-f, z.x, ci), fma(-f, z.y, -cr));
}

__device__ __forceinline__ void lean_link(double2 &r, double re, double im, double2 v, bool row) {
  im = row ? im : -im;  // R v_ij of state i's records, conj(R) v_ij of state j's
  r.x = fma(re, v.x, fma(-im, v.y, r.x));
  r.y = fma(re, v.y, fma(im, v.x, r.y));
}

// The link records of a thread's element: slots [0, ni) of state i from record ib, then those of state j from jb.
struct LeanLinks {
  int ib, jb, ni, nq;
};
__device__ __forceinline__ LeanLinks lean_links(const LeanSmem &s, const LeanPair &p, int n) {
  const uint32_t a = s.rng[p.la * n + p.i], b = s.rng[p.la * n + p.j];
  LeanLinks l;
  l.ib = a & 0xffff;
  l.ni = (int)(a >> 16) - l.ib;
  l.nq = l.ni + (int)(b >> 16) - (int)(b & 0xffff);
  l.jb = (int)(b & 0xffff) - l.ni;
  return l;
}

template <typename BT>
__device__ __forceinline__ const LinkRec<double> *lean_recs(const StageCommon &c, int64_t lo) {
  constexpr bool OWN_HEAD = sizeof(BT) == 4;
  return reinterpret_cast<const LinkRec<double> *>(OWN_HEAD ? c.recs_head : c.recs_body) + lo;
}

// Link ranges of the chunk's ADOs u0 + la du, a warp for each in turn; s.rng is zero before, a __syncthreads follows.
template <typename BT>
__device__ __forceinline__ void lean_ranges(const LeanSmem &s, const StageCommon &c, int u0, int du, int cnt) {
  const int lane = threadIdx.x & 31;
  uint16_t *half = reinterpret_cast<uint16_t *>(s.rng);
  for (int la = threadIdx.x >> 5; la < cnt; la += blockDim.x >> 5) {
    const int64_t lo = __ldg(c.link_off + u0 + la * du);
    const int nrec = heom_rec_batch(c.err, lo, (int)(__ldg(c.link_off + u0 + la * du + 1) - lo), 0,
                                    sizeof(BT) == 4 ? c.rec_split : c.n_recs);
    const LinkRec<double> *recs = lean_recs<BT>(c, lo);
    for (int t = lane; t < nrec; t += 32) {
      const int st = __ldg(&recs[t].s) & kRecStateMask;
      if (!HEOM_IN_RANGE(c.err, st, 0, c.n)) continue;
      const int o = la * c.n + st;
      if (t == 0 || (__ldg(&recs[t - 1].s) & kRecStateMask) != st) half[2 * o] = (uint16_t)t;
      if (t + 1 == nrec || (__ldg(&recs[t + 1].s) & kRecStateMask) != st) half[2 * o + 1] = (uint16_t)(t + 1);
    }
  }
}

// Chunks first, first + stride, ... of one stage.
template <typename BT, bool FIXED>
__device__ __forceinline__ void lean_chunks(const LeanSmem &s, const LeanPair &p, const StageCommon &c, double ch,
                                            const ElConsts &kc, int first, int stride) {
  constexpr bool OWN_HEAD = sizeof(BT) == 4;
  const int n = c.n, A = s.ados;
  const int chunks = (c.u_end - c.u_begin + A - 1) / A;
  const bool has_y = el_set(c.y), same_y = c.y.head == c.zin.head && c.y.body == c.zin.body;
  const double Tij = p.la < A ? s.T[p.e] : 0.0;
  for (int w = first; w < chunks; w += stride) {
    const int u0 = c.u_begin + w * A, cnt = min(A, c.u_end - u0), u = u0 + p.la;
    const bool have = p.la < cnt;
    double2 z = make_double2(0, 0), y = z;
    double f = 0;
    const double2 *zt = el_own<double, BT, OWN_HEAD>(c.zin, c, u);
    const LinkRec<double> *recs = nullptr;
    if (have) {
      z = __ldcg(zt + p.e);
      if (has_y) y = same_y ? z : __ldcg(el_own<double, BT, OWN_HEAD>(c.y, c, u) + p.e);
      f = __ldg(c.gsum + u) + Tij;
      recs = lean_recs<BT>(c, __ldg(c.link_off + u));
    }
    __syncthreads();  // the previous chunk is done with the shared buffers
    for (int t = threadIdx.x; t < cnt * n; t += blockDim.x) s.rng[t] = 0;
    if (threadIdx.x < 2 * A) s.key[threadIdx.x] = 0;
    __syncthreads();
    lean_ranges<BT>(s, c, u0, 1, cnt);
    lean_key<FIXED>(s, p, s.key, z);
    __syncthreads();
    LeanLinks l{0, 0, 0, 0};
    ElRec<double> rec[kLeanSlots];
    double2 v[kLeanSlots];
    if (have) {
      l = lean_links(s, p, n);
#pragma unroll
      for (int q = 0; q < kLeanSlots; ++q)
        if (q < l.nq) rec[q] = el_rec<double>(recs + (q < l.ni ? l.ib : l.jb) + q);
#pragma unroll
      for (int q = 0; q < kLeanSlots; ++q) {
        v[q] = make_double2(0, 0);
        if (q < l.nq && HEOM_IN_RANGE(c.err, rec[q].v, 0, c.n_ado)) v[q] = el_fetch<double, BT>(c.zin, c, rec[q].v, p.e);
      }
      lean_limbs<FIXED>(s, p, n, s.key, z);
    }
    __syncthreads();
    if (!have) continue;
    double2 r = lean_comm<FIXED>(s, p, n, s.key, z, f, zt, kc);
#pragma unroll
    for (int q = 0; q < kLeanSlots; ++q)
      if (q < l.nq) lean_link(r, rec[q].re, rec[q].im, v[q], q < l.ni);
    for (int q = kLeanSlots; q < l.nq; ++q) {
      const ElRec<double> x = el_rec<double>(recs + (q < l.ni ? l.ib : l.jb) + q);
      if (HEOM_IN_RANGE(c.err, x.v, 0, c.n_ado)) lean_link(r, x.re, x.im, el_fetch<double, BT>(c.zin, c, x.v, p.e), q < l.ni);
    }
    if (p.i == p.j) r.y = 0;  // exactly Hermitian, as the state is
    double2 o;
    o.x = has_y ? fma(ch, r.x, y.x) : ch * r.x;
    o.y = has_y ? fma(ch, r.y, y.y) : ch * r.y;
    double2 *d = el_own<double, BT, OWN_HEAD>(c.out, c, u);
    __stcg(d + p.e, o);
    if (p.i != p.j) __stcg(d + p.em, make_double2(o.x, -o.y));
  }
}

// A CTA that keeps its ADOs first, first + stride, ... (at most s.ados: hierarchy levels spread evenly over the CTAs)
// for all stages of a launch: z and y of its pairs stay in registers, the tiles in shared memory, the
// slots' coefficients too.
struct LeanState {
  double2 z, y;
  double f;
  int v[kLeanKept];
  LeanLinks l;
  const LinkRec<double> *recs;
  int u, buf;
  bool have;
};

template <typename BT, bool FIXED>
__device__ __forceinline__ void lean_begin(LeanState &t, const LeanSmem &s, const LeanPair &p, const StageCommon &c, int first,
                                           int stride) {
  constexpr bool OWN_HEAD = sizeof(BT) == 4;
  const int n = c.n, A = s.ados, u0 = c.u_begin + first;
  const int cnt = u0 < c.u_end ? min(A, (c.u_end - 1 - u0) / stride + 1) : 0;
  t.have = p.la < cnt;
  t.u = u0 + p.la * stride;
  t.buf = 0;
  t.l = LeanLinks{0, 0, 0, 0};
  t.z = t.y = make_double2(0, 0);
  t.f = 0;
  t.recs = nullptr;
  for (int k = threadIdx.x; k < A * n; k += blockDim.x) s.rng[k] = 0;
  for (int k = threadIdx.x; k < 4 * A; k += blockDim.x) s.key[k] = 0;
  __syncthreads();
  lean_ranges<BT>(s, c, u0, stride, cnt);
  if (t.have) {
    t.z = __ldcg(el_own<double, BT, OWN_HEAD>(c.y, c, t.u) + p.e);
    t.f = __ldg(c.gsum + t.u) + s.T[p.e];
    t.recs = lean_recs<BT>(c, __ldg(c.link_off + t.u));
  }
  lean_key<FIXED>(s, p, s.key, t.z);
  __syncthreads();
  if (t.have) {
    t.l = lean_links(s, p, n);
#pragma unroll
    for (int q = 0; q < kLeanKept; ++q) {
      t.v[q] = 0;
      if (q < t.l.nq) {
        const ElRec<double> r = el_rec<double>(t.recs + (q < t.l.ni ? t.l.ib : t.l.jb) + q);
        s.coef[q * blockDim.x + threadIdx.x] = make_double2(r.re, q < t.l.ni ? r.im : -r.im);
        t.v[q] = HEOM_IN_RANGE(c.err, r.v, 0, c.n_ado) ? r.v : 0;
      }
    }
  }
}

// One stage; the first of a step also takes y = z, and the last one leaves the step's result in z.
template <typename BT, bool FIXED>
__device__ __forceinline__ void lean_step(LeanState &t, const LeanSmem &s, const LeanPair &p, const StageCommon &c, double ch,
                                          const ElConsts &kc, bool begins) {
  constexpr bool OWN_HEAD = sizeof(BT) == 4;
  const int n = c.n, A = s.ados;
  int *key = s.key + t.buf * 2 * A, *next = s.key + (t.buf ^ 1) * 2 * A;
  t.buf ^= 1;
  double2 v[kLeanKept];
  if (t.have) {
    if (begins) t.y = t.z;
#pragma unroll
    for (int q = 0; q < kLeanKept; ++q)
      if (q < t.l.nq) v[q] = el_fetch<double, BT>(c.zin, c, t.v[q], p.e);
    lean_limbs<FIXED>(s, p, n, key, t.z);
  }
  if (threadIdx.x < 2 * A) next[threadIdx.x] = 0;
  __syncthreads();
  if (t.have) {
    double2 r = lean_comm<FIXED>(s, p, n, key, t.z, t.f, el_own<double, BT, OWN_HEAD>(c.zin, c, t.u), kc);
#pragma unroll
    for (int q = 0; q < kLeanKept; ++q)
      if (q < t.l.nq) {
        const double2 k = s.coef[q * blockDim.x + threadIdx.x];
        lean_link(r, k.x, k.y, v[q], true);
      }
    for (int q = kLeanKept; q < t.l.nq; ++q) {
      const ElRec<double> x = el_rec<double>(t.recs + (q < t.l.ni ? t.l.ib : t.l.jb) + q);
      if (HEOM_IN_RANGE(c.err, x.v, 0, c.n_ado)) lean_link(r, x.re, x.im, el_fetch<double, BT>(c.zin, c, x.v, p.e), q < t.l.ni);
    }
    if (p.i == p.j) r.y = 0;
    t.z.x = fma(ch, r.x, t.y.x);
    t.z.y = fma(ch, r.y, t.y.y);
    double2 *d = el_own<double, BT, OWN_HEAD>(c.out, c, t.u);
    __stcg(d + p.e, t.z);
    if (p.i != p.j) __stcg(d + p.em, make_double2(t.z.x, -t.z.y));
  }
  lean_key<FIXED>(s, p, next, t.z);
}

// One stage of a range of ADOs.
template <typename BT, bool FIXED>
__global__ void __launch_bounds__(kLeanThreads, 2) lean_stage_kernel(const __grid_constant__ ElStageArgs a) {
  extern __shared__ __align__(16) unsigned char el_sm[];
  const LeanSmem s = lean_carve(el_sm, a.c.n, a.apu, 0);
  lean_consts<FIXED>(s, a.k, a.c.n);
  const LeanPair p = lean_pair(a.c.n);
  lean_chunks<BT, FIXED>(s, p, a.c, a.c1, a.k, blockIdx.x, gridDim.x);
}

}  // namespace heom
