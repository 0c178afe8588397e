// FP64 stage kernel for Hermitian runs with a real H, column form (sm_103a).
//
// Same operation as stage_kernel: for every ADO u in [u_begin, u_end),
//     out_u = y_u + ch * (L zin)_u          (or ch * (L zin)_u when there is no y)
// with L the right-hand side of Eq. HEOM (arXiv 1803.03498, section "HEOM formalism", with the ADO
// rescaling; hbar = 1, energies in rad/fs).  For a Hermitian run (Hermitian H and ADOs, real c: every
// ADO stays Hermitian) the result is R = Q + Q^dagger with
//     Q_ij = -i (H s)_ij + coef_ij s_ij + sum over the links of state s = i of R_link v_ij
//     coef_ij = -(g / 2 + Delta_i)  (i != j),   coef_ii = -g / 2,     g = sum_l n_l gamma_l
// because s H = (H s)^dagger, the terminator (Delta_i + Delta_j) s_ij (i != j) splits into a row and
// a column part, and a link adds R v_sj to row s, conj(R) v_is = conj(R v_si) to column s and
// 2 Re(R) v_ss to the diagonal (see LinkRec).
//
// Bound and form: GB300 issues one FP64 instruction per 64 clocks and SM partition (18.7 clocks per SM measured), two
// 32 x 32 + 64 bit integer multiply-adds per clock and SM.  The commutator, 2 N^3 multiply-adds per ADO, therefore runs
// in integers (fixed_point.cuh: three limbs of 28 bits, one rounding at the end of a sum), and the FP64 pipe keeps
// what is cheaper there than in integers: the sums' conversion (2 additions), the decay, the links (2 per
// record and lane), R and the RK4 combination (4 per pair of elements).  A lane owns one column of one part: lane (a, p, j)
// computes column j of Q_re (p = 0, from H Im s) or of Q_im (p = 1, from -H Re s) of ADO a -- 2N columns
// per ADO -- so the scale of its operands is its own column's largest element, without a word to other lanes, and
// the limbs of H come from shared memory, one 16-byte broadcast each (as 16-byte constant loads: 187 ms against 177 for
// four steps at the LHCII size).  A warp takes chunks of G
// consecutive ADOs, G chosen so that 2 N G is a multiple of 32, and covers their 2 N G columns in P = 2 N G / 32
// passes with every lane busy (N = 14: 8 ADOs in 7 passes).  Per pass a lane
//   - loads column j of its ADO's zin tile from global memory (the 2N lanes of an ADO read whole rows:
//     coalesced) and splits the part it multiplies into limbs;
//   - forms the N entries of its column of H (Im s) or -H (Re s), each a sum of 6 N integer products, plus
//     coef * (own part);
//   - writes the column in FP64 into its ADO's slot of a per-warp ring of Q tiles in shared memory.
// An ADO whose last column was computed in this pass is finalised by the warp: the
// row s of every linked neighbour (gathered into shared memory by cp.async while the pass computed)
// is added to row s of Q, records in order; then the lanes take the pairs i <= j: R_ij = Q_ij + conj(Q_ji),
// out = y + ch R, written to (i, j) and, conjugated, to (j, i).  Warps are independent (only __syncwarp).  Every output
// element sums the same terms in the same order under every launch schedule.
// A column with Inf, NaN or exponents near the ends of the range takes FP64 FMAs instead, and so does a row of it whose sum
// is weak beside the column (fx_weak).
#pragma once
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>

#include "fixed_point.cuh"
#include "heom_internal.h"

namespace heom {

// Most ADOs of C columns that one pass of 32 consecutive columns touches, over the P passes of a chunk.
__host__ __device__ constexpr int col_ring(int C, int P) {
  int m = 1;
  for (int q = 0; q < P; ++q) {
    const int t = (32 * q + 31) / C - (32 * q) / C + 1;
    m = t > m ? t : m;
  }
  return m;
}

template <int N>
struct ColShape {
  static constexpr int C = 2 * N;                  // columns per ADO (both parts)
  static constexpr int G = 32 / col_gcd(C, 32);    // ADOs per warp chunk
  static constexpr int P = col_passes(N);          // passes of 32 columns per chunk
  static_assert(P * 32 == C * G, "whole passes");
  static constexpr int E = N * N;
  static constexpr int RING = col_ring(C, P);      // Q slots: the ADOs one pass touches (N = 14: 2)
  static constexpr int RB = 12;                    // link records per batch and finalising ADO
  static constexpr int WARPS = 4;                  // 4 CTAs of 4 warps per SM (128 registers, < 57 KB)
  static_assert(C >= 16 && G <= 31, "column kernel covers 8 <= N <= 16");
};

// Per-warp shared memory (byte offsets; every region 16-byte aligned).
template <int N>
struct ColSmem {
  using S = ColShape<N>;
  static constexpr int q = 0;                                    // [RING][2][N][N] double
  static constexpr int coef = q + S::RING * 2 * S::E * 8;        // [G][N] double: -(g/2 + Delta_i)
  static constexpr int gh = coef + S::G * N * 8;                 // [G] double: -g/2
  static constexpr int rec = (gh + S::G * 8 + 15) & ~15;         // [2 RB] LinkRec<double>
  static constexpr int gbuf = rec + 2 * S::RB * 32;              // [2 RB][N] double2: gathered rows
  static constexpr int total = gbuf + 2 * S::RB * N * 16;
};

__device__ __forceinline__ void col_cp16(void *smem, const void *gmem) {
  const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(s), "l"(gmem) : "memory");
}
__device__ __forceinline__ void col_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
__device__ __forceinline__ void col_wait_all() { asm volatile("cp.async.wait_group 0;\n" ::: "memory"); }

// -x without an FP64 instruction (sign bit of the high word)
__device__ __forceinline__ double col_neg(double x) {
  return __hiloint2double(__double2hiint(x) ^ (int)0x80000000, __double2loint(x));
}

// Records [lo, lo + nr) into rec (32 bytes each), one cp.async group.
__device__ __forceinline__ void col_load_recs(const LinkRec<double> *recs, int64_t lo, int nr, LinkRec<double> *rec,
                                              int lane) {
  const char *src = reinterpret_cast<const char *>(recs + lo);
  char *dst = reinterpret_cast<char *>(rec);
  for (int o = lane * 16; o < nr * 32; o += 32 * 16) col_cp16(dst + o, src + o);
  col_commit();
}

// Row s of the neighbour of each of the nr records into gbuf[r][0..N), one cp.async group.
template <int N>
__device__ __forceinline__ void col_gather(const StageCommon &c, const double2 *zin, int Ep, const LinkRec<double> *rec,
                                           int nr, double2 *gbuf, int lane) {
  for (int t = lane; t < nr * N; t += 32) {
    const int r = t / N, k = t - r * N;
    const int s = rec[r].s & kRecStateMask;
    if (HEOM_IN_RANGE(c.err, rec[r].v, 0, c.n_ado) && HEOM_IN_RANGE(c.err, s, 0, N))
      col_cp16(gbuf + r * N + k, zin + (int64_t)rec[r].v * Ep + s * N + k);
  }
  col_commit();
}

// Adds the nr records of rec (gathered rows in gbuf) to row s of the Q tile qs ([2][N][N]): lane
// (p, j) owns element (s, j) of part p; records are ordered by s, so each lane keeps its element in a
// register while s stays the same.  R v = (Rr vr - Ri vi) + i (Rr vi + Ri vr).
template <int N>
__device__ __forceinline__ void col_links(const LinkRec<double> *rec, int nr, const double2 *gbuf, double *qs, int lane) {
  if (lane >= 2 * N) return;
  const int p = lane / N, j = lane - p * N;
  double *qp = qs + p * N * N;
  int cur = -1;
  double acc = 0;
  for (int r = 0; r < nr; ++r) {
    const int s = rec[r].s & kRecStateMask;
    if (s != cur) {
      if (cur >= 0) qp[cur * N + j] = acc;
      cur = s;
      acc = qp[s * N + j];
    }
    const double2 v = gbuf[r * N + j];
    const double rr = rec[r].re, ri = rec[r].im;
    const double a1 = p ? v.y : v.x;             // Re part: Rr vr - Ri vi;  Im part: Rr vi + Ri vr
    const double a2 = p ? v.x : v.y;
    const double b2 = p ? ri : col_neg(ri);
    acc = fma(rr, a1, fma(b2, a2, acc));
  }
  if (cur >= 0) qp[cur * N + j] = acc;
}

struct ColArgs {
  StageCommon c;
  double ch;
  int ex;                                // |H| < 2^(ex - 1022)
  double term[kMaxStates];               // terminator Delta per state
  double H[kMaxStates * kMaxStates];     // Re H - h0 I, rad/fs (columns out of range)
  int4 Hx[kMaxStates * kMaxStates];      // its limbs
};

// Row i of column zt[0], zt[N], ... of H Im s (p = 0) or -H Re s (p = 1) by FP64 FMAs.
template <int N>
__device__ __noinline__ double col_fma_row(const ColArgs &a, const double2 *zt, int p, int i) {
  double acc = 0;
  for (int k = 0; k < N; ++k) {
    const double2 z = zt[k * N];
    acc = fma(a.H[i * kMaxStates + k], p ? -z.x : z.y, acc);
  }
  return acc;
}
// Column j of part p of -i H s + coef s the same way, into q[i * N + j].
template <int N>
__device__ __noinline__ void col_fma(const ColArgs &a, const double2 *zt, int p, int j, double g, double *q) {
  for (int i = 0; i < N; ++i) {
    const double acc = col_fma_row<N>(a, zt, p, i);
    const double2 z = zt[i * N];
    q[i * N + j] = fma(i == j ? -0.5 * g : fma(-0.5, g, -a.term[i]), p ? z.y : z.x, acc);
  }
}

template <int N>
__global__ void __launch_bounds__(ColShape<N>::WARPS * 32, 4) stage_col_kernel(const __grid_constant__ ColArgs a) {
  using S = ColShape<N>;
  using W = ColSmem<N>;
  constexpr int C = S::C, G = S::G, P = S::P, E = S::E, RB = S::RB;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ int4 Hs[N * N];  // the limbs of H
  for (int e = threadIdx.x; e < N * N; e += blockDim.x) Hs[e] = a.Hx[(e / N) * kMaxStates + e % N];
  __syncthreads();
  const StageCommon &c = a.c;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  unsigned char *wb = smem_raw + warp * W::total;
  double *qring = reinterpret_cast<double *>(wb + W::q);
  double *coef = reinterpret_cast<double *>(wb + W::coef);
  double *gh = reinterpret_cast<double *>(wb + W::gh);
  LinkRec<double> *recb = reinterpret_cast<LinkRec<double> *>(wb + W::rec);
  double2 *gbuf = reinterpret_cast<double2 *>(wb + W::gbuf);

  const double2 *zin = reinterpret_cast<const double2 *>(c.zin.body);
  double *out = reinterpret_cast<double *>(c.out.body);
  const double *yv = reinterpret_cast<const double *>(c.y.body);
  const bool has_y = yv != nullptr;
  const LinkRec<double> *recs = reinterpret_cast<const LinkRec<double> *>(c.recs_body);
  const int Ep = c.Ep;
  const double ch = a.ch;

  // the lane's pairs (i <= jj, numbered row by row): i << 8 | jj
  int pairs[(N * (N + 1) / 2 + 31) / 32];
#pragma unroll
  for (int t0 = 0; t0 < N * (N + 1) / 2; t0 += 32) {
    const int t = t0 + lane;
    int i = 0;
#pragma unroll
    for (int w = 1; w < N; ++w) i += t >= w * N - w * (w - 1) / 2;
    pairs[t0 / 32] = i << 8 | (t - (i * N - i * (i - 1) / 2) + i);
  }

  const int n_chunks = (c.u_end - c.u_begin + G - 1) / G;
  const int nwarps = gridDim.x * S::WARPS;
  for (int chn = blockIdx.x * S::WARPS + warp; chn < n_chunks; chn += nwarps) {
    const int u0 = c.u_begin + chn * G;
    const int cnt = min(G, c.u_end - u0);
    // lane a <= cnt holds link_off[u0 + a]
    const int64_t off = (lane <= cnt) ? c.link_off[u0 + lane] : (int64_t)0;
    // per-ADO coefficients of this chunk
    for (int t = lane; t < cnt * N; t += 32) {
      const int ad = t / N, i = t - ad * N;
      coef[t] = fma(-0.5, c.gsum[u0 + ad], -a.term[i]);
    }
    if (lane < cnt) gh[lane] = -0.5 * c.gsum[u0 + lane];
    __syncwarp();

    for (int q = 0; q < P; ++q) {
      // ADOs whose last column falls in this pass: [fa, fb)
      const int fa = (32 * q) / C, fb = min((32 * q + 32) / C, cnt);
      // first record batch of each finalising ADO (at most 2 per pass for C >= 16) and its gathers
      int nrf0 = 0, nrf1 = 0;
      for (int f = fa, k = 0; f < fb; ++f, ++k) {
        const int64_t lo = __shfl_sync(0xffffffffu, off, f), hi = __shfl_sync(0xffffffffu, off, f + 1);
        const int nr = heom_rec_batch(c.err, lo, (int)min(hi - lo, (int64_t)RB), 0, c.n_recs);
        if (k == 0) nrf0 = nr;
        else nrf1 = nr;
        col_load_recs(recs, lo, nr, recb + k * RB, lane);
      }
      // this pass's column: lane -> (ADO ad, part p, column j)
      const int col = 32 * q + lane;
      const int ad = col / C, rem = col - ad * C;
      const int p = rem / N, j = rem - p * N;
      const bool act = ad < cnt;
      double zc[N];  // column j of the part that H multiplies: Im s for Q_re, Re s for Q_im
      if (act) {
        const double *zt = reinterpret_cast<const double *>(zin + (int64_t)(u0 + ad) * Ep + j) + (1 - p);
#pragma unroll
        for (int k = 0; k < N; ++k) zc[k] = zt[2 * k * N];
      }
      col_wait_all();
      __syncwarp();
      for (int f = fa, k = 0; f < fb; ++f, ++k)
        col_gather<N>(c, zin, Ep, recb + k * RB, k == 0 ? nrf0 : nrf1, gbuf + k * RB * N, lane);
      if (act) {
        // p = 0: Q_re = H Im s + coef Re s;  p = 1: Q_im = -H Re s + coef Im s
        int key = 0;
#pragma unroll
        for (int k = 0; k < N; ++k) key = max(key, fx_key(zc[k]));
        double *qs = qring + (ad % S::RING) * 2 * E + p * E;
        if (fx_ok(a.ex << 20, key)) {
          const int ex = fx_exp(key);
          int2 src[N];
          int rest[N];
#pragma unroll
          for (int k = 0; k < N; ++k) src[k] = fx_split(p ? col_neg(zc[k]) : zc[k], ex, rest[k]);
          const double *cf = coef + ad * N;
          const double gd = gh[ad];
          const int e2 = key ? fx_unit(a.ex << 20, key) : 0;  // a zero column: any scale in range
          unsigned weak = 0;  // rows to be taken from the FMA chain: after the loop, whose rows then overlap
          const double *zo = reinterpret_cast<const double *>(zin + (int64_t)(u0 + ad) * Ep + j) + p;  // own part
          // Rows in a loop, one at a time: unrolled over all of them the code outgrew the instruction cache and the kernel
          // took more than twice as long (two limbs: 20 ms per launch against 8.4); two at a time 182 ms for four steps at the
          // LHCII size, one 177 (3 CTAs per SM with 168 registers: 188)
#pragma unroll 1
          for (int i = 0; i < N; ++i) {
            const double own = zo[2 * i * N], ci = i == j ? gd : cf[i];
            FxSum r;
#pragma unroll
            for (int k = 0; k < N; ++k) {
              const int4 hx = Hs[i * N + k];
              r.add(hx.x, hx.y, hx.z, src[k].x, src[k].y, rest[k]);
            }
            unsigned f;
            const long long w = r.whole(f);
            weak |= (unsigned)fx_weak(w) << i;
            qs[i * N + j] = fma(ci, own, fx_double_add(w, f, e2));
          }
          if (weak && key) {
            for (int i = 0; i < N; ++i)
              if (weak >> i & 1)
                qs[i * N + j] = fma(i == j ? gd : cf[i], zo[2 * i * N], col_fma_row<N>(a, zin + (int64_t)(u0 + ad) * Ep + j, p, i));
          }
        } else {
          col_fma<N>(a, zin + (int64_t)(u0 + ad) * Ep + j, p, j, c.gsum[u0 + ad], qs);
        }
      }
      col_wait_all();  // gathers
      __syncwarp();
      // finalise every ADO completed in this pass
      for (int f = fa, k = 0; f < fb; ++f, ++k) {
        const int u = u0 + f;
        double *qs = qring + (f % S::RING) * 2 * E;
        const int64_t lo = __shfl_sync(0xffffffffu, off, f), hi = __shfl_sync(0xffffffffu, off, f + 1);
        const int nr0 = k == 0 ? nrf0 : nrf1;
        col_links<N>(recb + k * RB, nr0, gbuf + k * RB * N, qs, lane);
        for (int64_t blo = lo + nr0; blo < hi; blo += RB) {  // further record batches
          __syncwarp();
          const int nr = heom_rec_batch(c.err, blo, (int)min(hi - blo, (int64_t)RB), 0, c.n_recs);
          col_load_recs(recs, blo, nr, recb + k * RB, lane);
          col_wait_all();
          __syncwarp();
          col_gather<N>(c, zin, Ep, recb + k * RB, nr, gbuf + k * RB * N, lane);
          col_wait_all();
          __syncwarp();
          col_links<N>(recb + k * RB, nr, gbuf + k * RB * N, qs, lane);
        }
        __syncwarp();
        {  // R = Q + Q^dagger, out = y + ch R: lane t takes pairs t, t + 32, ... (i <= j, row by row)
          const double2 *y2 = reinterpret_cast<const double2 *>(yv) + (int64_t)u * Ep;
          double2 *o2 = reinterpret_cast<double2 *>(out) + (int64_t)u * Ep;
          constexpr int PR = N * (N + 1) / 2;
#pragma unroll
          for (int t0 = 0; t0 < PR; t0 += 32) {
            const int t = t0 + lane;
            if (t < PR) {
              const int i = pairs[t0 / 32] >> 8, jj = pairs[t0 / 32] & 255;
              double2 yr = make_double2(0, 0);
              if (has_y) yr = y2[i * N + jj];
              const double rx = qs[i * N + jj] + qs[jj * N + i];  // Re R symmetric, Im R antisymmetric
              const double ry = qs[E + i * N + jj] - qs[E + jj * N + i];
              double2 o;
              o.x = has_y ? fma(ch, rx, yr.x) : ch * rx;
              o.y = has_y ? fma(ch, ry, yr.y) : ch * ry;
              o2[i * N + jj] = o;
              if (i != jj) o2[jj * N + i] = make_double2(o.x, col_neg(o.y));
            }
          }
        }
        __syncwarp();
      }
    }
  }
  col_wait_all();
}

template <int N>
int launch_col(const StageCommon &c, double ch, const double *term, const double *H, cudaStream_t st,
               int sm_count) {
  ColArgs a;
  a.c = c;
  a.ch = ch;
  double top = 0;
  for (int i = 0; i < c.n * c.n; ++i) top = std::max(top, std::fabs(H[i]));
  a.ex = top > 0 && std::isfinite(top) ? std::min(std::max(std::ilogb(top) + 1023, 1), 2046) : top > 0 ? 2047 : 1023;
  for (int i = 0; i < kMaxStates; ++i) a.term[i] = (i < c.n) ? term[i] : 0.0;
  for (int i = 0; i < kMaxStates * kMaxStates; ++i) {
    a.H[i] = 0.0;
    a.Hx[i] = make_int4(0, 0, 0, 0);
  }
  for (int i = 0; i < c.n; ++i)
    for (int j = 0; j < c.n; ++j) {
      const double h = H[i * c.n + j];
      a.H[i * kMaxStates + j] = h;
      if (a.ex == 2047) continue;
      // as fx_split: |h| < 2^(ex - 1022); the last limb rounded
      const double x = std::ldexp(h, 2 * kFxBits - 1 - (a.ex - 1022));
      const long long v = std::llrint(x);
      const long long lo = ((v + (1ll << (kFxBits - 1))) & ((1ll << kFxBits) - 1)) - (1ll << (kFxBits - 1));
      a.Hx[i * kMaxStates + j] = make_int4((int)((v - lo) >> kFxBits), (int)lo, (int)std::llrint(std::ldexp(x - (double)v, kFxBits)), 0);
    }
  constexpr int WARPS = ColShape<N>::WARPS;
  const size_t smem = (size_t)WARPS * ColSmem<N>::total;
  static int per_sm = 0;
  if (per_sm == 0) {
    if (smem > 48 * 1024) {
      cudaError_t e = cudaFuncSetAttribute(stage_col_kernel<N>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
      if (e != cudaSuccess) {
        set_error(std::string("column stage kernel: shared memory attribute: ") + cudaGetErrorString(e));
        return -4;
      }
    }
    int ps = 0;
    cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&ps, stage_col_kernel<N>, WARPS * 32, smem);
    if (e != cudaSuccess || ps < 1) {
      set_error(std::string("column stage kernel: occupancy query failed or zero blocks: ") + cudaGetErrorString(e));
      return -4;
    }
    per_sm = ps;
  }
  constexpr int G = ColShape<N>::G;
  const int n_chunks = (c.u_end - c.u_begin + G - 1) / G;
  const int blocks_needed = (n_chunks + WARPS - 1) / WARPS;
  const int grid = std::max(1, std::min(blocks_needed, sched_ctas(per_sm, c.occ_pct) * sm_count));
  stage_col_kernel<N><<<grid, WARPS * 32, smem, st>>>(a);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) {
    set_error(std::string("column stage kernel launch: ") + cudaGetErrorString(e));
    return -4;
  }
  return 0;
}

}  // namespace heom
