// Elements of a hierarchy state in any layout, and the FP64 observable record of sigma_0.
#pragma once
#include <cuda_runtime.h>

#include <cstdint>

#include "heom_internal.h"

namespace heom {

__device__ __forceinline__ double2 ld_any(const StateView &s, int E, int Ep, int u_split, int body_fp32, int64_t v,
                                          int64_t e) {
  if (v < u_split) return __ldcg(s.head + v * E + e);
  if (body_fp32) {
    const float2 f = __ldcg(reinterpret_cast<const float2 *>(s.body) + (v - u_split) * Ep + e);
    return make_double2(f.x, f.y);
  }
  return __ldcg(reinterpret_cast<const double2 *>(s.body) + (v - u_split) * Ep + e);
}

// Element e = i n + j of ADO v in the run's layout: matrix tiles, or (vec) column 0 only.
__device__ __forceinline__ double2 ld_elem(const StateView &s, int n, int Ep, int u_split, int body_fp32, int vec,
                                           int64_t v, int64_t e) {
  if (!vec) return ld_any(s, n * n, Ep, u_split, body_fp32, v, e);
  const int64_t i = e / n, j = e - i * n;
  if (j != 0) return make_double2(0.0, 0.0);
  return ld_any(s, n, n, u_split, body_fp32, v, i);
}

// One observable record of sigma_0 (FP64) by the lanes of one warp: populations, trace, dipole correlation,
// Hermiticity.  Lane a handles rows a, a + 32, ...; sums and the maximum are reduced across the warp.
// A row of a Hermitian sigma_0 differs from its column by exactly zero, and hypot(0, 0) = 0 leaves the
// maximum as it is, so hypot runs only where a difference is not zero: it was the serial chain that
// made a record cost up to 14 us (29 states).  Loads go past the L1 cache (see resident.cuh).
__device__ __forceinline__ void record_warp(const StateView &y, int u_split, int body_fp32, int vec, int n, const double *w,
                                            double *records, int64_t *rec_count, int64_t max_records) {
  const int lane = threadIdx.x & 31;
  const int64_t idx = __ldcg(reinterpret_cast<const long long *>(rec_count));
  if (idx >= max_records) return;
  const int E = n * n;
  double *rec = records + idx * (n + 5);
  double tr = 0, ti = 0, cr = 0, ci = 0, herm = 0;
  for (int a = lane; a < n; a += 32) {
    const double2 d = ld_elem(y, n, E, u_split, body_fp32, vec, 0, (int64_t)a * n + a);
    rec[a] = d.x;
    tr += d.x;
    ti += d.y;
    const double2 c0 = ld_elem(y, n, E, u_split, body_fp32, vec, 0, (int64_t)a * n);
    cr += w[a] * c0.x;
    ci += w[a] * c0.y;
#pragma unroll 4
    for (int b = 0; b < n; ++b) {
      const double2 x = ld_elem(y, n, E, u_split, body_fp32, vec, 0, (int64_t)a * n + b);
      const double2 z = ld_elem(y, n, E, u_split, body_fp32, vec, 0, (int64_t)b * n + a);
      const double dx = x.x - z.x, dy = x.y + z.y;
      if (dx != 0.0 || dy != 0.0) herm = fmax(herm, hypot(dx, dy));
    }
  }
  for (int o = 16; o > 0; o >>= 1) {
    tr += __shfl_down_sync(0xffffffffu, tr, o);
    ti += __shfl_down_sync(0xffffffffu, ti, o);
    cr += __shfl_down_sync(0xffffffffu, cr, o);
    ci += __shfl_down_sync(0xffffffffu, ci, o);
    herm = fmax(herm, __shfl_down_sync(0xffffffffu, herm, o));
  }
  if (lane == 0) {
    rec[n] = tr;
    rec[n + 1] = ti;
    rec[n + 2] = cr;
    rec[n + 3] = ci;
    rec[n + 4] = herm;
    *rec_count = idx + 1;
  }
}

}  // namespace heom
