// Small kernels of libheom: the FP64 observable record of sigma_0 and the state scatter / gather
// through the host layout.
#include <cuda_runtime.h>

#include <cstdint>

#include "heom_internal.h"
#include "record.cuh"

// ------------------------------------------------------------------------------------------------
// small kernels

namespace heom {

__global__ void record_kernel(StateView y, int u_split, int body_fp32, int vec, int n, const double *w, double *records,
                              int64_t *rec_count, int64_t max_records) {
  record_warp(y, u_split, body_fp32, vec, n, w, records, rec_count, max_records);
}

__global__ void scatter_kernel(StateView dst, int Ep, int u_split, int body_fp32, int vec, int n, int64_t u0, int64_t count,
                               const double *re, const double *im) {
  const int64_t E = (int64_t)n * n;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < count * E; t += (int64_t)gridDim.x * blockDim.x) {
    const int64_t c = t / E;
    int64_t e = t - c * E;
    const int64_t v = u0 + c;
    int64_t TE = E, TP = Ep;
    if (vec) {  // column 0 only (the host checked that the rest is zero)
      if (e % n != 0) continue;
      e /= n;
      TE = n;
      TP = n;
    }
    if (v < u_split) {
      dst.head[v * TE + e] = make_double2(re[t], im[t]);
    } else if (body_fp32) {
      reinterpret_cast<float2 *>(dst.body)[(v - u_split) * TP + e] = make_float2((float)re[t], (float)im[t]);
    } else {
      reinterpret_cast<double2 *>(dst.body)[(v - u_split) * TP + e] = make_double2(re[t], im[t]);
    }
  }
}

// status (or nullptr): takes the run's error word err, so that a small read is one copy.
__global__ void gather_kernel(StateView src, int Ep, int u_split, int body_fp32, int vec, int n, int64_t u0, int64_t count,
                              double *re, double *im, const int *err, double *status) {
  if (status && blockIdx.x == 0 && threadIdx.x == 0) *status = *err;
  const int64_t E = (int64_t)n * n;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < count * E; t += (int64_t)gridDim.x * blockDim.x) {
    const int64_t c = t / E, e = t - c * E;
    const double2 d = ld_elem(src, n, Ep, u_split, body_fp32, vec, u0 + c, e);
    re[t] = d.x;
    im[t] = d.y;
  }
}

}  // namespace heom
