// Index arithmetic of cells and faces, and the least-squares weight (shared by the build kernels).
#pragma once
#include <math.h>
#include <stdint.h>

#include "eb_internal.cuh"

namespace eb {

__device__ __forceinline__ void cell_xyz(const Dims& dm, int64_t c, int* x) {
  const uint32_t q = (uint32_t)c, n0 = (uint32_t)dm.n[0], n1 = (uint32_t)dm.n[1], r = q / n0;  // ids are below 2^32
  x[0] = (int)(q - r * n0);
  x[2] = (int)(r / n1);
  x[1] = (int)(r - (uint32_t)x[2] * n1);
}
__device__ __forceinline__ int64_t cell_id(const Dims& dm, const int* x) {
  return (int64_t)x[0] + (int64_t)dm.n[0] * ((int64_t)x[1] + (int64_t)dm.n[1] * x[2]);
}
__device__ __forceinline__ bool in_domain(const Dims& dm, const int* x) {
  for (int d = 0; d < 3; ++d)
    if (x[d] < 0 || x[d] >= dm.n[d]) return false;
  return true;
}
// local index of the face normal to d whose coordinates are x (x[d] in 0..n_d)
__device__ __forceinline__ int64_t face_local(const Dims& dm, int d, const int* x) {
  int64_t m0 = dm.n[0] + (d == 0), m1 = dm.n[1] + (d == 1);
  return (int64_t)x[0] + m0 * ((int64_t)x[1] + m1 * x[2]);
}
__device__ __forceinline__ void face_xyz(const Dims& dm, int d, int64_t f, int* x) {
  const uint32_t q = (uint32_t)f, m0 = (uint32_t)(dm.n[0] + (d == 0)), m1 = (uint32_t)(dm.n[1] + (d == 1)), r = q / m0;
  x[0] = (int)(q - r * m0);
  x[2] = (int)(r / m1);
  x[1] = (int)(r - (uint32_t)x[2] * m1);
}

__device__ __forceinline__ double weight_of(const Dims& dm, double r2) {
  // Sec. 2.4: W_ii = 1 if r < 1/2, else (2r)^-5, r = |x_i - x0| / h
  if (!dm.weighted || r2 < dm.w_threshold * dm.w_threshold) return 1.0;
  return pow(4.0 * r2, -0.5 * dm.w_power);
}

}  // namespace eb
