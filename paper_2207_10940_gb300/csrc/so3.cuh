// FP64 rotation algebra for the solver kernels (Sec. II conventions, Eq. 2).
// Hamilton quaternions (w, x, y, z); 3x3 matrices row-major; global (left)
// perturbations q <- exp(da) (x) q.
#pragma once

#include <cuda_runtime.h>

namespace dri {

// Below this theta^2 (theta < 0.05 rad) the rotation functions use their Taylor
// series in theta^2 (five terms, relative error below 1e-16 there): on this GPU a
// dependent FP64 FMA costs ~64 cycles but a sincos ~1.4k and a sqrt or divide
// several hundred, and most angles here (IMU pieces, residuals, GN steps) are small.
constexpr double kSeriesT2 = 2.5e-3;

__device__ __forceinline__ void m3_vec(const double* A, const double* x, double* y) {
#pragma unroll
  for (int i = 0; i < 3; ++i) y[i] = A[3 * i] * x[0] + A[3 * i + 1] * x[1] + A[3 * i + 2] * x[2];
}

__device__ __forceinline__ void hat3(const double* w, double* K) {
  K[0] = 0.0;   K[1] = -w[2]; K[2] = w[1];
  K[3] = w[2];  K[4] = 0.0;   K[5] = -w[0];
  K[6] = -w[1]; K[7] = w[0];  K[8] = 0.0;
}

// Rotation matrix of a unit quaternion (every quaternion stored here is kept unit).
__device__ __forceinline__ void quat_to_rot(const double* q, double* R) {
  const double w = q[0], x = q[1], y = q[2], z = q[3];
  R[0] = 1 - 2 * (y * y + z * z); R[1] = 2 * (x * y - w * z);     R[2] = 2 * (x * z + w * y);
  R[3] = 2 * (x * y + w * z);     R[4] = 1 - 2 * (x * x + z * z); R[5] = 2 * (y * z - w * x);
  R[6] = 2 * (x * z - w * y);     R[7] = 2 * (y * z + w * x);     R[8] = 1 - 2 * (x * x + y * y);
}

}  // namespace dri
