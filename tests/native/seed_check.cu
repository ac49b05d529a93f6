// Largest relative errors of recip and rsqrt_nr (csrc/fixed.cuh) over x = m 2^e, e in -120 .. 120, against
// CUDA's FP64 division and square root (each within 2^-53 of the exact value): prints both.
#include <cstdio>

#include "fixed.cuh"

__global__ void check(double* err) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;  // 241 exponents x 1,024 significands
  if (i >= 241 * 1024) return;
  const double m = 1.0 + (i % 1024 + 0.618 * (i % 7) / 7.0) / 1025.0;
  const double x = ldexp(m, i / 1024 - 120);
  const double a = qf::recip(x), b = 1.0 / x, c = qf::rsqrt_nr(x), d = 1.0 / sqrt(x);
  const double s = qf::recip(-x);
  err[2 * i] = fmax(fabs(a - b) / b, fabs(s + b) / b);
  err[2 * i + 1] = fabs(c - d) / d;
}

int main() {
  const int n = 241 * 1024;
  double* err = nullptr;
  if (cudaMallocManaged(&err, sizeof(double) * 2 * n) != cudaSuccess) return 1;
  check<<<(n + 255) / 256, 256>>>(err);
  if (cudaDeviceSynchronize() != cudaSuccess) return 2;
  double e[2] = {0.0, 0.0};
  for (int i = 0; i < 2 * n; ++i) {
    if (!(err[i] < 1.0)) return 3;
    if (err[i] > e[i & 1]) e[i & 1] = err[i];
  }
  std::printf("%.17g %.17g\n", e[0], e[1]);
  cudaFree(err);
  return 0;
}
