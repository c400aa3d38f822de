// The FP64 reciprocal, quotient and square root of csrc/fp64_util.cuh on arrays of host values.
#include "fp64_util.cuh"

__global__ void probe(int which, int n, const double *a, const double *b, double *out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  if (which == 0) out[i] = mhd::rcp3(a[i]);
  if (which == 1) out[i] = mhd::quotient(a[i], b[i], mhd::rcp3(b[i]));
  if (which == 2) out[i] = mhd::sqrt3(a[i]);
  if (which == 3) out[i] = mhd::rcp3_covers(a[i]) ? 1.0 : 0.0;
  if (which == 4) out[i] = mhd::rcp_any(a[i]);
}

// Returns the CUDA status (0: success).
extern "C" int fp64_util_probe(int which, int n, const double *a, const double *b, double *out) {
  double *d = nullptr;
  const size_t bytes = (size_t)n * sizeof(double);
  cudaError_t e = cudaMalloc(&d, 3 * bytes);
  if (e != cudaSuccess) return (int)e;
  e = cudaMemcpy(d, a, bytes, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMemcpy(d + n, b, bytes, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) {
    probe<<<(n + 255) / 256, 256>>>(which, n, d, d + n, d + 2 * n);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaMemcpy(out, d + 2 * n, bytes, cudaMemcpyDeviceToHost);
  cudaFree(d);
  return (int)e;
}
