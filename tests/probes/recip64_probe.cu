// recip64_probe.cu - test harness: the FP64 reciprocal of the march and the
// small-grid kernels (lanes.cuh) for a host array of x.  Built and loaded by
// tests/test_gpu_recip64.py.
#include <cuda_runtime.h>

#include "../../paper_1106_0785_gb300/csrc/lanes.cuh"

namespace {
__global__ void recip64_probe_kernel(const double* x, double* out, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) out[i] = mrtlb::split_recip(x[i]);
}
}  // namespace

extern "C" int recip64_probe(const double* x_host, double* out_host, int n) {
  double *x = nullptr, *out = nullptr;
  if (n < 1 || cudaMalloc(&x, n * sizeof(double)) != cudaSuccess) return 1;
  if (cudaMalloc(&out, n * sizeof(double)) != cudaSuccess) {
    cudaFree(x);
    return 1;
  }
  int rc = cudaMemcpy(x, x_host, n * sizeof(double), cudaMemcpyHostToDevice) != cudaSuccess;
  if (!rc) {
    recip64_probe_kernel<<<(n + 255) / 256, 256>>>(x, out, n);
    rc = cudaGetLastError() != cudaSuccess;
  }
  if (!rc) rc = cudaMemcpy(out_host, out, n * sizeof(double), cudaMemcpyDeviceToHost) != cudaSuccess;
  cudaFree(x);
  cudaFree(out);
  return rc;
}
