// Applies the FP64 reciprocals of csrc/fp64fast.cuh to an array
// (tests/test_gpu_fp64_forms.py builds and calls this).
#include "fp64fast.cuh"

__global__ void k_forms(const double *x, double *rcp, double *rsq, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  rcp[i] = sph::rcp64(x[i]);
  rsq[i] = sph::rsqrt64(x[i]);
}

extern "C" int fp64_forms(const double *x, double *rcp, double *rsq, int n, void *stream) {
  k_forms<<<(n + 255) / 256, 256, 0, (cudaStream_t)stream>>>(x, rcp, rsq, n);
  return (int)cudaGetLastError();
}
