// The FP64 reciprocal and square root of the flux kernels, for the test that
// compares them with the correctly rounded results.
#include "../paper_2209_04481_gb300/csrc/mhd_device.cuh"

__global__ void ops(const double* x, double* rcp, double* root, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  rcp[i] = crn::frcp(x[i]);
  root[i] = crn::fsqrt(x[i]);
}

extern "C" int run_ops(const double* x, double* rcp, double* root, int n) {
  ops<<<(n + 255) / 256, 256>>>(x, rcp, root, n);
  return (int)cudaDeviceSynchronize();
}
