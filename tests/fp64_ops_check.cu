// The FP64 reciprocal and square root of the flux kernels, for the test that
// compares them with the correctly rounded results.
#include "../paper_2209_04481_gb300/csrc/mhd_device.cuh"

__global__ void ops(const double* x, double* rcp, double* root, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  rcp[i] = crn::frcp(x[i]);
  root[i] = crn::fsqrt(x[i]);
}

// lambda of a face from the flux (which forms only the speeds it needs) and from
// both sides' speeds
__global__ void lambdas(const double* wl, const double* wr, const double* nrm, double ch, double* lam, double* ref,
                        int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  crn::Phys<double> ph{};
  ph.gamma = 1.05;
  ph.igm1 = 20.0;
  ph.ch = ch;
  ph.ch2 = ch * ch;
  double a[9], b[9], f[9], la;
  for (int v = 0; v < 9; ++v) { a[v] = wl[v * n + i]; b[v] = wr[v * n + i]; }
  const double nx = nrm[i], ny = nrm[n + i], nz = nrm[2 * n + i];
  crn::rusanov(a, b, nx, ny, nz, 1.0, ph, f, la);
  lam[i] = la;
  const crn::Side<double> L = crn::side_terms<true>(a, nx, ny, nz, ph), R = crn::side_terms<true>(b, nx, ny, nz, ph);
  const double sl = crn::signal_speed(a[0], a[7], L.un, L.bn, L.sp, ph);
  const double sr = crn::signal_speed(b[0], b[7], R.un, R.bn, R.sp, ph);
  double m = sl > sr ? sl : sr;
  ref[i] = m > ch ? m : ch;
}

extern "C" int run_lambdas(const double* wl, const double* wr, const double* nrm, double ch, double* lam, double* ref,
                           int n) {
  lambdas<<<(n + 255) / 256, 256>>>(wl, wr, nrm, ch, lam, ref, n);
  return (int)cudaDeviceSynchronize();
}

__global__ void quotients(const double* a, const double* b, double* q, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) q[i] = crn::quotient(a[i], b[i]);
}

extern "C" int run_quotients(const double* a, const double* b, double* q, int n) {
  quotients<<<(n + 255) / 256, 256>>>(a, b, q, n);
  return (int)cudaDeviceSynchronize();
}

extern "C" int run_ops(const double* x, double* rcp, double* root, int n) {
  ops<<<(n + 255) / 256, 256>>>(x, rcp, root, n);
  return (int)cudaDeviceSynchronize();
}
