// The FP32 flux of a face, and the same with the other product of the momentum's
// sum rounded, for the test that compares their errors.
#include "../paper_2209_04481_gb300/csrc/mhd_device.cuh"

__global__ void fluxes(const float* wl, const float* wr, const float* nrm, float* f, float* other, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  crn::Phys<float> ph{};
  ph.gamma = 1.05f;
  ph.igm1 = 20.f;
  ph.ch = ph.ch2 = 1.f;
  float a[9], b[9], x[9], la;
  for (int v = 0; v < 9; ++v) { a[v] = wl[v * n + i]; b[v] = wr[v * n + i]; }
  const float m[3] = {nrm[i], nrm[n + i], nrm[2 * n + i]};
  crn::rusanov<true>(a, b, m[0], m[1], m[2], 1.f, ph, x, la);
  const crn::Side<float> L = crn::side_terms<true>(a, m[0], m[1], m[2], ph), R = crn::side_terms<true>(b, m[0], m[1], m[2], ph);
  const float ml = a[0] * L.un, mr = b[0] * R.un, d = 0.5f * la;
  for (int c = 0; c < 3; ++c) {
    f[c * n + i] = x[1 + c];
    const float p = fmaf(-a[4 + c], L.bn, fmaf(ml, a[1 + c], L.pt * m[c]));
    const float q = fmaf(-b[4 + c], R.bn, fmaf(mr, b[1 + c], R.pt * m[c]));
    other[c * n + i] = 0.5f * (p + q) - d * (b[0] * b[1 + c] - a[0] * a[1 + c]);
  }
}

extern "C" int run_fluxes(const float* wl, const float* wr, const float* nrm, float* f, float* other, int n) {
  fluxes<<<(n + 255) / 256, 256>>>(wl, wr, nrm, f, other, n);
  return (int)cudaDeviceSynchronize();
}
