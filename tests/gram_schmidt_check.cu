// The Gram-Schmidt launches of the Newton-Krylov solver on vectors of the caller,
// for the test that compares them with sums in 64 bits.
#include "../paper_2209_04481_gb300/csrc/gram_schmidt.cuh"

// out: h[cnt], then |w|^2 before, |w|^2 after, 1 / |w|, whether the pass was repeated
template <class TV>
int run(const TV* V, long long n, int cnt, TV* x, double* part, double* coef, unsigned int* counter, double* out,
        int nsm) {
  const crn::GsOut o{out, out + cnt, out + cnt + 1, out + cnt + 2, coef, out + cnt + 3, counter};
  crn::gs_launch<TV>(V, n, cnt, x, part, o, nsm, 1024, nullptr);
  return (int)cudaDeviceSynchronize();
}

extern "C" int run32(const float* V, long long n, int cnt, float* x, double* part, double* coef, unsigned int* counter,
                     double* out, int nsm) {
  return run<float>(V, n, cnt, x, part, coef, counter, out, nsm);
}
extern "C" int run64(const double* V, long long n, int cnt, double* x, double* part, double* coef,
                     unsigned int* counter, double* out, int nsm) {
  return run<double>(V, n, cnt, x, part, coef, counter, out, nsm);
}
