// gram_schmidt.cuh -- orthogonalisation of a Krylov vector on the device.
#pragma once

#include <algorithm>
#include <cstdint>

#include <cuda_runtime.h>

#include "fp_bits.cuh"

namespace crn {

constexpr int NKB = 256;  // threads per block of the elementwise kernels
constexpr int NKD = 512;  // threads per block of the Gram-Schmidt kernels
constexpr int MD = 8;     // vectors a Gram-Schmidt pass takes at a time

// whether this block is the last of the grid to get here; its threads then see
// everything the others wrote before (*counter is zero before and after)
__device__ __forceinline__ bool last_block(unsigned int* counter) {
  __shared__ unsigned int s_last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) {
    s_last = atomicAdd(counter, 1u) == gridDim.x * gridDim.y - 1 ? 1u : 0u;
    if (s_last) *counter = 0u;
  }
  __syncthreads();
  if (!s_last) return false;
  __threadfence();
  return true;
}

// an FP32 Krylov vector widens on the integer pipe (exact): the FP64 pipe also
// runs the conversion instruction
__device__ __forceinline__ double as_double(float x) { return widen_f32(x); }
__device__ __forceinline__ double as_double(double x) { return x; }

// ---- Gram-Schmidt on the device -------------------------------------------
// Classical Gram-Schmidt of w against V_0 .. V_(cnt-1), repeated once if the
// norm dropped to below 0.7: dots, update (which also takes the new norm and
// decides), and the same two kernels again, which return at once if the repeat
// is not needed.  The host reads the column of the Hessenberg matrix once per
// Krylov step.  An FP32 basis keeps the products on the FP32 pipe (GB300 runs
// FP64 FMAs at 1/64 of the FP32 rate): sums over a thread's elements in FP32
// with a running compensation (one rounding a term, however long the vector:
// plain sums of the 121 terms a thread has of 128 x 64 x 128 cells lost 29 where
// the products were alike), across threads in FP64.  What bounds these kernels is the traffic of V for
// large shells and, for small ones, the FP64 adds of the reductions, which a
// warp issues at one per 16 clocks: eight sums of 32 lanes take 9 adds by
// recursive halving (40 with a shuffle tree each), the grid is one block per SM
// so that few partials remain, and the last block adds those.  A Krylov step's
// products with V on 32 x 16 x 32: four launches of 13 us (cold), where sums over
// one vector at a time took five of 20 us and five of 5 us over their partials.
struct GsOut {
  double* h;             // [m + 1] the column: h_t
  double* ww;            // [1] |w|^2 before the first pass
  double* after;         // [1] |w|^2 after the last pass
  double* inv;           // [1] 1 / |w| then (0 for w = 0)
  double* coef;          // [m + 1] -h_t of the pass
  double* redo;          // [1] 1: the second pass is needed
  unsigned int* counter;
};

template <class T> struct Vec;
template <> struct Vec<float> { using type = float4; static constexpr int N = 4; };
template <> struct Vec<double> { using type = double2; static constexpr int N = 2; };
// a thread's sum of products
template <class T> struct Dot;
template <> struct Dot<double> {
  double s = 0.0;
  __device__ __forceinline__ void add(const double2& a, const double2& b) { s = fma(a.y, b.y, fma(a.x, b.x, s)); }
  __device__ __forceinline__ double total() const { return s; }
};
template <> struct Dot<float> {
  float s = 0.f, c = 0.f;  // the sum and what its last addition rounded up by
  __device__ __forceinline__ void add(float a, float b) {
    const float y = fmaf(a, b, -c), t = s + y;
    c = (t - s) - y;
    s = t;
  }
  __device__ __forceinline__ void add(const float4& a, const float4& b) {
    add(a.x, b.x); add(a.y, b.y); add(a.z, b.z); add(a.w, b.w);
  }
  __device__ __forceinline__ double total() const { return as_double(s) - as_double(c); }
};
__device__ __forceinline__ void vaxpy(float4& w, float c, const float4& v) {
  w.x = fmaf(c, v.x, w.x); w.y = fmaf(c, v.y, w.y); w.z = fmaf(c, v.z, w.z); w.w = fmaf(c, v.w, w.w);
}
__device__ __forceinline__ void vaxpy(double2& w, double c, const double2& v) {
  w.x = fma(c, v.x, w.x); w.y = fma(c, v.y, w.y);
}

// eight sums over a warp by recursive halving: lane l returns the sum of
// a[l >> 2] (the same in its group of four lanes)
__device__ __forceinline__ double warp_sum8(double (&a)[MD], int lane) {
#pragma unroll
  for (int w = 4, bit = 16; w > 0; w >>= 1, bit >>= 1) {
    const bool hi = (lane & bit) != 0;
#pragma unroll
    for (int t = 0; t < w; ++t) {
      const double give = hi ? a[t] : a[t + w], keep = hi ? a[t + w] : a[t];
      a[t] = keep + __shfl_xor_sync(0xffffffffu, give, bit);
    }
  }
  double s = a[0];
  s += __shfl_xor_sync(0xffffffffu, s, 2);
  s += __shfl_xor_sync(0xffffffffu, s, 1);
  return s;
}

// the block's sums of eight values per thread into part[(row + t) * nblk + block], t < cnt
__device__ __forceinline__ void block_sum8(double (&a)[MD], double* part, int nblk, int row, int cnt) {
  __shared__ double sm[(NKD / 32) * MD];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const double s = warp_sum8(a, lane);
  __syncthreads();  // sm may still be read for the previous eight
  if ((lane & 3) == 0) sm[wid * MD + (lane >> 2)] = s;
  __syncthreads();
  if ((int)threadIdx.x < cnt) {
    double x = 0.0;
#pragma unroll
    for (int q = 0; q < NKD / 32; ++q) x += sm[q * MD + threadIdx.x];
    part[(size_t)(row + threadIdx.x) * nblk + blockIdx.x] = x;
  }
}

// the last block's sums over the partials of `rows` rows: one warp takes eight
// rows at a time; put(row, sum) runs on one lane per row
template <class F>
__device__ __forceinline__ void sum_partials(const double* part, int nblk, int rows, F put) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  for (int r0 = wid * MD; r0 < rows; r0 += (NKD / 32) * MD) {
    double a[MD];
#pragma unroll
    for (int t = 0; t < MD; ++t) {
      a[t] = 0.0;
      if (r0 + t < rows)
        for (int q = lane; q < nblk; q += 32) a[t] += __ldcg(part + (size_t)(r0 + t) * nblk + q);
    }
    const double s = warp_sum8(a, lane);
    const int r = r0 + (lane >> 2);
    if ((lane & 3) == 0 && r < rows) put(r, s);
  }
}

// h_t = <V_t, w> for t < cnt; pass 0 also |w|^2, pass 1 only if the repeat is
// needed, its h_t added to the first's
template <class TV>
__global__ void __launch_bounds__(NKD)
gs_dots_kernel(const TV* __restrict__ V, int64_t n, int cnt, const TV* __restrict__ w, double* __restrict__ part,
               GsOut o, int pass) {
  if (pass == 1 && *o.redo == 0.0) return;
  using V4 = typename Vec<TV>::type;
  const int64_t nv = n / Vec<TV>::N;
  const int64_t stride = (int64_t)gridDim.x * NKD, first = (int64_t)blockIdx.x * NKD + threadIdx.x;
  const V4* w4 = reinterpret_cast<const V4*>(w);
  const int nblk = gridDim.x;
  // rows: the cnt dots, then |w|^2; block y takes eight vectors (their dots side
  // by side: one after the other, a small shell's took 20 us for 16)
  if (pass == 0 && blockIdx.y == 0) {
    Dot<TV> s;
    for (int64_t e = first; e < nv; e += stride) { const V4 x = w4[e]; s.add(x, x); }
    double b[MD] = {s.total()};
    block_sum8(b, part, nblk, cnt, 1);
  }
  const int i0 = blockIdx.y * MD, c = min(MD, cnt - i0);
  if (c > 0) {
    const V4* v4 = reinterpret_cast<const V4*>(V + (int64_t)i0 * n);
    Dot<TV> a[MD];
    if (c == MD) {
      for (int64_t e = first; e < nv; e += stride) {
        const V4 x = w4[e];
#pragma unroll
        for (int t = 0; t < MD; ++t) a[t].add(v4[(int64_t)t * nv + e], x);
      }
    } else {
      for (int64_t e = first; e < nv; e += stride) {
        const V4 x = w4[e];
#pragma unroll
        for (int t = 0; t < MD; ++t)
          if (t < c) a[t].add(v4[(int64_t)t * nv + e], x);
      }
    }
    double b[MD];
#pragma unroll
    for (int t = 0; t < MD; ++t) b[t] = a[t].total();
    block_sum8(b, part, nblk, i0, c);
  }
  if (!last_block(o.counter)) return;
  sum_partials(part, nblk, cnt + (pass == 0 ? 1 : 0), [&](int r, double s) {
    if (r == cnt) {
      *o.ww = s;
    } else {
      o.coef[r] = -s;
      o.h[r] = pass == 0 ? s : o.h[r] + s;
    }
  });
}

// w += sum_t coef_t V_t, then |w|^2; pass 0 decides whether the norm dropped
// enough for a second pass, pass 1 runs only then
template <class TV>
__global__ void __launch_bounds__(NKD)
gs_update_kernel(TV* __restrict__ w, const TV* __restrict__ V, int64_t n, int cnt, double* __restrict__ part,
                 GsOut o, int pass) {
  if (pass == 1 && *o.redo == 0.0) return;
  using V4 = typename Vec<TV>::type;
  __shared__ TV sc[512];
  for (int t = threadIdx.x; t < cnt; t += NKD) sc[t] = (TV)o.coef[t];
  __syncthreads();
  const int64_t nv = n / Vec<TV>::N;
  const int64_t stride = (int64_t)gridDim.x * NKD;
  const V4* v4 = reinterpret_cast<const V4*>(V);
  V4* w4 = reinterpret_cast<V4*>(w);
  Dot<TV> s;
  for (int64_t e = (int64_t)blockIdx.x * NKD + threadIdx.x; e < nv; e += stride) {
    V4 x = w4[e];
#pragma unroll 16
    for (int t = 0; t < cnt; ++t) vaxpy(x, sc[t], v4[(int64_t)t * nv + e]);
    w4[e] = x;
    s.add(x, x);
  }
  double b[MD] = {s.total()};
  block_sum8(b, part, gridDim.x, 0, 1);
  if (!last_block(o.counter)) return;
  sum_partials(part, gridDim.x, 1, [&](int, double a) {
    *o.after = a;
    *o.inv = a > 0.0 ? 1.0 / sqrt(a) : 0.0;
    if (pass == 0) *o.redo = sqrt(fmax(a, 0.0)) < 0.7 * sqrt(fmax(*o.ww, 0.0)) ? 1.0 : 0.0;
  });
}

// V_j = w / |w| (w may be V_j); nothing if |w| is 0.  1 / |w| comes from the
// update's last block: a square root and a division in every thread are 40 slots
// of the FP64 pipe, 7 us on a small shell.
template <class TV>
__global__ void __launch_bounds__(NKB)
gs_scale_kernel(TV* y, const TV* x, int64_t n, const double* __restrict__ inv) {
  using V4 = typename Vec<TV>::type;
  const TV f = (TV)*inv;
  if (!(f > (TV)0)) return;
  const int64_t nv = n / Vec<TV>::N, stride = (int64_t)gridDim.x * NKB;
  for (int64_t e = (int64_t)blockIdx.x * NKB + threadIdx.x; e < nv; e += stride) {
    V4 v = reinterpret_cast<const V4*>(x)[e];
    v.x *= f;
    v.y *= f;
    if constexpr (sizeof(TV) == 4) {
      v.z *= f;
      v.w *= f;
    }
    reinterpret_cast<V4*>(y)[e] = v;
  }
}

// blocks of the Gram-Schmidt kernels: one per SM, fewer for a short vector
template <class TV>
inline unsigned gs_blocks(int64_t n, int nsm) {
  return (unsigned)std::max<int64_t>(1, std::min<int64_t>((n / Vec<TV>::N + NKD - 1) / NKD, nsm));
}

// x orthogonalised against base_0 .. base_(cnt-1) and scaled to one; n a multiple of
// four, all vectors 16-byte aligned; part: (cnt + 1) x gs_blocks values.  Returns
// the launches made (nscale blocks for the scaling).
template <class TV>
int gs_launch(const TV* base, int64_t n, int cnt, TV* x, double* part, const GsOut& o, int nsm, unsigned nscale,
              cudaStream_t st) {
  const unsigned nb = gs_blocks<TV>(n, nsm);
  for (int pass = 0; pass < 2; ++pass) {
    gs_dots_kernel<TV><<<dim3(nb, (unsigned)((cnt + MD - 1) / MD)), NKD, 0, st>>>(base, n, cnt, x, part, o, pass);
    gs_update_kernel<TV><<<nb, NKD, 0, st>>>(x, base, n, cnt, part, o, pass);
  }
  gs_scale_kernel<TV><<<nscale, NKB, 0, st>>>(x, x, n, o.inv);
  return 5;
}

}  // namespace crn
