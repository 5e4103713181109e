// residual.cuh -- residual kernels of the MHD + GLM finite-volume operator.
//
// Two kernels evaluate the same operator R = dU/dt (arXiv 2209.04481,
// Sect. 2.1 second-order FV + HDC, Sect. 2.2 equations, Sect. 3.2 inner
// boundary, Sect. 4.1 outer boundary):
//
//  * residual_tiled   -- the production kernel.  A CTA owns a TT x TP block of
//    (theta, phi) columns and marches outwards in r over a chunk of planes.
//    Each cell (and a 2-cell theta/phi halo) is loaded and its primitives
//    recovered once per tile; a thread keeps its own column in registers, the
//    neighbours see the plane in shared memory.  Every face flux of the tile is
//    computed once and gathered by the two cells it separates (no atomics).
//    Residual norms and the step bound are reduced per thread, per warp
//    (shuffles), per CTA, and across CTAs by the last CTA to finish (fixed
//    order, bitwise reproducible).
//  * residual_cellwise -- a deliberately simple reference kernel: one thread
//    per cell re-evaluates all six of its faces from global memory.
#pragma once

#include "mhd_device.cuh"

namespace crn {

// where the reductions and error reports go
struct Reduce {
  double* partials;          // [gridDim.x * gridDim.y][16]
  unsigned int* counter;     // CTA arrival counter, reset by the last CTA
  double* norms_out;         // [9] L2 norms, where the kernel forms them
  double* dt_out;            // [1] min V / sum lambda |S|, likewise
  double* norms_user;        // optional copy for the caller
  double* dt_user;           // optional copy for the caller
  unsigned int* err_flags;   // bit 0: non-physical or non-finite cell
  unsigned long long* err_cell;  // lowest flagged cell
  double* log_out;           // if set: write log10 of the 9 norms here instead
};

// ---------------------------------------------------------------------------
// accumulators: FP64 directly, or compensated FP32 (Kahan) per thread that is
// promoted to FP64 for the cross-thread reduction
// ---------------------------------------------------------------------------
template <class T> struct Acc;
template <> struct Acc<double> {
  double s[NV];
  __device__ void init() {
#pragma unroll
    for (int v = 0; v < NV; ++v) s[v] = 0.0;
  }
  __device__ __forceinline__ void add(int v, double x) { s[v] = fma(x, x, s[v]); }
  __device__ double total(int v) const { return s[v]; }
};
template <> struct Acc<float> {
  float s[NV], c[NV];
  __device__ void init() {
#pragma unroll
    for (int v = 0; v < NV; ++v) { s[v] = 0.f; c[v] = 0.f; }
  }
  __device__ __forceinline__ void add(int v, float x) {
    const float y = fmaf(x, x, -c[v]);
    const float t = s[v] + y;
    c[v] = (t - s[v]) - y;
    s[v] = t;
  }
  __device__ double total(int v) const { return (double)s[v] - (double)c[v]; }
};

__device__ __forceinline__ void flag_bad(const Reduce& red, long long cell) {
  atomicOr(red.err_flags, 1u);
  atomicMin(red.err_cell, (unsigned long long)cell);
}

// the smaller of two positive doubles (or +inf), on the integer pipe
__device__ __forceinline__ double min_positive(double a, double b) {
  return __double_as_longlong(b) < __double_as_longlong(a) ? b : a;
}

// Block + grid reduction of 9 sums of squares and one minimum from the warps'
// values (S = float or double; lane 0 of every warp holds its warp's).  Every
// thread of every CTA calls it once at the end of the kernel.  The FP64 adds
// of one warp take 16 clocks of the SM's FP64 pipe however few lanes are
// active, and the last CTA's are the tail of the whole launch, so they are
// packed: ten threads add and convert the block's warp sums, and the last CTA
// reads the partials 16 lanes to a row of ten (320 rows: 160 warp adds, where
// one row per thread with a shuffle tree per quantity took 540).
template <int NTHREADS, class S>
__device__ void reduce_and_finalize_at(const S (&sum)[NV], S dtmin, const Reduce& red,
                                       double* scratch /* >= (NTHREADS/32) * RED_STRIDE doubles */,
                                       int bid, int nblocks) {
  constexpr int NW = NTHREADS / 32;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  S* sc = reinterpret_cast<S*>(scratch);
  __syncthreads();  // scratch may alias buffers still in use
  if (lane == 0) {
#pragma unroll
    for (int q = 0; q < NV; ++q) sc[warp * RED_STRIDE + q] = sum[q];
    sc[warp * RED_STRIDE + NV] = dtmin;
  }
  __syncthreads();
  if (threadIdx.x <= NV) {
    const int q = threadIdx.x;
    double a = (double)sc[q];
    for (int w = 1; w < NW; ++w) {
      const double x = (double)sc[w * RED_STRIDE + q];
      a = q < NV ? a + x : min_positive(a, x);
    }
    red.partials[(size_t)bid * RED_STRIDE + q] = a;
  }
  __shared__ unsigned int s_last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) s_last = (atomicAdd(red.counter, 1u) == (unsigned)(nblocks - 1));
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  // last CTA: fixed-order reduction of all partials
  constexpr int NS = NTHREADS / RED_STRIDE;
  const int q = threadIdx.x % RED_STRIDE;
  double acc = q < NV ? 0.0 : INFINITY;
  if (q <= NV) {
#pragma unroll 4
    for (int b = threadIdx.x / RED_STRIDE; b < nblocks; b += NS) {
      const double x = __ldcg(red.partials + (size_t)b * RED_STRIDE + q);
      acc = q < NV ? acc + x : min_positive(acc, x);
    }
  }
  {
    const double x = __shfl_xor_sync(0xffffffffu, acc, RED_STRIDE);
    acc = q < NV ? acc + x : min_positive(acc, x);
  }
  if (lane <= NV) scratch[warp * RED_STRIDE + lane] = acc;
  __syncthreads();
  if (threadIdx.x <= NV) {
    double a = scratch[q];
    for (int w = 1; w < NW; ++w) {
      const double x = scratch[w * RED_STRIDE + q];
      a = q < NV ? a + x : min_positive(a, x);
    }
    if (red.log_out) {
      if (q < NV) red.log_out[q] = log10(sqrt(a));
    } else if (q < NV) {
      const double nrm = sqrt(a);
      red.norms_out[q] = nrm;
      if (red.norms_user) red.norms_user[q] = nrm;
    } else {
      red.dt_out[0] = a;
      if (red.dt_user) red.dt_user[0] = a;
    }
  }
  if (threadIdx.x == 0) *red.counter = 0u;
}

// The minimum alone (the pseudo-time march wants the step bound, not the norms):
// no sums to carry, add and convert, and a last CTA that reads one double per
// CTA: 5 us of a pseudo-time step of 32 x 16 x 32 FP64 cells (66 us), 8 us of one
// of 128 x 64 x 128 FP32 cells (125 us).
template <int NTHREADS>
__device__ void reduce_min_at(double dtmin, const Reduce& red, double* scratch /* >= NTHREADS/32 doubles */,
                              int bid, int nblocks) {
  constexpr int NW = NTHREADS / 32;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  __shared__ unsigned int s_last;
  __syncthreads();  // scratch may alias buffers still in use
  if (lane == 0) scratch[warp] = dtmin;
  __syncthreads();
  if (threadIdx.x == 0) {
    double a = scratch[0];
    for (int w = 1; w < NW; ++w) a = min_positive(a, scratch[w]);
    red.partials[bid] = a;
    __threadfence();
    s_last = atomicAdd(red.counter, 1u) == (unsigned)(nblocks - 1);
  }
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  double a = INFINITY;
  for (int b = threadIdx.x; b < nblocks; b += NTHREADS) a = min_positive(a, __ldcg(red.partials + b));
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) a = min_positive(a, __shfl_xor_sync(0xffffffffu, a, off));
  if (lane == 0) scratch[warp] = a;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < NW; ++w) a = min_positive(a, scratch[w]);
    red.dt_out[0] = a;
    if (red.dt_user) red.dt_user[0] = a;
    *red.counter = 0u;
  }
}

// sums and minimum from per-thread values, for the block id and count of the launch grid
template <int NTHREADS>
__device__ __forceinline__ void reduce_and_finalize(double (&sum)[NV], double dtmin, const Reduce& red,
                                                    double* scratch) {
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
#pragma unroll
    for (int v = 0; v < NV; ++v) sum[v] += __shfl_xor_sync(0xffffffffu, sum[v], off);
    dtmin = min_positive(dtmin, __shfl_xor_sync(0xffffffffu, dtmin, off));
  }
  reduce_and_finalize_at<NTHREADS>(sum, dtmin, red, scratch, blockIdx.y * gridDim.x + blockIdx.x,
                                   gridDim.x * gridDim.y);
}

// ---------------------------------------------------------------------------
// reference kernel: one thread per cell
// ---------------------------------------------------------------------------
template <class T>
__device__ __forceinline__ void load_recover(const T* __restrict__ U, int64_t N, int64_t cell,
                                             const Phys<T>& ph, T (&w)[NV]) {
  T u[NV];
#pragma unroll
  for (int v = 0; v < NV; ++v) u[v] = __ldg(U + v * N + cell);
  recover(u, ph, w);
}

template <class T>
__device__ void cell_prim(const Shape& sh, const Geo<T>& g, const Phys<T>& ph,
                          const double* __restrict__ Br, const T* __restrict__ U, int k, int j,
                          int i, T (&w)[NV]) {
  map_column(j, i, sh.nt, sh.np);
  const int64_t col = (int64_t)j * sh.np + i;
  const int64_t plane = (int64_t)sh.nt * sh.np;
  if (k < 0) {
    T wi[NV];
    load_recover(U, sh.ncell, col, ph, wi);
    const int64_t cs = (int64_t)sh.nt * sh.np;
    inner_ghost_at(wi, Br, col, cs, (double)g.rhat[col], (double)g.rhat[cs + col],
                   (double)g.rhat[2 * cs + col], ph, w);
  } else if (k >= sh.nr) {
    T wi[NV];
    load_recover(U, sh.ncell, (int64_t)(sh.nr - 1) * plane + col, ph, wi);
    const int64_t cs = (int64_t)sh.nt * sh.np;
    outer_ghost(wi, g.rhat[col], g.rhat[cs + col], g.rhat[2 * cs + col], ph, w);
  } else {
    load_recover(U, sh.ncell, (int64_t)k * plane + col, ph, w);
  }
}

// face states from a 4-cell stencil ll, l | r, rr; slopes in units per
// distance (im, ip: inverse centre distances of the two cells' neighbours;
// hl: centre-to-face offset of l, hr: of r)
template <int LIM, class T>
__device__ __forceinline__ void face_states(const T (&ll)[NV], const T (&l)[NV], const T (&r)[NV],
                                            const T (&rr)[NV], T im_l, T ip_l, T hl, T im_r,
                                            T ip_r, T hr, T eps, T (&wl)[NV], T (&wr)[NV]) {
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    const T d = r[v] - l[v];
    const T sl = limited_slope<LIM>((l[v] - ll[v]) * im_l, d * ip_l, eps);
    const T sr = limited_slope<LIM>(d * im_r, (rr[v] - r[v]) * ip_r, eps);
    wl[v] = l[v] + sl * hl;
    wr[v] = r[v] - sr * hr;
  }
}

template <class T, int LIM>
__global__ void __launch_bounds__(256)
residual_cellwise(Shape sh, Geo<T> g, Phys<T> ph, const double* __restrict__ Br,
                  const T* __restrict__ U, T* __restrict__ R, Reduce red) {
  __shared__ double scratch[8 * RED_STRIDE];
  const int64_t cell = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  double sq[NV];
#pragma unroll
  for (int v = 0; v < NV; ++v) sq[v] = 0.0;
  double dtmin = INFINITY;
  if (cell < sh.ncell) {
    const int i = (int)(cell % sh.np);
    const int j = (int)((cell / sh.np) % sh.nt);
    const int k = (int)(cell / ((int64_t)sh.np * sh.nt));
    const int64_t cs = (int64_t)sh.nt * sh.np;
    const int64_t col = (int64_t)j * sh.np + i;
    T acc[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) acc[v] = (T)0;
    T lam_sum = (T)0;
    T wc[NV];
    cell_prim(sh, g, ph, Br, U, k, j, i, wc);
    const T one = (T)1, half = (T)0.5;
    // ---- r faces: lower (k - 1/2) and upper (k + 1/2)
    for (int side = 0; side < 2; ++side) {
      const int kl = side == 0 ? k - 1 : k;  // lower cell of the face
      T wl[NV], wr[NV];
      if (kl < 0 || kl >= sh.nr - 1) {  // boundary face: first order
        T a[NV], b[NV];
        cell_prim(sh, g, ph, Br, U, kl, j, i, a);
        cell_prim(sh, g, ph, Br, U, kl + 1, j, i, b);
#pragma unroll
        for (int v = 0; v < NV; ++v) { wl[v] = a[v]; wr[v] = b[v]; }
      } else {
        T a[NV], b[NV], c[NV], d[NV];
        cell_prim(sh, g, ph, Br, U, kl - 1, j, i, a);
        cell_prim(sh, g, ph, Br, U, kl, j, i, b);
        cell_prim(sh, g, ph, Br, U, kl + 1, j, i, c);
        cell_prim(sh, g, ph, Br, U, kl + 2, j, i, d);
        face_states<LIM>(a, b, c, d, g.inv_dm[kl], g.inv_dp[kl], g.hp[kl], g.inv_dm[kl + 1],
                         g.inv_dp[kl + 1], g.hm[kl + 1], ph.eps, wl, wr);
      }
      const T area = g.ra[kl + 1] * g.ar[j];
      T f[NV], la;
      rusanov(wl, wr, g.nr[col], g.nr[cs + col], g.nr[2 * cs + col], area, ph, f, la);
      const T sgn = side == 0 ? one : -one;
#pragma unroll
      for (int v = 0; v < NV; ++v) acc[v] += sgn * f[v];
      lam_sum += la;
    }
    // ---- theta faces
    const int64_t ts = (int64_t)(sh.nt + 1) * sh.np;
    for (int side = 0; side < 2; ++side) {
      const int jf = side == 0 ? j : j + 1;  // face index
      if (jf == 0 || jf == sh.nt) continue;  // pole faces have zero area
      T a[NV], b[NV], c[NV], d[NV], wl[NV], wr[NV];
      cell_prim(sh, g, ph, Br, U, k, jf - 2, i, a);
      cell_prim(sh, g, ph, Br, U, k, jf - 1, i, b);
      cell_prim(sh, g, ph, Br, U, k, jf, i, c);
      cell_prim(sh, g, ph, Br, U, k, jf + 1, i, d);
      face_states<LIM>(a, b, c, d, one, one, half, one, one, half, ph.eps, wl, wr);
      const int64_t fc = (int64_t)jf * sh.np + i;
      const T area = g.rb[k] * g.at[jf];
      T f[NV], la;
      rusanov(wl, wr, g.nth[fc], g.nth[ts + fc], g.nth[2 * ts + fc], area, ph, f, la);
      const T sgn = side == 0 ? one : -one;
#pragma unroll
      for (int v = 0; v < NV; ++v) acc[v] += sgn * f[v];
      lam_sum += la;
    }
    // ---- phi faces (periodic)
    for (int side = 0; side < 2; ++side) {
      const int ifc = side == 0 ? i : i + 1;
      T a[NV], b[NV], c[NV], d[NV], wl[NV], wr[NV];
      cell_prim(sh, g, ph, Br, U, k, j, ifc - 2, a);
      cell_prim(sh, g, ph, Br, U, k, j, ifc - 1, b);
      cell_prim(sh, g, ph, Br, U, k, j, ifc, c);
      cell_prim(sh, g, ph, Br, U, k, j, ifc + 1, d);
      face_states<LIM>(a, b, c, d, one, one, half, one, one, half, ph.eps, wl, wr);
      const int iw = ifc % sh.np;
      const T area = g.rb[k] * g.dtheta;
      T f[NV], la;
      rusanov(wl, wr, g.nph[iw], g.nph[sh.np + iw], (T)0, area, ph, f, la);
      const T sgn = side == 0 ? one : -one;
#pragma unroll
      for (int v = 0; v < NV; ++v) acc[v] += sgn * f[v];
      lam_sum += la;
    }
    // ---- divide by the volume, gravity source [Sect. 2.2], GLM damping
    const T vol = g.rv[k] * g.av[j];
    const T ivol = one / vol;
    T r[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) r[v] = acc[v] * ivol;
    const T gk = -g.grav[k];
    const T gx = gk * g.rhat[col], gy = gk * g.rhat[cs + col], gz = gk * g.rhat[2 * cs + col];
    const T rho = wc[0];
    r[1] += rho * gx;
    r[2] += rho * gy;
    r[3] += rho * gz;
    r[7] += rho * (wc[1] * gx + wc[2] * gy + wc[3] * gz);
    r[8] -= ph.psi_damp * wc[8];
    double chk = 0.0;
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      R[v * sh.ncell + cell] = r[v];
      sq[v] = (double)r[v] * (double)r[v];
      chk += sq[v];
    }
    dtmin = (double)vol / (double)lam_sum;
    if (!(wc[0] > (T)0) || !(wc[7] > (T)0) || !(chk <= 1.7e308)) flag_bad(red, cell);
  }
  reduce_and_finalize<256>(sq, dtmin, red, scratch);
}

// ---------------------------------------------------------------------------
// boundary electric field diagnostic: E = -V_b x B_b of the face-mean state at
// every inner face, in FP64 [Sect. 2.2 E = -V x B; Sect. 3.2]
// ---------------------------------------------------------------------------
template <class T>
__global__ void __launch_bounds__(128)
boundary_efield_kernel(Shape sh, Geo<T> g, Phys<T> ph, const double* __restrict__ Br,
                       const T* __restrict__ U, double* __restrict__ E) {
  const int64_t cs = (int64_t)sh.nt * sh.np;
  const int64_t col = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (col >= cs) return;
  T wi[NV], wg[NV];
  load_recover(U, sh.ncell, col, ph, wi);
  inner_ghost_at(wi, Br, col, cs, (double)g.rhat[col], (double)g.rhat[cs + col],
                 (double)g.rhat[2 * cs + col], ph, wg);
  double v[3], b[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    v[c] = 0.5 * ((double)wg[1 + c] + (double)wi[1 + c]);
    b[c] = 0.5 * ((double)wg[4 + c] + (double)wi[4 + c]);
  }
  E[col] = -(v[1] * b[2] - v[2] * b[1]);
  E[cs + col] = -(v[2] * b[0] - v[0] * b[2]);
  E[2 * cs + col] = -(v[0] * b[1] - v[1] * b[0]);
}

// cell-centred E = -V x B = -(m x B) / rho of every cell in FP64 (the volume
// field of Sect. 3.1); E[3][ncell], one cell per thread, grid-stride.
template <class T>
__global__ void __launch_bounds__(256)
cell_efield_kernel(int64_t ncell, const T* __restrict__ U, double* __restrict__ E) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; c < ncell; c += stride) {
    const double rho = (double)U[c];
    const double m0 = (double)U[ncell + c], m1 = (double)U[2 * ncell + c], m2 = (double)U[3 * ncell + c];
    const double b0 = (double)U[4 * ncell + c], b1 = (double)U[5 * ncell + c], b2 = (double)U[6 * ncell + c];
    const double v0 = m0 / rho, v1 = m1 / rho, v2 = m2 / rho;
    E[c] = -(v1 * b2 - v2 * b1);
    E[ncell + c] = -(v2 * b0 - v0 * b2);
    E[2 * ncell + c] = -(v0 * b1 - v1 * b0);
  }
}

// whether the squares of a cell's residuals and their sum are finite
__device__ __forceinline__ bool squares_finite(const float (&r)[NV]) {
  float s = 0.f;
#pragma unroll
  for (int v = 0; v < NV; ++v) s = fmaf(r[v], r[v], s);
  return fabsf(s) < INFINITY;
}
// FP64: on the integer pipe, |r| < 2^511 from the exponents
__device__ __forceinline__ bool squares_finite(const double (&r)[NV]) {
  int m = 0;
#pragma unroll
  for (int v = 0; v < NV; ++v) m = max(m, __double2hiint(r[v]) & 0x7fffffff);
  return m < 0x5fe00000;
}

// ---------------------------------------------------------------------------
// production kernel: radial marching over a (theta, phi) tile
// ---------------------------------------------------------------------------
// Thread (jj, ii) owns column (j0 + jj, i0 + ii) of the tile and keeps the
// primitives of planes k and k + 1 of it in registers; shared memory holds the
// halo'd plane k.  Two phases per plane, a barrier after each:
//   1  gather the six faces of the cell of plane k - 1 into R; the theta and
//      phi slopes of plane k: the cell's lower face values stay in registers,
//      its upper ones go to the face above it; the halo cells' slopes are
//      spread over all threads, three variables of one cell each
//   2  the cell's lower theta and phi face (Rusanov + GLM) into shared
//      memory; the faces past the tile's last row and column on its last
//      warps; the r slope of plane k + 1 and the r face k + 1/2 in registers;
//      plane k + 1 replaces plane k in shared memory; the loads of the own
//      cell of plane k + 3 and the halo of plane k + 2 are issued
//
// FP32 is bound by instruction issue at 16 warps per SM (128 registers): 66 %
// of the slots at 1545 instructions per cell.  128 x 64 x 128, R alone: 64 us
// (90 us with three phases per plane, a ring of three planes, both face values
// in shared memory, a global load per radial factor and the sums always; 72 us
// with the halo items worked out from their number on every plane).  FP64 is
// bound by the FP64 pipe (88 % busy): about 790 operations per cell, 1.53 ms
// (2.65 ms with 1208).
template <int TT, int TP>
struct TileDims {
  static constexpr int NT = TT * TP;                            // threads = own columns
  static constexpr int HT = TT + 4, HP = TP + 4, HC = HT * HP;  // halo'd plane
  static constexpr int NHALO = 4 * (TT + TP);                   // halo positions (a cross: no corners)
  static constexpr int NTV = (TT + 1) * TP;                     // theta faces (rows 0..TT)
  static constexpr int NPV = TT * (TP + 1);                     // phi faces (cols 0..TP)
  static constexpr int NFA = NTV + NPV;                         // both, theta faces first
  static constexpr int NF = NV + 1;                             // 9 fluxes + lambda |S|
  static constexpr int NEXTRA_V = 2 * (TT + TP);                // halo cells needing a face value
  static constexpr int NEXTRA_F = TT + TP;                      // faces beyond the own lower faces
  static constexpr int NUV = NFA + NEXTRA_F;                    // L states, then the R states of those faces
  static constexpr int NITEM = (3 * NEXTRA_V + 1) & ~1;         // items of three variables of one halo cell
  // item x -> what it does, packed: source offset in the halo'd planes, target
  // offset in the face states, theta neighbours (else phi), upper value (else lower)
  __device__ static unsigned item(int x) {
    const int e = x % NEXTRA_V, v0 = 3 * (x / NEXTRA_V);
    int h, dst;
    unsigned flags;
    if (e < TP) {                  // theta row -1: upper value -> face row 0
      h = HP + e + 2; dst = e; flags = 3u;
    } else if (e < TP + TT) {      // phi col -1 of row r: upper value -> face col 0
      const int r = e - TP;
      h = (r + 2) * HP + 1; dst = NTV + r * (TP + 1); flags = 2u;
    } else if (e < 2 * TP + TT) {  // theta row TT: lower value, R state of face row TT
      const int c = e - TP - TT;
      h = (TT + 2) * HP + c + 2; dst = NFA + c; flags = 1u;
    } else {                       // phi col TP of row r: lower value, R state of face col TP
      const int r = e - 2 * TP - TT;
      h = (r + 2) * HP + TP + 2; dst = NFA + TP + r; flags = 0u;
    }
    return (unsigned)(h + v0 * HC) | ((unsigned)(dst + v0 * NUV) << 15) | (flags << 30);
  }
  // per-CTA geometry staged once: theta-face normals, phi-face normals, own
  // r-face normals, own radial unit vectors, theta factors of the areas/volumes
  static constexpr int NGEO = 3 * NTV + 2 * (TP + 1) + 6 * NT + (TT + 1) + 2 * TT;
  static constexpr int NRAD = 8;                                // radial factors of a plane, three planes held
  static constexpr int NROW = 6 * (TT + 1);                     // factors of the tile's rows in one plane (1 / V: two)
  template <class T>
  static constexpr size_t smem_bytes() {
    return sizeof(unsigned) * (size_t)NITEM +
           sizeof(T) * ((size_t)NV * HC + (size_t)NV * NUV + (size_t)NF * NFA +
                        (size_t)NV * NHALO + (size_t)3 * NRAD + (size_t)NROW + (size_t)NGEO);
  }
  // halo position h in [0, NHALO) -> halo'd (row, col)
  __device__ static void halo_rc(int h, int& row, int& col) {
    if (h < 4 * TP) { const int r = h / TP; row = r < 2 ? r : TT + r; col = 2 + h % TP; }
    else { h -= 4 * TP; row = 2 + h / 4; const int c = h % 4; col = c < 2 ? c : TP + c; }
  }
};

template <class T>
__device__ __forceinline__ void load_raw(const T* __restrict__ src, int64_t N, int64_t c, T (&u)[NV]) {
#pragma unroll
  for (int v = 0; v < NV; ++v) u[v] = __ldg(src + v * N + c);
}

// asynchronous copy of one element from global to shared memory, the wait for
// all of the thread's copies
template <class T>
__device__ __forceinline__ void copy_async(T* dst, const T* src) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  if constexpr (sizeof(T) == 4)
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(d), "l"(src) : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void copy_async_wait() {
  asm volatile("cp.async.wait_all;" ::: "memory");
}

// resident CTAs per SM the register allocation is sized for: 16 FP32 warps;
// 8 FP64 warps (the FP64 pipe needs no more, and their state is twice as wide)
template <class T, int NT> struct MinCtas { static constexpr int value = (sizeof(T) == 4 ? 512 : 256) / NT; };

// One work item of the tiled residual: tile `tile` (row-major over the
// (theta, phi) tiles) and radial chunk `chunk` of one grid; `bid` / `nblocks`
// number the items of that grid for its cross-CTA reduction.  The grid's
// description is read where it lies (kernel parameters, or the ensemble's copy
// in shared memory) at each use.  What else is wanted is a
// template switch (the running sums are registers the FP32 kernel has to spill
// for): SUMS_NONE, R alone; SUMS_DT, the step bound; SUMS_ALL, the norms too.
template <class T, int LIM, int TT, int TP, int SUMS>
__device__ __forceinline__ void tiled_item(const Shape& sh, const Geo<T>& g, const Phys<T>& ph,
                                           const double* const& Br, const T* const& U,
                                           T* const& R, const Reduce& red, int kchunk, int tile,
                                           int chunk, int bid, int nblocks, unsigned char* smem_raw) {
  using D = TileDims<TT, TP>;
  constexpr int NT = D::NT, HP = D::HP, HC = D::HC, NTV = D::NTV, NFA = D::NFA, NUV = D::NUV, NF = D::NF;
  constexpr int NX = D::NEXTRA_V, NXF = D::NEXTRA_F;
  static_assert(D::NRAD <= D::NHALO, "the halo threads wait for the radial factors too");
  static_assert(D::NHALO <= NT, "each thread stores at most one halo position");
  static_assert(NXF <= NT && NT % 32 == 0 && NV * HC < (1 << 15) && NV * D::NUV < (1 << 15), "tile shape");
  T* sp = reinterpret_cast<T*>(smem_raw);    // [NV][HC]   primitives of plane k
  T* uv = sp + NV * HC;                      // [NV][NUV]  L state of each face (upper value of the cell below),
                                             //   then the R states of the faces past the last row / column
  T* fx = uv + NV * NUV;                     // [NF][NFA]  flux x area of each face, lambda x area last
  T* hr = fx + NF * NFA;                     // [NV][NHALO] raw halo cells of plane k + 1
  T* s_rad = hr + NV * D::NHALO;             // [3][NRAD] radial factors of planes k .. k + 2
  T* s_row = s_rad + 3 * D::NRAD;            // [6][TT + 1] by row: r and theta face areas, V, gravity x V of plane k,
                                             //   1 / V of planes k and k - 1
  T* s_nth = s_row + D::NROW;                // [3][NTV]
  T* s_nph = s_nth + 3 * NTV;                // [2][TP + 1]
  T* s_nr = s_nph + 2 * (TP + 1);            // [3][NT]
  T* s_rh = s_nr + 3 * NT;                   // [3][NT]
  T* s_at = s_rh + 3 * NT;                   // [TT + 1]
  T* s_ar = s_at + (TT + 1);                 // [TT]
  T* s_av = s_ar + TT;                       // [TT]
  unsigned* s_item = reinterpret_cast<unsigned*>(s_av + TT);  // [NITEM]

  const int nr = sh.nr, nt = sh.nt, np = sh.np;
  const int64_t N = sh.ncell, cs = (int64_t)nt * np;
  const int tid = threadIdx.x;
  const int ntp = (np + TP - 1) / TP;
  const int j0 = (tile / ntp) * TT, i0 = (tile % ntp) * TP;
  const int k0 = chunk * kchunk;
  const int k1 = min(nr, k0 + kchunk);
  const int jj = tid / TP, ii = tid % TP;
  const int jo = j0 + jj, io = i0 + ii;
  const bool own = jo < nt && io < np;
  const int hown = (jj + 2) * HP + (ii + 2);
  // global column of the own position and of this thread's halo position
  int c_own, c_halo = 0;
  int h_halo = -1;
  {
    int j = jo, i = io;
    map_column(j, i, nt, np);
    c_own = j * np + i;
    if (tid < D::NHALO) {
      int row, col;
      D::halo_rc(tid, row, col);
      h_halo = row * HP + col;
      int jh = j0 - 2 + row, ih = i0 - 2 + col;
      map_column(jh, ih, nt, np);
      c_halo = jh * np + ih;
    }
  }
  const int ocol = own ? c_own : 0;
  const T one = (T)1, half = (T)0.5;

  // ---------------- preamble: every load of the chunk's first planes at once
  T wc[NV], w1[NV];   // primitives of planes k and k + 1 of the own column
  T rL[NV];           // L state of r face k + 1/2 (upper r value of plane k)
  T frl[NF];          // flux x area of r face k - 1/2, lambda x area last
  T pf_own[NV];       // raw own cell of plane k + 2
  // FP64: the forward difference of plane k, which is the backward one of plane
  // k + 1 (the same two cells over the same distance).  FP32 forms it again: its
  // registers are full.
  constexpr bool CARRY = sizeof(T) == 8;
  T fwd[CARRY ? NV : 1];
  // radial factor tid of plane p: r_b, r_v and gravity of p, face area factor of
  // its upper face, slope and face distances of plane p + 1.  They come in with
  // the halo cells, two planes ahead: a global load where they are used would
  // stall every warp just after a barrier.
  const T* rad_src = nullptr;
  if (tid < D::NRAD) {
    const T* const src[D::NRAD] = {g.rb, g.rv, g.grav, g.ra + 1, g.inv_dm, g.inv_dp, g.hm, g.hp};
#pragma unroll
    for (int q = 0; q < D::NRAD; ++q) rad_src = tid == q ? src[q] : rad_src;
  }
  auto rad_at = [&](int p) -> const T* { return rad_src + (tid < 4 ? p : min(p + 1, nr - 1)); };
  auto rad_slot = [&](int p) -> T* { return s_rad + (p % 3) * D::NRAD; };
  // the halo cell of plane p into its slot of hr, read back by the same thread:
  // held in registers its nine values would spill
  auto fetch_halo = [&](int p) {
    const T* src = U + (int64_t)p * cs + c_halo;
#pragma unroll
    for (int v = 0; v < NV; ++v) copy_async(hr + v * D::NHALO + tid, src + v * N);
  };
  {
    T um1[NV], um2[NV], u0[NV], u1[NV], uh[NV];
    load_raw(U + (int64_t)k0 * cs, N, c_own, u0);
    if (h_halo >= 0) load_raw(U + (int64_t)k0 * cs, N, c_halo, uh);
    if (h_halo >= 0 && k0 + 1 < k1) fetch_halo(k0 + 1);
    if (k0 + 1 < nr) load_raw(U + (int64_t)(k0 + 1) * cs, N, c_own, u1);
    if (k0 >= 1) load_raw(U + (int64_t)(k0 - 1) * cs, N, c_own, um1);
    if (k0 >= 2) load_raw(U + (int64_t)(k0 - 2) * cs, N, c_own, um2);
    if (k0 + 2 < nr) load_raw(U + (int64_t)(k0 + 2) * cs, N, c_own, pf_own);
    {
      const int64_t ts = (int64_t)(nt + 1) * np;
      for (int q = tid; q < NTV; q += NT) {
        const int f = q / TP, col = q % TP;
        const int jf = min(j0 + f, nt), ic = min(i0 + col, np - 1);
        const int64_t fc = (int64_t)jf * np + ic;
        s_nth[q] = g.nth[fc];
        s_nth[NTV + q] = g.nth[ts + fc];
        s_nth[2 * NTV + q] = g.nth[2 * ts + fc];
      }
      for (int q = tid; q <= TP; q += NT) {
        int ic = i0 + q;
        ic = ic >= np ? ic - np : ic;
        s_nph[q] = g.nph[ic];
        s_nph[TP + 1 + q] = g.nph[np + ic];
      }
      s_nr[tid] = g.nr[ocol];
      s_nr[NT + tid] = g.nr[cs + ocol];
      s_nr[2 * NT + tid] = g.nr[2 * cs + ocol];
      s_rh[tid] = g.rhat[c_own];
      s_rh[NT + tid] = g.rhat[cs + c_own];
      s_rh[2 * NT + tid] = g.rhat[2 * cs + c_own];
      if (tid < D::NRAD) {
        rad_slot(k0)[tid] = *rad_at(k0);
        if (k0 + 1 < k1) rad_slot(k0 + 1)[tid] = *rad_at(k0 + 1);
      }
      for (int x = tid; x < 3 * NX; x += NT) s_item[x] = D::item(x);
      if (tid <= TT) s_at[tid] = g.at[min(j0 + tid, nt)];
      if (tid < TT) {
        s_ar[tid] = g.ar[min(j0 + tid, nt - 1)];
        s_av[tid] = g.av[min(j0 + tid, nt - 1)];
      }
    }
    recover(u0, ph, wc);
#pragma unroll
    for (int v = 0; v < NV; ++v) sp[v * HC + hown] = wc[v];
    if (h_halo >= 0) {
      T w[NV];
      recover(uh, ph, w);
#pragma unroll
      for (int v = 0; v < NV; ++v) sp[v * HC + h_halo] = w[v];
    }
    __syncthreads();
    if (k0 + 1 < nr)
      recover(u1, ph, w1);
    else
      outer_ghost(wc, s_rh[tid], s_rh[NT + tid], s_rh[2 * NT + tid], ph, w1);
    T wm1[NV], wm2[NV];
    if (k0 >= 1) {
      recover(um1, ph, wm1);
    } else {  // inner ghost for plane -1
      inner_ghost_at(wc, Br, c_own, cs, (double)g.rhat[c_own], (double)g.rhat[cs + c_own],
                     (double)g.rhat[2 * cs + c_own], ph, wm1);
    }
    if (k0 >= 2) {
      recover(um2, ph, wm2);
    } else if (k0 == 1) {
      inner_ghost_at(wm1, Br, c_own, cs, (double)g.rhat[c_own], (double)g.rhat[cs + c_own],
                     (double)g.rhat[2 * cs + c_own], ph, wm2);
    }
    // r face k0 - 1/2
    T wl[NV], wr[NV];
    {
      const T im = g.inv_dm[k0], ip = g.inv_dp[k0], hm = g.hm[k0], hp = g.hp[k0];
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        const T s = limited_slope<LIM>(product(wc[v] - wm1[v], im), product(w1[v] - wc[v], ip), ph.eps);
        if constexpr (CARRY) fwd[v] = product(w1[v] - wc[v], ip);
        wr[v] = fmat(-s, hm, wc[v]);
        rL[v] = fmat(s, hp, wc[v]);
      }
    }
    if (k0 == 0) {
#pragma unroll
      for (int v = 0; v < NV; ++v) { wl[v] = wm1[v]; wr[v] = wc[v]; }  // boundary: first order
    } else {
      const T im = g.inv_dm[k0 - 1], ip = g.inv_dp[k0 - 1], hp = g.hp[k0 - 1];
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        const T s = limited_slope<LIM>(product(wm1[v] - wm2[v], im), product(wc[v] - wm1[v], ip), ph.eps);
        wl[v] = fmat(s, hp, wm1[v]);
      }
    }
    if (own) {
      T f[NV], la;
      rusanov<true>(wl, wr, s_nr[tid], s_nr[NT + tid], s_nr[2 * NT + tid], g.ra[k0] * s_ar[jj], ph, f, la);
#pragma unroll
      for (int v = 0; v < NV; ++v) frl[v] = f[v];
      frl[NV] = la;
    } else {
#pragma unroll
      for (int v = 0; v < NF; ++v) frl[v] = (T)0;
    }
  }

  T sq[NV];
#pragma unroll
  for (int v = 0; v < NV; ++v) sq[v] = (T)0;
  // the thread's step bound: FP64 as the largest lambda |S| / V, whose reciprocal is
  // taken once (a division in every cell is 10 operations of the FP64 pipe); FP32 as
  // the smallest V / (lambda |S|), a rounding of 1 / V less (8.3e-8 rms against 9.6e-8
  // over 60 shells)
  T rate = (T)0, bound = (T)INFINITY;
  T dr[NF];           // r faces' contribution to the cell being gathered
  // FP64: the plane's factors of each row once, by one thread per row: a product
  // or a reciprocal in every thread is an operation of the FP64 pipe per warp.
  // FP32 forms them in place (with the table the ensemble was 1 % slower).
  constexpr bool ROWS = sizeof(T) == 8;
  T* const row_ar = s_row, * const row_at = s_row + (TT + 1), * const row_v = s_row + 2 * (TT + 1);
  T* const row_gv = s_row + 3 * (TT + 1), * const row_iv = s_row + 4 * (TT + 1);
  bool bad = false;   // rho <= 0 or p <= 0 in that cell

  for (int k = k0;; ++k) {
    // ======== phase 1
    if (k > k0 && own) {  // the six faces and the sources of cell (k - 1, jo, io)
      const int kg = k - 1;
      const int tl = tid, tu = tid + TP;
      const int pl = NTV + jj * (TP + 1) + ii, pu = pl + 1;
      T r[NV];
#pragma unroll
      for (int v = 0; v < NV; ++v)
        r[v] = dr[v] + (fx[v * NFA + tl] - fx[v * NFA + tu]) + (fx[v * NFA + pl] - fx[v * NFA + pu]);
      const T vol = ROWS ? one : rad_slot(kg)[1] * s_av[jj];
      // (FP32: rounded as the including file's flags have it, approximate but in the static entry)
      const T ivol = ROWS ? row_iv[(kg & 1) * (TT + 1) + jj] : one / vol;
      if (SUMS != SUMS_NONE) {
        const T lam = dr[NV] + (fx[NV * NFA + tl] + fx[NV * NFA + tu]) + (fx[NV * NFA + pl] + fx[NV * NFA + pu]);
        if constexpr (ROWS) {
          const T x = lam * ivol;
          rate = greater(x, rate) ? x : rate;
        } else {
          const T x = vol / lam;
          bound = x < bound ? x : bound;
        }
      }
      T* dst = R + (int64_t)kg * cs + ocol;
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        r[v] *= ivol;
        dst[v * N] = r[v];
        if (SUMS == SUMS_ALL) sq[v] = fmat(r[v], r[v], sq[v]);
      }
      if (bad || !squares_finite(r)) flag_bad(red, (int64_t)kg * cs + ocol);
    }
    if (k >= k1) break;
    if (ROWS && tid >= NT - 32 && tid - (NT - 32) <= TT) {
      const int q = tid - (NT - 32);
      const T* rad = rad_slot(k);
      row_at[q] = rad[0] * s_at[q];
      if (q < TT) {
        const T vol = rad[1] * s_av[q];
        row_ar[q] = rad[3] * s_ar[q];
        row_v[q] = vol;
        row_gv[q] = -(rad[2] * vol);
        row_iv[(k & 1) * (TT + 1) + q] = frcp(vol);
      }
    }
    T tlo[NV], plo[NV];  // the cell's lower theta and phi face values
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      const T* q = sp + v * HC + hown;
      const T w = wc[v];
      const T st = limited_slope<LIM>(w - q[-HP], q[HP] - w, ph.eps);
      const T sf = limited_slope<LIM>(w - q[-1], q[1] - w, ph.eps);
      // explicit FMAs: the same rounding in every kernel inlining this
      tlo[v] = fmat(-half, st, w);
      uv[v * NUV + tid + TP] = fmat(half, st, w);
      plo[v] = fmat(-half, sf, w);
      uv[v * NUV + NTV + jj * (TP + 1) + ii + 1] = fmat(half, sf, w);
    }
    // halo cells whose face values the tile's boundary faces need: three
    // variables of one cell per item, the items packed once per CTA (worked out
    // from x on every plane they took 8 us of 72 in FP32 and 75 of 1670 in FP64)
    for (int x = tid; x < 3 * NX; x += NT) {
      const unsigned it = s_item[x];
      const int step = (it & (1u << 30)) ? HP : 1;
      const T sgn = (it & (1u << 31)) ? half : -half;
      const T* q = sp + (it & 0x7fffu);
      T* o = uv + ((it >> 15) & 0x7fffu);
#pragma unroll
      for (int v = 0; v < 3; ++v) {
        const T w = q[v * HC];
        const T s = limited_slope<LIM>(w - q[v * HC - step], q[v * HC + step] - w, ph.eps);
        o[v * NUV] = fmat(sgn, s, w);
      }
    }
    __syncthreads();
    // ======== phase 2
    const T* rad = rad_slot(k);
    const T rbk = rad[0];
    {  // lower theta face of the own cell; poles and ragged rows / columns carry nothing
      T fl[NV], la = (T)0;
      if (jo > 0 && jo < nt && io < np) {
        T wl[NV];
#pragma unroll
        for (int v = 0; v < NV; ++v) wl[v] = uv[v * NUV + tid];
        rusanov<true>(wl, tlo, s_nth[tid], s_nth[NTV + tid], s_nth[2 * NTV + tid], ROWS ? row_at[jj] : rbk * s_at[jj], ph, fl, la);
      } else {
#pragma unroll
        for (int v = 0; v < NV; ++v) fl[v] = (T)0;
      }
#pragma unroll
      for (int v = 0; v < NV; ++v) fx[v * NFA + tid] = fl[v];
      if (SUMS != SUMS_NONE) fx[NV * NFA + tid] = la;
    }
    {  // lower phi face of the own cell
      const int f = NTV + jj * (TP + 1) + ii;
      T fl[NV], la = (T)0;
      if (jo < nt && io <= np) {
        T wl[NV];
#pragma unroll
        for (int v = 0; v < NV; ++v) wl[v] = uv[v * NUV + f];
        rusanov<false>(wl, plo, s_nph[ii], s_nph[TP + 1 + ii], (T)0, rbk * g.dtheta, ph, fl, la);
      } else {
#pragma unroll
        for (int v = 0; v < NV; ++v) fl[v] = (T)0;
      }
#pragma unroll
      for (int v = 0; v < NV; ++v) fx[v * NFA + f] = fl[v];
      if (SUMS != SUMS_NONE) fx[NV * NFA + f] = la;
    }
    if (tid >= NT - ((NXF + 31) / 32) * 32) {  // the faces past the last row and column: the last warps
      const int e = tid - (NT - ((NXF + 31) / 32) * 32);
      if (e < NXF) {
        int f;
        T nx, ny, nz, area;
        bool live;
        if (e < TP) {
          f = TT * TP + e;
          live = j0 + TT < nt && i0 + e < np;
          nx = s_nth[f]; ny = s_nth[NTV + f]; nz = s_nth[2 * NTV + f];
          area = ROWS ? row_at[TT] : rbk * s_at[TT];
        } else {
          const int r = e - TP;
          f = NTV + r * (TP + 1) + TP;
          live = j0 + r < nt && i0 + TP <= np;
          nx = s_nph[TP]; ny = s_nph[2 * TP + 1]; nz = (T)0;
          area = rbk * g.dtheta;
        }
        T fl[NV], la = (T)0;
        if (live) {
          T wl[NV], wr[NV];
#pragma unroll
          for (int v = 0; v < NV; ++v) { wl[v] = uv[v * NUV + f]; wr[v] = uv[v * NUV + NFA + e]; }
          rusanov<true>(wl, wr, nx, ny, nz, area, ph, fl, la);
        } else {
#pragma unroll
          for (int v = 0; v < NV; ++v) fl[v] = (T)0;
        }
#pragma unroll
        for (int v = 0; v < NV; ++v) fx[v * NFA + f] = fl[v];
        if (SUMS != SUMS_NONE) fx[NV * NFA + f] = la;
      }
    }
    // r face k + 1/2 and the plane k + 1 that follows
    T w2[NV], rLn[NV];
    if (k + 2 < nr)
      recover(pf_own, ph, w2);
    else if (k + 2 == nr)
      outer_ghost(w1, s_rh[tid], s_rh[NT + tid], s_rh[2 * NT + tid], ph, w2);
    if (k + 3 < nr && k + 2 < k1 + 1) load_raw(U + (int64_t)(k + 3) * cs, N, c_own, pf_own);
    {
      T rR[NV];
      if (k + 1 < nr) {
        const T im = rad[4], ip = rad[5], hm = rad[6], hp = rad[7];
#pragma unroll
        for (int v = 0; v < NV; ++v) {
          T s;
          if constexpr (CARRY) {
            const T b = product(w2[v] - w1[v], ip);
            s = limited_slope<LIM>(fwd[v], b, ph.eps);
            fwd[v] = b;
          } else {
            s = limited_slope<LIM>(product(w1[v] - wc[v], im), product(w2[v] - w1[v], ip), ph.eps);
          }
          rR[v] = fmat(-s, hm, w1[v]);
          rLn[v] = fmat(s, hp, w1[v]);
        }
      } else {  // outer boundary face: first order, interior | ghost
#pragma unroll
        for (int v = 0; v < NV; ++v) { rL[v] = wc[v]; rR[v] = w1[v]; }
      }
      if (own) {
        T f[NV], la;
        rusanov<true>(rL, rR, s_nr[tid], s_nr[NT + tid], s_nr[2 * NT + tid], ROWS ? row_ar[jj] : rad[3] * s_ar[jj], ph, f, la);
#pragma unroll
        for (int v = 0; v < NV; ++v) { dr[v] = frl[v] - f[v]; frl[v] = f[v]; }
        dr[NV] = frl[NV] + la;
        frl[NV] = la;
        // the sources in flux units (x V): gravity [Sect. 2.2] and GLM damping
        const T vol = ROWS ? row_v[jj] : rad[1] * s_av[jj];
        const T a = (ROWS ? row_gv[jj] : -(rad[2] * vol)) * wc[0];
        const T ex = s_rh[tid], ey = s_rh[NT + tid], ez = s_rh[2 * NT + tid];
        dr[1] = fmat(a, ex, dr[1]);
        dr[2] = fmat(a, ey, dr[2]);
        dr[3] = fmat(a, ez, dr[3]);
        dr[7] = fmat(a, fmat(wc[1], ex, fmat(wc[2], ey, wc[3] * ez)), dr[7]);
        dr[8] = fmat(-(ph.psi_damp * vol), wc[8], dr[8]);
        bad = !positive(wc[0]) || !positive(wc[7]);
      }
    }
    if (k + 1 < k1) {
#pragma unroll
      for (int v = 0; v < NV; ++v) sp[v * HC + hown] = w1[v];
      if (h_halo >= 0) {
        T u[NV], w[NV];
        copy_async_wait();
#pragma unroll
        for (int v = 0; v < NV; ++v) u[v] = hr[v * D::NHALO + tid];
        recover(u, ph, w);
#pragma unroll
        for (int v = 0; v < NV; ++v) sp[v * HC + h_halo] = w[v];
        if (k + 2 < k1) {
          fetch_halo(k + 2);
          if (tid < D::NRAD) copy_async(rad_slot(k + 2) + tid, rad_at(k + 2));
        }
      }
    }
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      wc[v] = w1[v];
      w1[v] = w2[v];
      rL[v] = rLn[v];
    }
    __syncthreads();
  }
  // ---------------- reductions: warp tree in T, then FP64 across warps and CTAs
  if (SUMS == SUMS_NONE) return;
  T dtm = bound;
  if (ROWS && rate > (T)0) dtm = one / rate;
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
#pragma unroll
    for (int v = 0; v < NV; ++v)
      if (SUMS == SUMS_ALL) sq[v] += __shfl_xor_sync(0xffffffffu, sq[v], off);
    const T o = __shfl_xor_sync(0xffffffffu, dtm, off);
    dtm = greater(dtm, o) ? o : dtm;
  }
  double* const scratch = reinterpret_cast<double*>(smem_raw);
  if (SUMS == SUMS_ALL)
    reduce_and_finalize_at<NT>(sq, dtm, red, scratch, bid, nblocks);
  else
    reduce_min_at<NT>((double)dtm, red, scratch, bid, nblocks);
}

// one grid: block (x, y) = (tile, radial chunk); with a second state, block z
// picks the state
template <class T, int LIM, int TT, int TP, int SUMS>
__global__ void __launch_bounds__(TT * TP, (MinCtas<T, TT * TP>::value))
residual_tiled(Shape sh, Geo<T> g, Phys<T> ph, const double* __restrict__ Br,
               const T* __restrict__ U, T* __restrict__ R, Reduce red, int kchunk, const T* __restrict__ U2,
               T* __restrict__ R2) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const double* br = Br;
  const T* u = blockIdx.z == 0 ? U : U2;
  T* r = blockIdx.z == 0 ? R : R2;
  tiled_item<T, LIM, TT, TP, SUMS>(sh, g, ph, br, u, r, red, kchunk, blockIdx.x, blockIdx.y,
                             blockIdx.y * gridDim.x + blockIdx.x, gridDim.x * gridDim.y, smem_raw);
}

// ---------------------------------------------------------------------------
// ensemble: many grids (same precision and limiter, any sizes) in one
// persistent launch.  Work items are (member, tile, radial chunk), numbered
// member by member; CTAs take items from a global counter (zeroed before the
// launch) until none are left.  Each member keeps its own reduction scratch,
// so its norms and dtmin come out exactly as from its own launch with the
// same radial chunk.  The kernel is instantiated per (theta, phi) tile shape;
// members with another shape go to that shape's launch.
// ---------------------------------------------------------------------------

template <class T>
struct EnsMember {
  Shape sh;
  Geo<T> g;
  Phys<T> ph;
  const double* Br;
  const T* U;
  T* R;
  Reduce red;
  int kchunk, ntiles, nitems, item0, tile;
};


template <class T, int LIM, int TT, int TP, int SUMS>
__global__ void __launch_bounds__(TT * TP, (MinCtas<T, TT * TP>::value))
residual_ensemble(const EnsMember<T>* __restrict__ mem, int nmem, int nitems, unsigned int* __restrict__ next) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ EnsMember<T> M;  // the item's member: its fields are read where they are used, not held in registers
  __shared__ int s_item, s_mem;
  static_assert(sizeof(EnsMember<T>) % 8 == 0, "copied as 64-bit words");
  if (threadIdx.x == 0) s_mem = -1;
  for (;;) {
    if (threadIdx.x == 0) s_item = (int)atomicAdd(next, 1u);
    __syncthreads();
    const int item = s_item;
    if (item >= nitems) break;
    int m = 0;
    while (m + 1 < nmem && mem[m + 1].item0 <= item) ++m;
    if (m != s_mem) {
      const unsigned long long* src = reinterpret_cast<const unsigned long long*>(mem + m);
      unsigned long long* dst = reinterpret_cast<unsigned long long*>(&M);
      for (int q = threadIdx.x; q < (int)(sizeof(EnsMember<T>) / 8); q += TT * TP) dst[q] = src[q];
      __syncthreads();
      if (threadIdx.x == 0) s_mem = m;
    }
    const int local = item - M.item0;
    tiled_item<T, LIM, TT, TP, SUMS>(M.sh, M.g, M.ph, M.Br, M.U, M.R, M.red, M.kchunk, local % M.ntiles,
                               local / M.ntiles, local, M.nitems, smem_raw);
    __syncthreads();  // shared memory and s_item are reused by the next item
  }
}

}  // namespace crn
