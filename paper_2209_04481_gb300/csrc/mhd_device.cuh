// mhd_device.cuh -- device arithmetic of the MHD + GLM residual (sm_103a).
//
// Per-cell and per-face building blocks shared by the residual kernels:
// primitive recovery, the inner "low-E" and outer ghost states, the slope
// limiters, and the Rusanov + GLM face flux.  Templated on the arithmetic type
// T (double: the plain FP64 path; float: the FP32-bulk path).
//
// Paper: arXiv 2209.04481.  Equations of ideal MHD with gravity (Sect. 2.2) in
// Alfven-speed units; second-order FV with hyperbolic divergence cleaning
// (Sect. 2.1, cleaning speed c_h of Sect. 3.3); inner boundary of Sect. 3.2;
// outer boundary laws of Sect. 4.1 / Table 2.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace crn {

// state indices: conservative (rho, mx, my, mz, bx, by, bz, E, psi) and
// primitive (rho, vx, vy, vz, bx, by, bz, p, psi) share positions 0, 4-6, 8.
constexpr int NV = 9;
// doubles per CTA in the reduction-partials array
constexpr int RED_STRIDE = 16;

// Geometry as 1D radial factors x per-column angular factors (all exact
// integrals of the shell, computed on the host in FP64):
//   |S_r(k face)|     = ra[k] * ar[j]          (ra = r^2)
//   |S_theta(j face)| = rb[k] * at[j face]     (rb = (r2^2 - r1^2) / 2)
//   |S_phi|           = rb[k] * dtheta
//   V(k, j)           = rv[k] * av[j]          (rv = (r2^3 - r1^3) / 3)
// Unit normals depend on (j, i) only.
template <class T>
struct Geo {
  const T* ra;      // [nr + 1]
  const T* rb;      // [nr]
  const T* rv;      // [nr]
  const T* inv_dm;  // [nr] 1 / (r_c(k) - r_c(k-1)), ghost centres mirrored
  const T* inv_dp;  // [nr] 1 / (r_c(k+1) - r_c(k))
  const T* hm;      // [nr] r_c(k) - r_f(k)
  const T* hp;      // [nr] r_f(k+1) - r_c(k)
  const T* grav;    // [nr] g0 / r_c(k)^2
  const T* ar;      // [nt]
  const T* at;      // [nt + 1] (0 at the poles)
  const T* av;      // [nt]
  const T* nr;      // [3][nt][np]      r-face unit normal
  const T* nth;     // [3][nt + 1][np]  theta-face unit normal
  const T* nph;     // [2][np]          phi-face unit normal (x, y; z = 0)
  const T* rhat;    // [3][nt][np]      radial unit vector at (theta_c, phi_c)
  T dtheta;
};

template <class T>
struct Phys {
  T gamma, gm1, igm1, ch, ch2, eps, rho_b, p_b;
  T fa, fb;        // outer ghost: rho, p and B_r factors (r_I / r_G)^a, ^b
  T fbp, fvr, fvp; // outer ghost: B_phi, V_r and V_phi factors
  T psi_out;       // outer ghost psi = psi_out * psi_I (-1: psi_b = 0, +1: zero-gradient)
  T psi_damp;      // GLM damping rate alpha: source -alpha psi in the psi equation (0: off)
  int inner_bc;    // inner boundary: 0 low-E, 1 large-E, 2 low-E with the V_r* magnitude
  double vr_star;  // large-E prescribed radial outflow
};

struct Shape {
  int nr, nt, np;
  int64_t ncell;
};

// (theta, phi) tile shapes of the tiled kernels: tile t has ens_tt(t) x
// ens_tp(t) columns per CTA.  A grid's own launch takes tile own_tile(): 8 x 32
// in FP32; 8 x 16 in FP64, whose CTA is bound by the FP64 pipe: half the
// columns cost 1.5 % more halo work per cell and give twice the CTAs to
// spread over the SMs.
constexpr int kEnsTileCount = 3;
__host__ __device__ constexpr int ens_tt(int t) { return t == 1 ? 16 : 8; }
__host__ __device__ constexpr int ens_tp(int t) { return t == 0 ? 32 : 16; }
__host__ __device__ constexpr int own_tile(bool fp64) { return fp64 ? 2 : 0; }

template <class T> __device__ __forceinline__ T fmat(T a, T b, T c);
template <> __device__ __forceinline__ double fmat<double>(double a, double b, double c) { return fma(a, b, c); }
template <> __device__ __forceinline__ float fmat<float>(float a, float b, float c) { return fmaf(a, b, c); }

// a product that is rounded by itself in FP64 (not contracted into a sum), so that
// a kept one and one formed in place are the same number
__device__ __forceinline__ double product(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float product(float a, float b) { return a * b; }

// Reciprocal and square root.  The FP64 pipe runs at 1/64 of the FP32 rate, so
// their FP64 operations are counted: both start from the approximate PTX
// instructions (about 20 bits, not on the FP64 pipe) and take one cubic step.
//   1/x: y0 (1 + e + e^2) with e = 1 - x y0 (Newton's series cut after e^2:
//        error e^3 ~ 2^-60), 3 operations, within one unit in the last place.
//        Where y0 is 0, infinite or NaN it is the result (1/0, 1/inf; on the
//        integer pipe): the step would make it NaN.
//   sqrt x: Goldschmidt's step on g = x y0 and h = y0 / 2 (y0 ~ 1 / sqrt x), then
//        Newton's with the exact remainder x - g^2: 6 operations (h halves an
//        exponent), correctly rounded but for values next to a rounding
//        boundary.  In particular the square root of a rounded square is its
//        base: with it a face state of negative pressure and B_n = 0 keeps c_f = 0
//        where a last place less would make q + sqrt(q^2) negative.  0 below
//        the normal range, +inf for +inf (an overflowing speed has to stay the
//        larger one), NaN for x < 0.
template <class T> __device__ __forceinline__ T frcp(T x);
template <> __device__ __forceinline__ double frcp<double>(double x) {
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double e = fma(-x, y, 1.0);
  const double r = fma(y, fma(e, e, e), y);
  const unsigned ey = (unsigned)__double2hiint(y) & 0x7ff00000u;
  return ey - 0x00100000u < 0x7fe00000u ? r : y;
}
template <> __device__ __forceinline__ float frcp<float>(float x) { return __fdividef(1.0f, x); }
template <class T> __device__ __forceinline__ T fsqrt(T x);
template <> __device__ __forceinline__ double fsqrt<double>(double x) {
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double h = __hiloint2double(__double2hiint(y) - 0x00100000, __double2loint(y));
  const double g = x * y;
  const double e = fma(-h, g, 0.5);
  const double g1 = fma(g, e, g);
  const double r = fma(fma(-g1, g1, x), fma(h, e, h), g1);
  const int hx = __double2hiint(x);
  return (hx & 0x7ff00000) == 0 ? 0.0 : hx == 0x7ff00000 ? x : r;
}
template <> __device__ __forceinline__ float fsqrt<float>(float x) { return sqrtf(x); }

// n / d for d > 0.  FP32: the approximate reciprocal.  FP64: on the integer pipe
// (about 55 instructions, which issue in the time of one FP64 operation per SM
// and warp, against four FP64 operations): Newton's series y0 (1 + e + e^2) for
// 2^63 / d's significand from an FP32 reciprocal y0 (24 bits, e < 2^-22, so that
// e^3 is below the last bit kept), times n's significand, rounded once: within
// 0.51 units in the last place (truncations of 2^-60 at most before it).  A
// quotient below the normal range and one of a subnormal n are 0; an infinite or
// NaN operand gives a NaN.  128 x 64 x 128 FP64: 1906 -> 1668 us.
__device__ __forceinline__ float quotient(float n, float d) { return n * frcp(d); }
__device__ __forceinline__ double quotient(double n, double d) {
  typedef unsigned long long u64;
  const unsigned nh = (unsigned)__double2hiint(n), nl = (unsigned)__double2loint(n);
  const unsigned dh = (unsigned)__double2hiint(d), dl = (unsigned)__double2loint(d);
  const unsigned ne = nh & 0x7ff00000u, de = dh & 0x7ff00000u;
  // significands with their leading bit at 63
  const unsigned n1 = __funnelshift_l(nl, nh | 0x100000u, 11), n0 = nl << 11;
  const unsigned d1 = __funnelshift_l(dl, dh | 0x100000u, 11), d0 = dl << 11;
  // y0 ~ 2^24 / m, m = d's significand in [1, 2)
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(__uint_as_float(0x3f800000u | ((d1 << 1) >> 9))));
  const unsigned y0 = __float_as_uint(r) - 0x3e800000u;
  // e in units of 2^-62 (|e| < 2^40), w = e + e^2, y = y0 (1 + w) ~ 2^63 / m
  const unsigned y7 = y0 << 7;
  const long long e = (1ll << 62) - (long long)((u64)d1 * y7 + (((u64)d0 * y7) >> 32));
  const int eh = (int)(e >> 15);
  const long long w = e + (((long long)eh * eh) >> 32);
  const u64 y = ((u64)y7 << 32) + (((u64)y0 * (unsigned)w) >> 23) + (u64)(((long long)y0 * (int)(w >> 32)) << 9);
  u64 q = __umul64hi(((u64)n1 << 32) | n0, y);  // n / d in [1/2, 2) as 2^62
  const int below = (int)(~(q >> 62) & 1ull);   // 1: the quotient of the significands is below 1
  q = ((q << below) + 512ull) >> 10;
  const int ex = (int)ne - (int)de + ((1022 - below) << 20);
  const u64 bits = q + ((u64)(unsigned)ex << 32);
  // no branch: the nine variables' quotients interleave
  const bool zero = ne == 0u || ex < 0, nan = ne == 0x7ff00000u || de == 0x7ff00000u;
  const unsigned hi = nan ? 0x7ff80000u : (zero ? 0u : (unsigned)(bits >> 32)) | ((nh ^ dh) & 0x80000000u);
  return __hiloint2double((int)hi, zero ? 0 : (int)(unsigned)bits);
}

// Comparisons of FP64 values on the integer pipe (an FP64 compare takes a slot
// of the FP64 pipe): positive doubles order as their bit patterns.
// positive(x): x > 0; greater(x, y): x > y for y >= +0.  Both false for a NaN of
// either sign: as unsigned numbers NaNs and negative values lie above +inf.
__device__ __forceinline__ bool positive(float x) { return x > 0.f; }
__device__ __forceinline__ bool positive(double x) {
  return (unsigned long long)__double_as_longlong(x) - 1ull < 0x7ff0000000000000ull;
}
__device__ __forceinline__ bool greater(float x, float y) { return x > y; }
__device__ __forceinline__ bool greater(double x, double y) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  return b > (unsigned long long)__double_as_longlong(y) && b <= 0x7ff0000000000000ull;
}

// x / 2 and 2 x of a normal x >= 0 (or 0) by its exponent, on the integer pipe;
// infinities and NaNs stay
__device__ __forceinline__ double halved(double x) {
  const int hi = __double2hiint(x), e = hi & 0x7ff00000;
  return __hiloint2double(e != 0 && e != 0x7ff00000 ? hi - 0x00100000 : hi, __double2loint(x));
}
__device__ __forceinline__ double doubled(double x) {
  const int hi = __double2hiint(x), e = hi & 0x7ff00000;
  return __hiloint2double(e != 0 && e != 0x7ff00000 ? hi + 0x00100000 : hi, __double2loint(x));
}

// |x| to FP32, cut off (not rounded), by integer instructions: 0 below the FP32
// normal range, +inf above it and for NaN
__device__ __forceinline__ float magnitude_f32(double x) {
  const int e = (__double2hiint(x) & 0x7fffffff) - 0x38000000;
  const unsigned b = __funnelshift_l((unsigned)__double2loint(x), (unsigned)e, 3);
  return __uint_as_float(e < 0x00100000 ? 0u : (e < 0x0ff00000 ? b : 0x7f800000u));
}

// ---------------------------------------------------------------------------
// primitive recovery [Sect. 2.2: E = p/(gamma-1) + rho V^2/2 + B^2/2]
// ---------------------------------------------------------------------------
// Threshold for the FP64 island of the FP32-bulk path: where B^2/2 exceeds the
// FP32 estimate of the internal energy (plasma beta < 2 (gamma-1) / gamma-ish),
// E - B^2/2 cancels and the internal energy is recomputed in FP64.
__device__ __forceinline__ void recover(const double (&u)[NV], const Phys<double>& ph,
                                        double (&w)[NV]) {
  const double ir = frcp(u[0]);
  const double vx = u[1] * ir, vy = u[2] * ir, vz = u[3] * ir;
  // twice the kinetic and magnetic energy
  const double t = fma(u[1], vx, fma(u[2], vy, fma(u[3], vz, fma(u[4], u[4], fma(u[5], u[5], u[6] * u[6])))));
  w[0] = u[0];
  w[1] = vx; w[2] = vy; w[3] = vz;
  w[4] = u[4]; w[5] = u[5]; w[6] = u[6];
  w[7] = ph.gm1 * fma(-0.5, t, u[7]);
  w[8] = u[8];
}

__device__ __forceinline__ void recover(const float (&u)[NV], const Phys<float>& ph,
                                        float (&w)[NV]) {
  const float ir = __fdividef(1.0f, u[0]);
  const float vx = u[1] * ir, vy = u[2] * ir, vz = u[3] * ir;
  const float ek = 0.5f * (u[1] * vx + u[2] * vy + u[3] * vz);
  const float eb = 0.5f * (u[4] * u[4] + u[5] * u[5] + u[6] * u[6]);
  float ei = u[7] - ek - eb;
  if (eb > ei) {
    // FP64 island: low-beta cell, E and B^2/2 nearly cancel
    const double bx = u[4], by = u[5], bz = u[6];
    const double e = (double)u[7] - 0.5 * (bx * bx + by * by + bz * bz) - (double)ek;
    ei = (float)e;
  }
  w[0] = u[0];
  w[1] = vx; w[2] = vy; w[3] = vz;
  w[4] = u[4]; w[5] = u[5]; w[6] = u[6];
  w[7] = ph.gm1 * ei;
  w[8] = u[8];
}

// ---------------------------------------------------------------------------
// ghost states (primitive); ghost = 2 * boundary - interior for V and B
// ---------------------------------------------------------------------------
// Inner boundary, Sect. 3.2 "low E": B_b = B_r rhat + tangential part of the
// interior B (Neumann in B_theta, B_phi); V_b = (V_I . B_b) B_b / |B_b|^2 so
// that V_b x B_b = 0; rho, p Dirichlet at the ghost centre; psi_b = 0
// (Sect. 3.3).  The vector algebra runs in FP64 in both precisions.
// Inner boundary, Sect. 3.2 "large E" (Wind-Predict): B_r and B_theta
// prescribed, B_phi Neumann; V_b = V_par (B_r rhat + B_theta thetahat) with
// V_par = V_r* B_r / (B_r^2 + B_theta^2), i.e. V_r = V_par B_r, V_theta =
// V_par B_theta, V_phi = 0; rho, p Dirichlet; psi_b = 0.  FP64.
template <class T>
__device__ __forceinline__ void large_e_ghost(const T (&wi)[NV], double br, double bt, double ex,
                                              double ey, double ez, const Phys<T>& ph, T (&wg)[NV]) {
  const double st = sqrt(ex * ex + ey * ey);        // sin(theta_c) > 0 at cell centres
  const double cp = ex / st, sp = ey / st;
  const double et[3] = {ez * cp, ez * sp, -st};     // thetahat
  const double ep[3] = {-sp, cp, 0.0};              // phihat
  const double er[3] = {ex, ey, ez};
  const double bip = (double)wi[4] * ep[0] + (double)wi[5] * ep[1];
  const double bpol2 = br * br + bt * bt;
  const double vpar = ph.vr_star * br / fmax(bpol2, 1e-300);
  wg[0] = ph.rho_b;
  wg[7] = ph.p_b;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const double pol = br * er[c] + bt * et[c];
    wg[1 + c] = (T)(2.0 * vpar * pol - (double)wi[1 + c]);
    wg[4 + c] = (T)(2.0 * (pol + bip * ep[c]) - (double)wi[4 + c]);
  }
  wg[8] = -wi[8];
}

// The prescribed boundary field is read from br_plane[col] (B_r) and, for the
// large-E form, br_plane[nc + col] (B_theta).
template <class T>
__device__ __forceinline__ void inner_ghost_at(const T (&wi)[NV], const double* __restrict__ br_plane,
                                               int64_t col, int64_t nc, double ex, double ey,
                                               double ez, const Phys<T>& ph, T (&wg)[NV]);

template <class T>
__device__ __forceinline__ void inner_ghost(const T (&wi)[NV], double br, double ex, double ey,
                                            double ez, const Phys<T>& ph, T (&wg)[NV]) {
  const double bix = wi[4], biy = wi[5], biz = wi[6];
  const double vix = wi[1], viy = wi[2], viz = wi[3];
  const double bir = bix * ex + biy * ey + biz * ez;
  const double bbx = br * ex + (bix - bir * ex);
  const double bby = br * ey + (biy - bir * ey);
  const double bbz = br * ez + (biz - bir * ez);
  const double bb2 = bbx * bbx + bby * bby + bbz * bbz;
  // V_b = s B_b: s from the interior velocity (low-E) or from the prescribed
  // outflow, s = V_r* B_r / |B_b|^2 (low-E with the Wind-Predict magnitude)
  const double s = ph.inner_bc == 2 ? ph.vr_star * br / fmax(bb2, 1e-300)
                                    : (vix * bbx + viy * bby + viz * bbz) / fmax(bb2, 1e-300);
  wg[0] = ph.rho_b;
  wg[1] = (T)(2.0 * s * bbx - vix);
  wg[2] = (T)(2.0 * s * bby - viy);
  wg[3] = (T)(2.0 * s * bbz - viz);
  wg[4] = (T)(2.0 * bbx - bix);
  wg[5] = (T)(2.0 * bby - biy);
  wg[6] = (T)(2.0 * bbz - biz);
  wg[7] = ph.p_b;
  wg[8] = -wi[8];
}

template <class T>
__device__ __forceinline__ void inner_ghost_at(const T (&wi)[NV], const double* __restrict__ br_plane,
                                               int64_t col, int64_t nc, double ex, double ey,
                                               double ez, const Phys<T>& ph, T (&wg)[NV]) {
  if (ph.inner_bc == 1)
    large_e_ghost(wi, br_plane[col], br_plane[nc + col], ex, ey, ez, ph, wg);
  else
    inner_ghost(wi, br_plane[col], ex, ey, ez, ph, wg);
}

// Outer boundary, Sect. 4.1 / Table 2 (all nine cases) and Sect. 4.2: with
// s = r_I / r_G (r_G mirrors r_I about r_out): rho_G = rho_I s^a, p_G = p_I s^a,
// B_r,G = B_r,I s^b, B_phi,G = B_phi,I s^c, V_r,G = V_r,I s^(2-a) (if V_r r^2
// rho = const) or V_r,I, V_phi,G = V_phi,I s^e; theta components
// zero-gradient; psi_G = -psi_I (psi_b = 0) or psi_I.  The factors are in ph.
template <class T>
__device__ __forceinline__ void outer_ghost(const T (&wi)[NV], T ex, T ey, T ez,
                                            const Phys<T>& ph, T (&wg)[NV]) {
  const T st = sqrt(ex * ex + ey * ey);
  const T px = -ey / st, py = ex / st;  // phihat (z component 0)
  const T bir = wi[4] * ex + wi[5] * ey + wi[6] * ez;
  const T bip = wi[4] * px + wi[5] * py;
  const T vir = wi[1] * ex + wi[2] * ey + wi[3] * ez;
  const T vip = wi[1] * px + wi[2] * py;
  const T dbr = bir * ph.fb - bir, dbp = bip * ph.fbp - bip;
  const T dvr = vir * ph.fvr - vir, dvp = vip * ph.fvp - vip;
  wg[0] = wi[0] * ph.fa;
  wg[1] = wi[1] + dvr * ex + dvp * px;
  wg[2] = wi[2] + dvr * ey + dvp * py;
  wg[3] = wi[3] + dvr * ez;
  wg[4] = wi[4] + dbr * ex + dbp * px;
  wg[5] = wi[5] + dbr * ey + dbp * py;
  wg[6] = wi[6] + dbr * ez;
  wg[7] = wi[7] * ph.fa;
  wg[8] = ph.psi_out * wi[8];
}

// ---------------------------------------------------------------------------
// slope limiters on the two one-sided slopes a (backward), b (forward)
// ---------------------------------------------------------------------------
template <int LIM, class T>
__device__ __forceinline__ T limited_slope(T a, T b, T eps) {
  if (LIM == 0) {  // unlimited central
    return (T)0.5 * (a + b);
  } else if (LIM == 1) {  // minmod
    if constexpr (sizeof(T) == 8) {
      // on the integer pipe (FP64 compares and products use the slow FP64
      // pipe): a b > 0 iff both are nonzero with equal sign bits, and the
      // magnitudes of non-negative doubles order as their bit patterns
      const unsigned long long ba = (unsigned long long)__double_as_longlong(a);
      const unsigned long long bb = (unsigned long long)__double_as_longlong(b);
      const unsigned long long ma = ba & 0x7fffffffffffffffull, mb = bb & 0x7fffffffffffffffull;
      const bool pos = ma != 0ull && mb != 0ull && ((ba ^ bb) >> 63) == 0ull;
      return pos ? (ma < mb ? a : b) : (T)0;
    } else {
      const T m = fabs(a) < fabs(b) ? a : b;
      return a * b > (T)0 ? m : (T)0;
    }
  } else {  // van Albada, smooth form: a (b^2 + eps) + b (a^2 + eps) is
            // (a + b)(a b + eps), one operation fewer; explicit FMAs so that
            // every kernel inlining this rounds it the same way
    const T num = (a + b) * fmat(a, b, eps);
    const T den = fmat(a, a, fmat(b, b, (T)2 * eps));
    return quotient(num, den);
  }
}

// ---------------------------------------------------------------------------
// Rusanov + GLM face flux through the unit normal n, times the face area.
// F* = (F(W_L) + F(W_R))/2 - lambda (U_R - U_L)/2,
// lambda = max(|u_n| + c_f over both sides, c_h);
// F_rho = rho u_n, F_m = rho V u_n + (p + B^2/2) n - B B_n,
// F_B = u_n B - B_n V + psi n, F_E = (E + p + B^2/2) u_n - B_n (V.B),
// F_psi = c_h^2 B_n.
//
// FP64: the flux is the longest chain of the residual (three per cell) on the
// slowest pipe, so its operations are counted: h = |S|/2 is multiplied into
// u_n, B_n and rho u_n once per side instead of into each of the nine sums, and
// the pressure and GLM gradient terms of both sides are added before they meet
// the normal: 109 operations, and 24 for each fast speed that is formed, against
// about 200 in all (every FMA explicit).  FP32
// keeps the sums by side: there the regrouping saved 3 % and moved the momentum
// of the polar cells, whose opposite faces nearly cancel, by 1e-7 per step.
// ---------------------------------------------------------------------------
template <class T>
struct Side {
  T un, bn, pt, en, vb, sp;
};

// NZ: the normal has a z component (phi faces have none)
template <bool NZ>
__device__ __forceinline__ Side<float> side_terms(const float (&w)[NV], float nx, float ny, float nz,
                                                  const Phys<float>& ph) {
  Side<float> s;
  const float ir = frcp(w[0]);
  s.un = w[1] * nx + w[2] * ny;
  s.bn = w[4] * nx + w[5] * ny;
  if (NZ) {
    s.un += w[3] * nz;
    s.bn += w[6] * nz;
  }
  const float b2 = w[4] * w[4] + w[5] * w[5] + w[6] * w[6];
  const float v2 = w[1] * w[1] + w[2] * w[2] + w[3] * w[3];
  s.vb = w[1] * w[4] + w[2] * w[5] + w[3] * w[6];
  s.pt = w[7] + 0.5f * b2;
  s.en = w[7] * ph.igm1 + 0.5f * (w[0] * v2 + b2);
  const float a2 = ph.gamma * w[7] * ir;
  const float sum = a2 + b2 * ir;
  float disc = sum * sum - 4.f * a2 * s.bn * s.bn * ir;
  disc = disc > 0.f ? disc : 0.f;
  const float cf = fsqrt(0.5f * (sum + fsqrt(disc)));
  s.sp = fabsf(s.un) + cf;
  return s;
}

// Whether a face state's signal speed is certainly below c_h, from an FP32 bound:
// for rho, p > 0, |u_n| + c_f <= |u_n| + sqrt(a^2 + B^2 / rho).  Then lambda = c_h
// and the FP64 fast speed (24 operations a side) need not be formed: both sides
// of three faces in four of a solar-wind shell.  The bound costs about 25
// integer and FP32 instructions, less than one FP64 operation; its margins
// (1e-5 of the squares, 1e-6 c_h) cover every rounding in it.
__device__ __forceinline__ bool speed_below_ch(double rho, double p, double un, double b2, const Phys<double>& ph) {
  const float r = magnitude_f32(rho), c = magnitude_f32(ph.ch);
  const float t = fmaf(-1e-6f, c, c) - magnitude_f32(un);
  const float q = fmaf(magnitude_f32(ph.gamma), magnitude_f32(p), magnitude_f32(b2));
  return (__double2hiint(rho) | __double2hiint(p)) >= 0 && r > 1e-20f && t > 0.f &&
         t * t * r > fmaf(1.00001f, q, 1e-18f * r);
}

// An FP32 estimate of |u_n| + c_f and a bound of its error, to tell which side of
// a face has the larger speed: only that side's is then formed in FP64.  Where
// the discriminant (a^2 - B^2/rho)^2 + 4 a^2 (B^2 - B_n^2)/rho nears zero its
// rounding, 1e-7 of q^2, moves the root by 1e-7 q^2 / root.  The error is
// infinite (either side may be larger) for rho, p <= 0 and out of FP32's range.
__device__ __forceinline__ float speed_estimate(double rho, double p, double un, double bn, double b2,
                                                const Phys<double>& ph, float& err) {
  const float r = magnitude_f32(rho), ir = __fdividef(1.f, r), u = magnitude_f32(un), b = magnitude_f32(bn);
  const float a2 = magnitude_f32(ph.gamma) * magnitude_f32(p) * ir, br = magnitude_f32(b2) * ir;
  const float q = a2 + br, d = a2 - br;
  const float root = sqrtf(fmaxf(fmaf(d, d, 4.f * a2 * fmaf(-b * ir, b, br)), 0.f));
  const float cf = sqrtf(0.5f * (q + root));
  err = fmaf(cf, fmaf(2e-6f, __fdividef(q, root), 2e-6f), 1e-6f * u);
  if (!((__double2hiint(rho) | __double2hiint(p)) >= 0 && r > 1e-20f && q > 1e-15f && q < 1e15f && err < 1e15f))
    err = INFINITY;
  return u + cf;
}

template <bool NZ>
__device__ __forceinline__ double dot_n(const double* w, double nx, double ny, double nz) {
  return NZ ? fma(w[0], nx, fma(w[1], ny, w[2] * nz)) : fma(w[0], nx, w[1] * ny);
}
__device__ __forceinline__ double dot3(const double* a, const double* b) {
  return fma(a[0], b[0], fma(a[1], b[1], a[2] * b[2]));
}

// |u_n| + c_f: c_f^2 = (q + sqrt(q^2 - 4 a^2 B_n^2 / rho)) / 2, q = a^2 + B^2 / rho
__device__ __forceinline__ double signal_speed(double rho, double p, double un, double bn, double b2,
                                               const Phys<double>& ph) {
  const double ir = frcp(rho);
  const double a2 = (ph.gamma * p) * ir;
  const double q = fma(b2, ir, a2);
  const double disc = fma(-4.0 * (a2 * ir), bn * bn, q * q);
  return fabs(un) + fsqrt(0.5 * (q + fsqrt(positive(disc) ? disc : 0.0)));
}

// sp holds B^2
template <bool NZ>
__device__ __forceinline__ Side<double> side_terms(const double (&w)[NV], double nx, double ny, double nz,
                                                   const Phys<double>& ph) {
  Side<double> s;
  s.un = dot_n<NZ>(w + 1, nx, ny, nz);
  s.bn = dot_n<NZ>(w + 4, nx, ny, nz);
  s.vb = dot3(w + 1, w + 4);
  s.sp = dot3(w + 4, w + 4);
  const double v2 = dot3(w + 1, w + 1);
  s.pt = fma(0.5, s.sp, w[7]);
  s.en = fma(0.5, fma(w[0], v2, s.sp), w[7] * ph.igm1);
  return s;
}

template <bool NZ = true>
__device__ __forceinline__ void rusanov(const float (&wl)[NV], const float (&wr)[NV], float nx, float ny,
                                        float nz, float area, const Phys<float>& ph, float (&f)[NV],
                                        float& lam_area) {
  const Side<float> L = side_terms<NZ>(wl, nx, ny, nz, ph);
  const Side<float> R = side_terms<NZ>(wr, nx, ny, nz, ph);
  float lam = L.sp > R.sp ? L.sp : R.sp;
  lam = lam > ph.ch ? lam : ph.ch;
  const float h = 0.5f * area;
  lam_area = lam * area;
  const float d = 0.5f * lam_area;  // halving is exact: the same value as (lam / 2) area
  const float n[3] = {nx, ny, nz};
  // mass
  const float ml = wl[0] * L.un, mr = wr[0] * R.un;
  f[0] = h * (ml + mr) - d * (wr[0] - wl[0]);
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const bool on = NZ || c < 2;
    // momentum: of the two products the pressure's is the exact one (explicit FMAs;
    // left to the compiler it was the mass flux's, and the mean error of the
    // momentum of a shell's cells 1.5 % larger)
    float a = ml * wl[1 + c], b = mr * wr[1 + c];
    if (on) { a = fmaf(L.pt, n[c], a); b = fmaf(R.pt, n[c], b); }
    a = fmaf(-wl[4 + c], L.bn, a);
    b = fmaf(-wr[4 + c], R.bn, b);
    f[1 + c] = h * (a + b) - d * (wr[0] * wr[1 + c] - wl[0] * wl[1 + c]);
    // induction with the GLM gradient term
    float p = L.un * wl[4 + c] - L.bn * wl[1 + c], q = R.un * wr[4 + c] - R.bn * wr[1 + c];
    if (on) { p += wl[8] * n[c]; q += wr[8] * n[c]; }
    f[4 + c] = h * (p + q) - d * (wr[4 + c] - wl[4 + c]);
  }
  // energy
  f[7] = h * (((L.en + L.pt) * L.un - L.bn * L.vb) + ((R.en + R.pt) * R.un - R.bn * R.vb))
         - d * (R.en - L.en);
  // cleaning scalar
  f[8] = h * (ph.ch2 * (L.bn + R.bn)) - d * (wr[8] - wl[8]);
}

template <bool NZ = true>
__device__ __forceinline__ void rusanov(const double (&wl)[NV], const double (&wr)[NV], double nx, double ny,
                                        double nz, double area, const Phys<double>& ph, double (&f)[NV],
                                        double& lam_area) {
  const Side<double> L = side_terms<NZ>(wl, nx, ny, nz, ph);
  const Side<double> R = side_terms<NZ>(wr, nx, ny, nz, ph);
  double lam = ph.ch;
  if (!(speed_below_ch(wl[0], wl[7], L.un, L.sp, ph) && speed_below_ch(wr[0], wr[7], R.un, R.sp, ph))) {
    float el, er;
    const float fl = speed_estimate(wl[0], wl[7], L.un, L.bn, L.sp, ph, el);
    const float fr = speed_estimate(wr[0], wr[7], R.un, R.bn, R.sp, ph, er);
    const bool left = fl > fr;
    lam = signal_speed(left ? wl[0] : wr[0], left ? wl[7] : wr[7], left ? L.un : R.un, left ? L.bn : R.bn,
                       left ? L.sp : R.sp, ph);
    if (!(fabsf(fl - fr) > el + er)) {  // too close to tell: the other side too
      const double o = signal_speed(left ? wr[0] : wl[0], left ? wr[7] : wl[7], left ? R.un : L.un,
                                    left ? R.bn : L.bn, left ? R.sp : L.sp, ph);
      // the larger, and the right one of a pair with a NaN left one
      const double sl = left ? lam : o, sr = left ? o : lam;
      lam = greater(sl, sr) ? sl : sr;
    }
    lam = greater(lam, ph.ch) ? lam : ph.ch;
  }
  const double h = halved(area);
  const double d = lam * h;
  lam_area = doubled(d);
  const double ul = h * L.un, ur = h * R.un, bl = h * L.bn, br = h * R.bn;
  const double ml = wl[0] * ul, mr = wr[0] * ur;
  const double pt = h * (L.pt + R.pt), ps = h * (wl[8] + wr[8]);
  const double n[3] = {nx, ny, nz};
  // mass
  f[0] = fma(-d, wr[0] - wl[0], ml + mr);
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const bool on = NZ || c < 2;
    // momentum
    double a = fma(mr, wr[1 + c], ml * wl[1 + c]);
    if (on) a = fma(pt, n[c], a);
    a = fma(-bl, wl[4 + c], a);
    a = fma(-br, wr[4 + c], a);
    f[1 + c] = fma(-d, fma(wr[0], wr[1 + c], -(wl[0] * wl[1 + c])), a);
    // induction with the GLM gradient term
    double e = fma(ur, wr[4 + c], ul * wl[4 + c]);
    e = fma(-bl, wl[1 + c], e);
    e = fma(-br, wr[1 + c], e);
    if (on) e = fma(ps, n[c], e);
    f[4 + c] = fma(-d, wr[4 + c] - wl[4 + c], e);
  }
  // energy
  double e = fma(R.en + R.pt, ur, (L.en + L.pt) * ul);
  e = fma(-bl, L.vb, e);
  e = fma(-br, R.vb, e);
  f[7] = fma(-d, R.en - L.en, e);
  // cleaning scalar
  f[8] = fma(-d, wr[8] - wl[8], ph.ch2 * (bl + br));
}

// across-pole / periodic mapping of a (possibly out-of-range) column (j, i):
// row -1 is row 0 and row -2 is row 1 on the opposite meridian (i + np/2),
// likewise beyond the south pole; phi is periodic.  Rows further out (only
// reached by the halo of a ragged tile, never by a used stencil) are clamped
// so that every mapped column is a valid index.
__device__ __forceinline__ void map_column(int& j, int& i, int nt, int np) {
  if (j < 0) { j = -1 - j; i += np / 2; }
  else if (j >= nt) { j = 2 * nt - 1 - j; i += np / 2; }
  j = j < 0 ? 0 : (j >= nt ? nt - 1 : j);
  while (i >= np) i -= np;  // i stays within a few periods: no integer division
  while (i < 0) i += np;
}

}  // namespace crn
