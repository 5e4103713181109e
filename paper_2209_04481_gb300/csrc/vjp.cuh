// vjp.cuh -- vector-Jacobian product of the residual: Ubar = (dR/dU)^T Rbar,
// Brbar = (dR/dB_r)^T Rbar.
//
// Reverse mode of the forward operator of residual.cuh, written by hand (the
// adjoint of every step: recovery, ghosts, limited reconstruction, the
// Rusanov + GLM flux, the accumulation and the gravity source).  With W the
// primitives, the face value of cell c on the side of a face is W_c +/- h s_c,
// s_c the limited slope L(a_c, b_c) of the one-sided differences a_c = (W_c -
// W_{c-1}) im_c, b_c = (W_{c+1} - W_c) ip_c.  A face's adjoint gives the
// cotangents u_c of the upper value of the cell below and l_c of the lower value
// of the cell above; the slope's cotangent is sbar_c = hp_c u_c - hm_c l_c, and
// with A_c = im_c sbar_c dL/da, B_c = ip_c sbar_c dL/db
//     Wbar_c += u_c + l_c + A_c - B_c,  Wbar_{c-1} -= A_c,  Wbar_{c+1} += B_c.
//
// Three passes through global memory, for the FP64 pipe (1/64 of the FP32
// rate): no slope and no face is evaluated twice, at 2.1 kB of scratch traffic
// per cell that hides under the arithmetic.
//   vjp_slopes  one thread per cell: its primitives and, along each axis and for
//               each variable, its limited slope with both derivatives
//   vjp_faces   one thread per face: its states from the slopes, the cotangent
//               fbar = Rbar_up / V_up - Rbar_lo / V_lo of its flux x area pulled
//               back to u and l
//   vjp_cells   one thread per cell: its own terms and those of its six
//               neighbours in a fixed order (no atomics), the ghosts' through the
//               ghost adjoints (inner ghost: also into Brbar), then the adjoints
//               of the recovery and of the sources
// The first version evaluated the slopes and their derivatives at each of the
// six faces that use them and stored 36 values per face: 3350 FP64 operations
// per cell, 5.67 ms on 128 x 64 x 128; now about 2100 and 3.62 ms (64 x 32 x 64:
// 0.75 -> 0.50 ms, of it slopes 0.18, faces 0.19, cells 0.13; 3.87 and 0.53 ms
// before the FP32 bound of the fast speeds).
// Non-smooth points follow the oracle's conventions: max(a, b) passes the
// derivative to a on a tie, d|x|/dx = +1 at 0, the clamp of the fast-speed
// discriminant at 0 has zero derivative.
#pragma once

#include "residual.cuh"

namespace crn {

// --------------------------------------------------------------------------
// limiter with its partial derivatives
// --------------------------------------------------------------------------
template <int LIM, class T>
__device__ __forceinline__ T slope_d(T a, T b, T eps, T& da, T& db) {
  if (LIM == 0) {
    da = (T)0.5; db = (T)0.5;
    return (T)0.5 * (a + b);
  } else if (LIM == 1) {
    if (!(a * b > (T)0)) { da = (T)0; db = (T)0; return (T)0; }
    if (fabs(a) < fabs(b)) { da = (T)1; db = (T)0; return a; }
    da = (T)0; db = (T)1;
    return b;
  } else if (sizeof(T) == 4) {
    const T N = a * (b * b + eps) + b * (a * a + eps);
    const T D = a * a + b * b + (T)2 * eps;
    const T iD = (T)1 / D;
    const T s = N * iD;
    da = ((b * b + eps) + (T)2 * a * b - s * (T)2 * a) * iD;
    db = ((T)2 * a * b + (a * a + eps) - s * (T)2 * b) * iD;
    return s;
  } else {
    // FP64, by count of operations: s = (a + b)(a b + eps) / D, D = a^2 + b^2 +
    // 2 eps; ds/da = (2 a b + b^2 + eps - 2 a s) / D and likewise ds/db
    const T p = fmat(a, b, eps), am = fmat(a, a, -eps), bm = fmat(b, b, -eps);
    const T iD = frcp(fmat((T)4, eps, am + bm));
    const T s = (a + b) * p * iD;
    const T s2 = s + s;
    da = fmat(-a, s2, fmat((T)2, p, bm)) * iD;
    db = fmat(-b, s2, fmat((T)2, p, am)) * iD;
    return s;
  }
}

// --------------------------------------------------------------------------
// adjoint of the Rusanov + GLM flux x area with respect to both face states
// --------------------------------------------------------------------------
template <class T>
struct SideFwd {
  T ir, un, bn, b2, v2, pt, en, a2, sum, sq, cf, sp, vb;
  bool clamp;
};

// FP32: the operations in the order the results of this kernel were pinned with
// (the clamp of the discriminant and the last bits of 1 / sqrt(disc) next to it
// move single cells by percents)
__device__ __forceinline__ SideFwd<float> side_fwd(const float (&w)[NV], float nx, float ny, float nz, const Phys<float>& ph) {
  SideFwd<float> s;
  s.ir = 1.f / w[0];
  s.un = w[1] * nx + w[2] * ny + w[3] * nz;
  s.bn = w[4] * nx + w[5] * ny + w[6] * nz;
  s.b2 = w[4] * w[4] + w[5] * w[5] + w[6] * w[6];
  s.v2 = w[1] * w[1] + w[2] * w[2] + w[3] * w[3];
  s.vb = w[1] * w[4] + w[2] * w[5] + w[3] * w[6];
  s.pt = w[7] + 0.5f * s.b2;
  s.en = w[7] * ph.igm1 + 0.5f * (w[0] * s.v2 + s.b2);
  s.a2 = ph.gamma * w[7] * s.ir;
  s.sum = s.a2 + s.b2 * s.ir;
  float disc = s.sum * s.sum - 4.f * s.a2 * s.bn * s.bn * s.ir;
  s.clamp = !(disc > 0.f);
  disc = s.clamp ? 0.f : disc;
  s.sq = sqrt(disc);
  s.cf = sqrt(0.5f * (s.sum + s.sq));
  s.sp = fabs(s.un) + s.cf;
  return s;
}

// cotangent wb of one side's primitive state; sig = -1 (left) / +1 (right);
// spb = cotangent reaching this side's signal speed
__device__ __forceinline__ void side_adjoint(const float (&w)[NV], const SideFwd<float>& s, float nx, float ny, float nz,
                                             float h, float d, float sig, float spb, const Phys<float>& ph,
                                             const float (&fb)[NV], float (&wb)[NV]) {
  const float n[3] = {nx, ny, nz};
  const float rho = w[0];
  const float v[3] = {w[1], w[2], w[3]};
  const float b[3] = {w[4], w[5], w[6]};
  const float m = rho * s.un;
  const float ds = d * sig;
  float rhob = -ds * fb[0];
  float mb = h * fb[0];
  float vb[3], bb[3];
  float ptb = 0.f, bnb = 0.f, unb = 0.f;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    // momentum: h (m v_c + pt n_c - b_c bn) - d sig rho v_c
    mb += h * fb[1 + c] * v[c];
    rhob -= ds * fb[1 + c] * v[c];
    vb[c] = h * fb[1 + c] * m - ds * fb[1 + c] * rho;
    ptb += h * fb[1 + c] * n[c];
    bb[c] = -h * fb[1 + c] * s.bn;
    bnb -= h * fb[1 + c] * b[c];
    // induction: h (un b_c - bn v_c + psi n_c) - d sig b_c
    unb += h * fb[4 + c] * b[c];
    bb[c] += h * fb[4 + c] * s.un - ds * fb[4 + c];
    bnb -= h * fb[4 + c] * v[c];
    vb[c] -= h * fb[4 + c] * s.bn;
  }
  float psib = h * (fb[4] * nx + fb[5] * ny + fb[6] * nz);
  // energy: h ((en + pt) un - bn vb) - d sig en
  const float enb = h * fb[7] * s.un - ds * fb[7];
  ptb += h * fb[7] * s.un;
  unb += h * fb[7] * (s.en + s.pt);
  bnb -= h * fb[7] * s.vb;
  const float vbdb = -h * fb[7] * s.bn;
  // cleaning scalar: h ch^2 bn - d sig psi
  bnb += h * ph.ch2 * fb[8];
  psib -= ds * fb[8];
  // m = rho un
  rhob += mb * s.un;
  unb += mb * rho;
  // en = p igm1 + (rho v2 + b2) / 2, pt = p + b2 / 2, vb = v.b
  float pb = enb * ph.igm1 + ptb;
  rhob += 0.5f * enb * s.v2;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    vb[c] += vbdb * b[c] + enb * rho * v[c];
    bb[c] += vbdb * v[c] + (enb + ptb) * b[c];
  }
  // signal speed sp = |un| + cf
  if (spb != 0.f) {
    unb += s.un >= 0.f ? spb : -spb;
    const float qb = spb / (2.f * s.cf);        // cf = sqrt(q), q = (sum + sq) / 2
    float sumb = 0.5f * qb;
    const float sqb = 0.5f * qb;
    const float discb = (s.clamp || !(s.sq > 0.f)) ? 0.f : sqb / (2.f * s.sq);
    // disc = sum^2 - 4 a2 bn^2 ir
    sumb += 2.f * s.sum * discb;
    float a2b = -4.f * s.bn * s.bn * s.ir * discb;
    bnb -= 8.f * s.a2 * s.bn * s.ir * discb;
    float irb = -4.f * s.a2 * s.bn * s.bn * discb;
    // sum = a2 + b2 ir
    a2b += sumb;
    const float b2b = sumb * s.ir;
    irb += sumb * s.b2;
    // a2 = gamma p ir
    pb += ph.gamma * s.ir * a2b;
    irb += ph.gamma * w[7] * a2b;
#pragma unroll
    for (int c = 0; c < 3; ++c) bb[c] += 2.f * b[c] * b2b;
    rhob -= s.ir * s.ir * irb;
  }
  // un = v.n, bn = b.n
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    vb[c] += unb * n[c];
    bb[c] += bnb * n[c];
  }
  wb[0] = rhob;
  wb[1] = vb[0]; wb[2] = vb[1]; wb[3] = vb[2];
  wb[4] = bb[0]; wb[5] = bb[1]; wb[6] = bb[2];
  wb[7] = pb;
  wb[8] = psib;
}

template <bool NZ = true>
__device__ void rusanov_adjoint(const float (&wl)[NV], const float (&wr)[NV], float nx, float ny, float nz, float area,
                                const Phys<float>& ph, const float (&fb)[NV], float (&wlb)[NV], float (&wrb)[NV]) {
  const SideFwd<float> L = side_fwd(wl, nx, ny, nz, ph);
  const SideFwd<float> R = side_fwd(wr, nx, ny, nz, ph);
  // lambda = max(max(sp_L, sp_R), c_h); a tie passes the derivative to the first argument
  const bool selR = R.sp > L.sp;
  const float lam_s = selR ? R.sp : L.sp;
  const bool useC = ph.ch > lam_s;
  const float lam = useC ? ph.ch : lam_s;
  const float h = 0.5f * area, d = 0.5f * lam * area;
  // lambda cotangent: f_v contains -lambda area (U_R - U_L)_v / 2
  const float dU[NV] = {wr[0] - wl[0],
                    wr[0] * wr[1] - wl[0] * wl[1],
                    wr[0] * wr[2] - wl[0] * wl[2],
                    wr[0] * wr[3] - wl[0] * wl[3],
                    wr[4] - wl[4], wr[5] - wl[5], wr[6] - wl[6],
                    R.en - L.en, wr[8] - wl[8]};
  float lamb = 0.f;
#pragma unroll
  for (int v = 0; v < NV; ++v) lamb -= 0.5f * area * fb[v] * dU[v];
  const float spbL = (!useC && !selR) ? lamb : 0.f;
  const float spbR = (!useC && selR) ? lamb : 0.f;
  side_adjoint(wl, L, nx, ny, nz, h, d, -1.f, spbL, ph, fb, wlb);
  side_adjoint(wr, R, nx, ny, nz, h, d, 1.f, spbR, ph, fb, wrb);
}

// FP64, by count of operations (about 305 against 410): h fb and d fb formed
// once for both sides, and the signal speed's adjoint taken once, on the side
// that sets lambda
template <bool NZ>
__device__ __forceinline__ SideFwd<double> side_fwd(const double (&w)[NV], double nx, double ny, double nz, const Phys<double>& ph) {
  SideFwd<double> s;
  s.un = fma(w[1], nx, w[2] * ny);
  s.bn = fma(w[4], nx, w[5] * ny);
  if (NZ) {
    s.un = fma(w[3], nz, s.un);
    s.bn = fma(w[6], nz, s.bn);
  }
  s.b2 = fma(w[4], w[4], fma(w[5], w[5], w[6] * w[6]));
  s.v2 = fma(w[1], w[1], fma(w[2], w[2], w[3] * w[3]));
  s.vb = fma(w[1], w[4], fma(w[2], w[5], w[3] * w[6]));
  s.pt = fma(0.5, s.b2, w[7]);
  s.en = fma(0.5, fma(w[0], s.v2, s.b2), w[7] * ph.igm1);
  return s;
}

// the signal speed of a side and what its adjoint needs
__device__ __forceinline__ void side_speed(double rho, double p, const Phys<double>& ph, SideFwd<double>& s) {
  s.ir = frcp(rho);
  s.a2 = (ph.gamma * p) * s.ir;
  s.sum = fma(s.b2, s.ir, s.a2);
  const double disc = fma(-4.0 * (s.a2 * s.ir), s.bn * s.bn, s.sum * s.sum);
  s.clamp = !positive(disc);
  s.sq = fsqrt(s.clamp ? 0.0 : disc);
  s.cf = fsqrt(0.5 * (s.sum + s.sq));
  s.sp = fabs(s.un) + s.cf;
}

// what both sides of a face share: h fb, d fb, and their sums along the normal
struct FaceBar {
  double hf[NV], df[NV], pn, sn;
};

// cotangent wb of one side's primitive state, without the signal speed and
// before the normal components: unb and bnb are the cotangents of u_n and B_n;
// alpha = h u_n -/+ d (the side's sign) weights fb in every U-like term
__device__ __forceinline__ void side_adjoint(const double (&w)[NV], const SideFwd<double>& s, double h, double d, double sig,
                                             const Phys<double>& ph, const double (&fb)[NV], const FaceBar& c,
                                             double (&wb)[NV], double& unb, double& bnb) {
  const double alpha = fma(h, s.un, -sig * d);
  const double kap = w[0] * alpha;
  // h (m + ...) : mb the cotangent of m = rho u_n
  const double mb = c.hf[0] + fma(c.hf[1], w[1], fma(c.hf[2], w[2], c.hf[3] * w[3]));
  const double dv = c.df[0] + fma(c.df[1], w[1], fma(c.df[2], w[2], c.df[3] * w[3]));
  const double enb = alpha * fb[7];
  const double ptb = fma(c.hf[7], s.un, c.pn);
  const double vbdb = -c.hf[7] * s.bn;
  const double er = enb * w[0], ep = enb + ptb;
  unb = fma(c.hf[4], w[4], fma(c.hf[5], w[5], c.hf[6] * w[6]));
  unb = fma(c.hf[7], s.en + s.pt, unb);
  unb = fma(mb, w[0], unb);
  bnb = fma(c.hf[1], w[4], fma(c.hf[2], w[5], c.hf[3] * w[6]));
  bnb = fma(c.hf[4], w[1], fma(c.hf[5], w[2], fma(c.hf[6], w[3], bnb)));
  bnb = fma(c.hf[7], s.vb, bnb);
  bnb = fma(ph.ch2, c.hf[8], -bnb);
  wb[0] = fma(0.5 * enb, s.v2, fma(mb, s.un, -sig * dv));
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    double v = fma(kap, fb[1 + q], -c.hf[4 + q] * s.bn);
    v = fma(vbdb, w[4 + q], v);
    wb[1 + q] = fma(er, w[1 + q], v);
    double b = fma(alpha, fb[4 + q], -c.hf[1 + q] * s.bn);
    b = fma(vbdb, w[1 + q], b);
    wb[4 + q] = fma(ep, w[4 + q], b);
  }
  wb[7] = fma(enb, ph.igm1, ptb);
  wb[8] = fma(-sig, c.df[8], c.sn);
}

// NZ: the normal has a z component (phi faces have none)
template <bool NZ = true>
__device__ __forceinline__ void rusanov_adjoint(const double (&wl)[NV], const double (&wr)[NV], double nx, double ny, double nz, double area,
                                                const Phys<double>& ph, const double (&fb)[NV], double (&wlb)[NV], double (&wrb)[NV]) {
  SideFwd<double> L = side_fwd<NZ>(wl, nx, ny, nz, ph);
  SideFwd<double> R = side_fwd<NZ>(wr, nx, ny, nz, ph);
  // lambda = max(max(sp_L, sp_R), c_h); a tie passes the derivative to the first argument
  bool selR = false, useC = true;
  double lam = ph.ch;
  if (!(speed_below_ch(wl[0], wl[7], L.un, L.b2, ph) && speed_below_ch(wr[0], wr[7], R.un, R.b2, ph))) {
    side_speed(wl[0], wl[7], ph, L);
    side_speed(wr[0], wr[7], ph, R);
    selR = greater(R.sp, L.sp);
    const double lam_s = selR ? R.sp : L.sp;
    useC = greater(ph.ch, lam_s);
    lam = useC ? ph.ch : lam_s;
  }
  const double h = 0.5 * area, d = lam * h;
  FaceBar c;
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    c.hf[v] = h * fb[v];
    c.df[v] = d * fb[v];
  }
  c.pn = fma(c.hf[1], nx, c.hf[2] * ny);
  c.sn = fma(c.hf[4], nx, c.hf[5] * ny);
  if (NZ) {
    c.pn = fma(c.hf[3], nz, c.pn);
    c.sn = fma(c.hf[6], nz, c.sn);
  }
  double unl, bnl, unr, bnr;
  side_adjoint(wl, L, h, d, -1.0, ph, fb, c, wlb, unl, bnl);
  side_adjoint(wr, R, h, d, 1.0, ph, fb, c, wrb, unr, bnr);
  if (!useC) {
    // lambda cotangent: f_v contains -lambda area (U_R - U_L)_v / 2
    double lamb = c.hf[0] * (wr[0] - wl[0]);
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      lamb = fma(c.hf[1 + q], fma(wr[0], wr[1 + q], -(wl[0] * wl[1 + q])), lamb);
      lamb = fma(c.hf[4 + q], wr[4 + q] - wl[4 + q], lamb);
    }
    lamb = fma(c.hf[7], R.en - L.en, lamb);
    lamb = -fma(c.hf[8], wr[8] - wl[8], lamb);
    if (lamb != 0.0) {
      // the signal speed of the side that sets lambda, sp = |un| + cf: once, on
      // that side's values
      const double un = selR ? R.un : L.un, bn = selR ? R.bn : L.bn, ir = selR ? R.ir : L.ir, a2 = selR ? R.a2 : L.a2;
      const double b2 = selR ? R.b2 : L.b2, sum = selR ? R.sum : L.sum, sq = selR ? R.sq : L.sq, cf = selR ? R.cf : L.cf;
      const double p = selR ? wr[7] : wl[7];
      const bool clamp = selR ? R.clamp : L.clamp;
      const double uns = un >= 0.0 ? lamb : -lamb;
      // cf = sqrt(q), q = (sum + sq) / 2; sq = sqrt(disc)
      const double half = 0.25 * lamb * frcp(cf);
      const double discb = clamp || !positive(sq) ? 0.0 : 0.5 * half * frcp(sq);
      // disc = sum^2 - 4 a2 bn^2 ir, sum = a2 + b2 ir, a2 = gamma p ir
      const double sumb = fma(2.0 * sum, discb, half);
      const double t = -4.0 * bn * discb;
      const double bni = t * bn * ir;               // -4 bn^2 ir discb
      const double a2b = bni + sumb;
      const double bns = 2.0 * t * a2 * ir;
      const double irb = fma(ph.gamma * p, a2b, fma(sumb, b2, t * bn * a2));
      const double pbs = ph.gamma * ir * a2b;
      const double b2b = 2.0 * sumb * ir;
      const double rhos = ir * ir * irb;
      const double zero = 0.0;
      unl += selR ? zero : uns;
      unr += selR ? uns : zero;
      bnl += selR ? zero : bns;
      bnr += selR ? bns : zero;
      wlb[0] -= selR ? zero : rhos;
      wrb[0] -= selR ? rhos : zero;
      wlb[7] += selR ? zero : pbs;
      wrb[7] += selR ? pbs : zero;
      const double bl = selR ? zero : b2b, br = selR ? b2b : zero;
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        wlb[4 + q] = fma(bl, wl[4 + q], wlb[4 + q]);
        wrb[4 + q] = fma(br, wr[4 + q], wrb[4 + q]);
      }
    }
  }
  // un = v.n, bn = b.n
  const double n[3] = {nx, ny, nz};
#pragma unroll
  for (int q = 0; q < (NZ ? 3 : 2); ++q) {
    wlb[1 + q] = fma(unl, n[q], wlb[1 + q]);
    wlb[4 + q] = fma(bnl, n[q], wlb[4 + q]);
    wrb[1 + q] = fma(unr, n[q], wrb[1 + q]);
    wrb[4 + q] = fma(bnr, n[q], wrb[4 + q]);
  }
}

// --------------------------------------------------------------------------
// adjoints of the ghost maps and of the primitive recovery
// --------------------------------------------------------------------------
// inner low-E ghost: from the ghost's cotangent gb, add to the interior
// primitive's cotangent wib and return the cotangent of the prescribed B_r
template <class T>
__device__ double inner_ghost_adjoint(const T (&wi)[NV], double br, double ex, double ey, double ez,
                                      const Phys<T>& ph, const T (&gb)[NV], T (&wib)[NV]) {
  const double e[3] = {ex, ey, ez};
  const double bi[3] = {wi[4], wi[5], wi[6]};
  const double vi[3] = {wi[1], wi[2], wi[3]};
  const double bir = bi[0] * ex + bi[1] * ey + bi[2] * ez;
  double bbd[3];
  for (int c = 0; c < 3; ++c) bbd[c] = br * e[c] + (bi[c] - bir * e[c]);
  const double bb2 = bbd[0] * bbd[0] + bbd[1] * bbd[1] + bbd[2] * bbd[2];
  const bool wp = ph.inner_bc == 2;
  const double num = wp ? ph.vr_star * br : vi[0] * bbd[0] + vi[1] * bbd[1] + vi[2] * bbd[2];
  const bool floor = !(bb2 > 1e-300);
  const double den = floor ? 1e-300 : bb2;
  const double s = num / den;
  // ghost: V_g = 2 s B_b - V_I, B_g = 2 B_b - B_I, psi_g = -psi_I (rho, p fixed)
  double Bbb[3], sb = 0.0;
  for (int c = 0; c < 3; ++c) {
    const double vgb = gb[1 + c], bgb = gb[4 + c];
    Bbb[c] = 2.0 * bgb + 2.0 * s * vgb;
    sb += 2.0 * vgb * bbd[c];
    wib[1 + c] -= (T)vgb;
    wib[4 + c] -= (T)bgb;
  }
  wib[8] -= gb[8];
  // s = num / den; num = V_I . B_b (low-E) or V_r* B_r (Wind-Predict magnitude)
  const double numb = sb / den;
  const double bb2b = floor ? 0.0 : -sb * s / den;
  double brb = 0.0;
  for (int c = 0; c < 3; ++c) Bbb[c] += 2.0 * bb2b * bbd[c];
  if (wp) {
    brb = numb * ph.vr_star;
  } else {
    for (int c = 0; c < 3; ++c) {
      wib[1 + c] += (T)(numb * bbd[c]);
      Bbb[c] += numb * vi[c];
    }
  }
  // B_b = B_r e + B_I - (B_I . e) e
  const double Be = Bbb[0] * ex + Bbb[1] * ey + Bbb[2] * ez;
  for (int c = 0; c < 3; ++c) wib[4 + c] += (T)(Bbb[c] - Be * e[c]);
  return brb + Be;
}

// large-E inner ghost: cotangents to the interior primitive and to the
// prescribed (B_r, B_theta), returned in brb[0], brb[1]
template <class T>
__device__ void large_e_ghost_adjoint(double br, double bt, double ex, double ey, double ez,
                                      const Phys<T>& ph, const T (&gb)[NV], T (&wib)[NV],
                                      double (&brb)[2]) {
  const double st = sqrt(ex * ex + ey * ey);
  const double cp = ex / st, sp = ey / st;
  const double et[3] = {ez * cp, ez * sp, -st};
  const double ep[3] = {-sp, cp, 0.0};
  const double er[3] = {ex, ey, ez};
  const double D = br * br + bt * bt;
  const bool floor = !(D > 1e-300);
  const double Dd = floor ? 1e-300 : D;
  const double vpar = ph.vr_star * br / Dd;
  double polb[3], vparb = 0.0, bipb = 0.0;
  for (int c = 0; c < 3; ++c) {
    const double vg = gb[1 + c], bg = gb[4 + c];
    const double pol = br * er[c] + bt * et[c];
    polb[c] = 2.0 * vpar * vg + 2.0 * bg;
    vparb += 2.0 * vg * pol;
    bipb += 2.0 * bg * ep[c];
    wib[1 + c] -= (T)vg;
    wib[4 + c] -= (T)bg;
  }
  wib[8] -= gb[8];
  for (int c = 0; c < 3; ++c) wib[4 + c] += (T)(bipb * ep[c]);
  brb[0] = polb[0] * er[0] + polb[1] * er[1] + polb[2] * er[2];
  brb[1] = polb[0] * et[0] + polb[1] * et[1] + polb[2] * et[2];
  // V_par = vr* B_r / D, D = B_r^2 + B_theta^2
  if (floor) {
    brb[0] += vparb * ph.vr_star / Dd;
  } else {
    brb[0] += vparb * (ph.vr_star / D - 2.0 * ph.vr_star * br * br / (D * D));
    brb[1] += vparb * (-2.0 * ph.vr_star * br * bt / (D * D));
  }
}

// generalized outer ghost (Table 2 laws): the ghost is a fixed linear map of
// the interior primitive state
template <class T>
__device__ __forceinline__ void outer_ghost_adjoint(T ex, T ey, T ez, const Phys<T>& ph,
                                                    const T (&gb)[NV], T (&wib)[NV]) {
  const T st = sqrt(ex * ex + ey * ey);
  const T px = -ey / st, py = ex / st;
  const T e[3] = {ex, ey, ez};
  const T pe[3] = {px, py, (T)0};
  wib[0] += ph.fa * gb[0];
  wib[7] += ph.fa * gb[7];
  const T bre = gb[4] * ex + gb[5] * ey + gb[6] * ez, bpe = gb[4] * px + gb[5] * py;
  const T vre = gb[1] * ex + gb[2] * ey + gb[3] * ez, vpe = gb[1] * px + gb[2] * py;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    wib[1 + c] += gb[1 + c] + (ph.fvr - (T)1) * vre * e[c] + (ph.fvp - (T)1) * vpe * pe[c];
    wib[4 + c] += gb[4 + c] + (ph.fb - (T)1) * bre * e[c] + (ph.fbp - (T)1) * bpe * pe[c];
  }
  wib[8] += ph.psi_out * gb[8];
}

// U -> W recovery adjoint (plain, no low-beta island: derivatives only)
template <class T>
__device__ __forceinline__ void recover_adjoint(const T (&u)[NV], const Phys<T>& ph,
                                                const T (&wb)[NV], T (&ub)[NV]) {
  const T ir = sizeof(T) == 4 ? (T)1 / u[0] : frcp(u[0]);
  const T v[3] = {u[1] * ir, u[2] * ir, u[3] * ir};
  const T pb = wb[7] * ph.gm1;
  T u0 = wb[0] + pb * (T)0.5 * (v[0] * v[0] + v[1] * v[1] + v[2] * v[2]);
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    u0 -= wb[1 + c] * v[c] * ir;
    ub[1 + c] = wb[1 + c] * ir - pb * v[c];
    ub[4 + c] = wb[4 + c] - pb * u[4 + c];
  }
  ub[0] = u0;
  ub[7] = pb;
  ub[8] = wb[8];
}

// --------------------------------------------------------------------------
// the three passes; scratch of one VJP, in elements of T
// --------------------------------------------------------------------------
// slopes: [3 axes][3: slope, d/da, d/db][NV][N]; face cotangents per axis
// [2: u of the cell below, l of the cell above][NV][faces]
template <class T>
struct VjpBufs {
  T* W;      // [NV][N] primitives
  T* S;      // slopes
  T* fr;     // r faces     (nr + 1) * nt * np
  T* ft;     // theta faces nr * (nt + 1) * np
  T* fp;     // phi faces   nr * nt * np
};

template <class T, int LIM>
__global__ void __launch_bounds__(128)
vjp_slopes(Shape sh, Geo<T> g, Phys<T> ph, const double* __restrict__ Br, const T* __restrict__ U,
           VjpBufs<T> out) {
  const int nr = sh.nr, nt = sh.nt, np = sh.np;
  const int64_t N = sh.ncell, cs = (int64_t)nt * np;
  const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= N) return;
  const int axis = blockIdx.y;  // 0 = r, 1 = theta, 2 = phi
  const int k = (int)(c / cs), col = (int)(c - k * cs), j = col / np, i = col - j * np;
  // the neighbours' columns and planes along the axis
  int64_t cm = c, cp = c;
  if (axis == 0) {
    cm = k > 0 ? c - cs : c;
    cp = k < nr - 1 ? c + cs : c;
  } else if (axis == 1) {  // across a pole: the opposite column's cell
    int io = i + np / 2;
    io = io >= np ? io - np : io;
    cm = j > 0 ? c - np : (int64_t)k * cs + io;
    cp = j < nt - 1 ? c + np : (int64_t)k * cs + (int64_t)(nt - 1) * np + io;
  } else {
    cm = i > 0 ? c - 1 : c + np - 1;
    cp = i < np - 1 ? c + 1 : c - np + 1;
  }
  T u[NV], um[NV], up[NV], w[NV], wm[NV], wp[NV];
  load_raw(U, N, c, u);
  load_raw(U, N, cm, um);
  load_raw(U, N, cp, up);
  recover(u, ph, w);
  T im = (T)1, ip = (T)1;
  if (axis == 0) {
    im = g.inv_dm[k];
    ip = g.inv_dp[k];
#pragma unroll
    for (int v = 0; v < NV; ++v) out.W[v * N + c] = w[v];
  }
  if (axis == 0 && k == 0)
    inner_ghost_at(w, Br, col, cs, (double)g.rhat[col], (double)g.rhat[cs + col], (double)g.rhat[2 * cs + col], ph, wm);
  else
    recover(um, ph, wm);
  if (axis == 0 && k == nr - 1)
    outer_ghost(w, g.rhat[col], g.rhat[cs + col], g.rhat[2 * cs + col], ph, wp);
  else
    recover(up, ph, wp);
  T* S = out.S + (int64_t)axis * 3 * NV * N;
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    T a = w[v] - wm[v], b = wp[v] - w[v];
    if (axis == 0) {
      a *= im;
      b *= ip;
    }
    T da, db;
    S[v * N + c] = slope_d<LIM>(a, b, ph.eps, da, db);
    S[(NV + v) * N + c] = da;
    S[(2 * NV + v) * N + c] = db;
  }
}

// the slopes of cell c = (k, j, i) along one axis with their derivatives: read
// from the first pass (FP64 grids), or formed again from its three cells
// (STORED = false: the FP32 reference variant, two launches)
template <int LIM, bool STORED, class T>
__device__ __forceinline__ void slopes_of(const Shape& sh, const Geo<T>& g, const Phys<T>& ph,
                                          const double* __restrict__ Br, const T* __restrict__ U,
                                          const VjpBufs<T>& b, int axis, int k, int j, int i, T (&s)[NV],
                                          T (&da)[NV], T (&db)[NV]) {
  if (STORED) {
    const int64_t N = sh.ncell, c = ((int64_t)k * sh.nt + j) * sh.np + i;
    const T* S = b.S + (int64_t)axis * 3 * NV * N + c;
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      s[v] = S[v * N];
      da[v] = S[(NV + v) * N];
      db[v] = S[(2 * NV + v) * N];
    }
  } else {
    T wm[NV], w[NV], wp[NV];
    cell_prim(sh, g, ph, Br, U, k - (axis == 0), j - (axis == 1), i - (axis == 2), wm);
    cell_prim(sh, g, ph, Br, U, k, j, i, w);
    cell_prim(sh, g, ph, Br, U, k + (axis == 0), j + (axis == 1), i + (axis == 2), wp);
    const T im = axis == 0 ? g.inv_dm[k] : (T)1, ip = axis == 0 ? g.inv_dp[k] : (T)1;
#pragma unroll
    for (int v = 0; v < NV; ++v)
      s[v] = slope_d<LIM>((w[v] - wm[v]) * im, (wp[v] - w[v]) * ip, ph.eps, da[v], db[v]);
  }
}

// One launch over the faces of all three axes (r faces, then theta, then
// phi): a thread per face, so that small grids still fill the GPU.
template <class T, int LIM, bool STORED>
__global__ void __launch_bounds__(128)
vjp_faces(Shape sh, Geo<T> g, Phys<T> ph, const double* __restrict__ Br, const T* __restrict__ U,
          const T* __restrict__ Rb, VjpBufs<T> buf) {
  const int nr = sh.nr, nt = sh.nt, np = sh.np;
  const int64_t cs = (int64_t)nt * np, N = sh.ncell;
  const int64_t nf0 = (int64_t)(nr + 1) * cs, nf1 = (int64_t)nr * (nt + 1) * np, nf2 = (int64_t)nr * cs;
  int64_t f = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  int axis = 0;
  int64_t nf = nf0;
  T* out = buf.fr;
  if (f >= nf0) {
    f -= nf0;
    axis = 1; nf = nf1; out = buf.ft;
    if (f >= nf1) {
      f -= nf1;
      axis = 2; nf = nf2; out = buf.fp;
      if (f >= nf2) return;
    }
  }
  // the cells below and above (indices of existing cells), 1 / V, the normal
  const T one = (T)1, half = (T)0.5;
  int64_t cl, cu;
  T nx, ny, nz, area, vl, vu, hl = half, hu = half;
  bool ghost_l = false, ghost_u = false;
  int col, kl, jl, il, ku, ju, iu;  // the two cells' places
  if (axis == 0) {
    const int a = (int)(f / cs);
    col = (int)(f - a * cs);
    const int j = col / np;
    kl = a - 1; ku = a; jl = ju = j; il = iu = col - j * np;
    ghost_l = a == 0;
    ghost_u = a == nr;
    cl = ghost_l ? f : f - cs;
    cu = ghost_u ? f - cs : f;
    nx = g.nr[col]; ny = g.nr[cs + col]; nz = g.nr[2 * cs + col];
    area = g.ra[a] * g.ar[j];
    vl = ghost_l ? one : g.rv[a - 1] * g.av[j];
    vu = ghost_u ? one : g.rv[a] * g.av[j];
    if (!ghost_l && !ghost_u) { hl = g.hp[a - 1]; hu = g.hm[a]; }
  } else if (axis == 1) {
    const int64_t row = f / np;
    const int i = (int)(f - row * np), k = (int)(row / (nt + 1)), a = (int)(row - (int64_t)k * (nt + 1));
    if (a == 0 || a == nt) {  // poles: zero area
#pragma unroll
      for (int v = 0; v < 2 * NV; ++v) out[v * nf + f] = (T)0;
      return;
    }
    kl = ku = k; jl = a - 1; ju = a; il = iu = i;
    cl = (int64_t)k * cs + (int64_t)(a - 1) * np + i;
    cu = cl + np;
    const int64_t ts = (int64_t)(nt + 1) * np, fc = (int64_t)a * np + i;
    nx = g.nth[fc]; ny = g.nth[ts + fc]; nz = g.nth[2 * ts + fc];
    area = g.rb[k] * g.at[a];
    vl = g.rv[k] * g.av[a - 1];
    vu = g.rv[k] * g.av[a];
    col = 0;
  } else {
    const int64_t row = f / np;
    const int a = (int)(f - row * np), k = (int)(row / nt), j = (int)(row - (int64_t)k * nt);
    kl = ku = k; jl = ju = j; iu = a; il = a > 0 ? a - 1 : np - 1;
    cu = f;
    cl = a > 0 ? f - 1 : f + np - 1;
    nx = g.nph[a]; ny = g.nph[np + a]; nz = (T)0;
    area = g.rb[k] * g.dtheta;
    vl = vu = g.rv[k] * g.av[j];
    col = 0;
  }
  const T sl = frcp(vl), su = frcp(vu);
  T wl[NV], wr[NV], fb[NV];
  if (STORED) {
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      wl[v] = buf.W[v * N + cl];
      wr[v] = buf.W[v * N + cu];
    }
  } else {
    load_recover(U, N, cl, ph, wl);
    load_recover(U, N, cu, ph, wr);
  }
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    const T rl = ghost_l ? (T)0 : Rb[v * N + cl], ru = ghost_u ? (T)0 : Rb[v * N + cu];
    fb[v] = fmat(ru, su, -(rl * sl));
  }
  if (ghost_l || ghost_u) {  // boundary faces: first order
    if (ghost_l) {
      T w0[NV];
#pragma unroll
      for (int v = 0; v < NV; ++v) w0[v] = wr[v];
      inner_ghost_at(w0, Br, col, cs, (double)g.rhat[col], (double)g.rhat[cs + col],
                     (double)g.rhat[2 * cs + col], ph, wl);
    } else {
      T w0[NV];
#pragma unroll
      for (int v = 0; v < NV; ++v) w0[v] = wl[v];
      outer_ghost(w0, g.rhat[col], g.rhat[cs + col], g.rhat[2 * cs + col], ph, wr);
    }
  } else {
    T ds[NV], us[NV], da[NV], db[NV];
    slopes_of<LIM, STORED>(sh, g, ph, Br, U, buf, axis, kl, jl, il, ds, da, db);
    slopes_of<LIM, STORED>(sh, g, ph, Br, U, buf, axis, ku, ju, iu, us, da, db);
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      wl[v] = fmat(hl, ds[v], wl[v]);
      wr[v] = fmat(-hu, us[v], wr[v]);
    }
  }
  T ul[NV], lu[NV];
  rusanov_adjoint(wl, wr, nx, ny, nz, area, ph, fb, ul, lu);
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    out[v * nf + f] = ul[v];
    out[(NV + v) * nf + f] = lu[v];
  }
}

template <class T, int LIM, bool STORED>
__global__ void __launch_bounds__(128)
vjp_cells(Shape sh, Geo<T> g, Phys<T> ph, const double* __restrict__ Br, const T* __restrict__ U,
          const T* __restrict__ Rb, VjpBufs<T> in, T* __restrict__ Ub, double* __restrict__ Brb) {
  const int nr = sh.nr, nt = sh.nt, np = sh.np;
  const int64_t cs = (int64_t)nt * np, N = sh.ncell;
  const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= N) return;
  const int k = (int)(c / cs), col = (int)(c - k * cs), j = col / np, i = col - j * np;
  const int64_t nfr = (int64_t)(nr + 1) * cs, nft = (int64_t)nr * (nt + 1) * np, nfp = (int64_t)nr * cs;
  const T half = (T)0.5;
  T wb[NV], gin[NV], gout[NV], none[NV];
  auto slopes = [&](int axis, int ks, int js, int is, T (&da)[NV], T (&db)[NV]) {
    T s[NV];
    slopes_of<LIM, STORED>(sh, g, ph, Br, U, in, axis, ks, js, is, s, da, db);
  };
  {  // r: first-order boundary faces reach the cell directly, not its slope
    const T im = g.inv_dm[k], ip = g.inv_dp[k], hp = g.hp[k], hm = g.hm[k];
    const bool lo = k > 0, hi = k < nr - 1;
    const T imp = hi ? g.inv_dm[k + 1] : (T)0, hpp = hi ? g.hp[k + 1] : (T)0, hmp = hi ? g.hm[k + 1] : (T)0;
    const T ipm = lo ? g.inv_dp[k - 1] : (T)0, hpm = lo ? g.hp[k - 1] : (T)0, hmm = lo ? g.hm[k - 1] : (T)0;
    T da[NV], db[NV], dbm[NV], dap[NV];
    slopes(0, k, j, i, da, db);
    if (lo) slopes(0, k - 1, j, i, none, dbm);
    if (hi) slopes(0, k + 1, j, i, dap, none);
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      const T* u = in.fr + v * nfr;             // u of the cell below face a: u[a cs + col]
      const T* l = in.fr + (NV + v) * nfr;      // l of the cell above it
      const T u0 = u[c + cs], l0 = l[c], ul = u[c], lu = l[c + cs];
      const T sb = hp * (hi ? u0 : (T)0) - hm * (lo ? l0 : (T)0);
      const T A = im * sb * da[v], B = ip * sb * db[v];
      T w = u0 + l0 + A - B;
      if (lo) {  // the plane below: its upper face is this cell's lower one
        const T s = hpm * ul - hmm * (k > 1 ? l[c - cs] : (T)0);
        w = fmat(ipm * s, dbm[v], w);
      }
      if (hi) {
        const T s = hpp * (k < nr - 2 ? u[c + 2 * cs] : (T)0) - hmp * lu;
        w = fmat(-(imp * s), dap[v], w);
      }
      wb[v] = w;
      gin[v] = ul - A;    // plane -1 (used at k = 0): L of face 0, plane 0's slope
      gout[v] = lu + B;   // plane nr (used at k = nr - 1)
    }
  }
  {  // theta: beyond a pole the neighbour is the opposite column's cell, whose
     // slope has this cell on the same side
    int io = i + np / 2;
    io = io >= np ? io - np : io;
    const int64_t f = ((int64_t)k * (nt + 1) + j) * np + i;   // lower face
    const int64_t fo = ((int64_t)k * (nt + 1) + j) * np + io;
    const bool south = j > 0, north = j < nt - 1;
    T da[NV], db[NV], dm[NV], dp[NV];
    slopes(1, k, j, i, da, db);
    if (south) slopes(1, k, j - 1, i, none, dm); else slopes(1, k, j, io, dm, none);
    if (north) slopes(1, k, j + 1, i, dp, none); else slopes(1, k, j, io, none, dp);
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      const T* u = in.ft + v * nft;
      const T* l = in.ft + (NV + v) * nft;
      const T u0 = u[f + np], l0 = l[f];
      const T sb = half * (u0 - l0);
      T w = wb[v] + (u0 + l0);
      w = fmat(sb, da[v] - db[v], w);
      w = fmat(south ? half * (u[f] - l[f - np]) : -half * (u[fo + np] - l[fo]), dm[v], w);
      w = fmat(north ? -half * (u[f + 2 * np] - l[f + np]) : half * (u[fo + np] - l[fo]), dp[v], w);
      wb[v] = w;
    }
  }
  {  // phi, periodic
    const int64_t row = c - i;
    const int64_t c1 = row + (i + 1 < np ? i + 1 : 0), c2 = row + (i + 2 < np ? i + 2 : i + 2 - np);
    const int64_t cm = row + (i > 0 ? i - 1 : np - 1);
    T da[NV], db[NV], dm[NV], dp[NV];
    slopes(2, k, j, i, da, db);
    slopes(2, k, j, (int)(cm - row), none, dm);
    slopes(2, k, j, (int)(c1 - row), dp, none);
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      const T* u = in.fp + v * nfp;
      const T* l = in.fp + (NV + v) * nfp;
      const T u0 = u[c1], l0 = l[c];
      const T sb = half * (u0 - l0);
      T w = wb[v] + (u0 + l0);
      w = fmat(sb, da[v] - db[v], w);
      w = fmat(half * (u[c] - l[cm]), dm[v], w);
      w = fmat(-half * (u[c2] - l[c1]), dp[v], w);
      wb[v] = w;
    }
  }
  // ---- ghosts
  T u[NV];
#pragma unroll
  for (int v = 0; v < NV; ++v) u[v] = U[v * N + c];
  if (k == 0) {
    const double ex = g.rhat[col], ey = g.rhat[cs + col], ez = g.rhat[2 * cs + col];
    if (ph.inner_bc == 1) {
      double brb[2];
      large_e_ghost_adjoint(Br[col], Br[cs + col], ex, ey, ez, ph, gin, wb, brb);
      if (Brb) { Brb[col] = brb[0]; Brb[cs + col] = brb[1]; }
    } else {
      T w[NV];
      recover(u, ph, w);
      const double brb = inner_ghost_adjoint(w, Br[col], ex, ey, ez, ph, gin, wb);
      if (Brb) Brb[col] = brb;
    }
  }
  if (k == nr - 1) outer_ghost_adjoint(g.rhat[col], g.rhat[cs + col], g.rhat[2 * cs + col], ph, gout, wb);
  // ---- recovery and gravity source
  T ub[NV];
  recover_adjoint(u, ph, wb, ub);
  const T gk = -g.grav[k];
  const T gx = gk * g.rhat[col], gy = gk * g.rhat[cs + col], gz = gk * g.rhat[2 * cs + col];
  // S_m = rho g, S_E = m . g
  ub[0] += Rb[1 * N + c] * gx + Rb[2 * N + c] * gy + Rb[3 * N + c] * gz;
  ub[1] += Rb[7 * N + c] * gx;
  ub[2] += Rb[7 * N + c] * gy;
  ub[3] += Rb[7 * N + c] * gz;
  ub[8] -= ph.psi_damp * Rb[8 * N + c];  // S_psi = -alpha psi
#pragma unroll
  for (int v = 0; v < NV; ++v) Ub[v * N + c] = ub[v];
}

}  // namespace crn
