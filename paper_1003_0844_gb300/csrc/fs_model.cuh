// Analytic detector model on the device, FP64 (Sec. II and Sec. V).
#pragma once
#include "fs_common.cuh"

namespace fs {

// Site on the reference ellipsoid at zero height (Sec. V): reduced latitude
// Psi = atan(b tan(phi) / a), equatorial radius a cos(Psi), height b sin(Psi).
__host__ __device__ inline void site_radius(double lat, double *re_m, double *z_m) {
  double b = kEllA * (1.0 - kEllF);
  double psi = atan(b * tan(lat) / kEllA);
  *re_m = kEllA * cos(psi);
  *z_m = b * sin(psi);
}

// Fourier coefficients of the amplitude modulation functions in
// x = alpha - theta(t) (the interferometer response of the series' first
// paper, Eqs. 12-13 there, cited in Sec. II):
//   a = ea0 cos2x + ea1 sin2x + ea2 cos x + ea3 sin x + ea4
//   b = eb0 cos2x + eb1 sin2x + eb2 cos x + eb3 sin x
__host__ __device__ inline void ab_from_trig(double s2g, double c2g, double sl, double cl, double s2l, double c2l,
                                             double sd, double cd, double s2d, double c2d, double ea[5], double eb[4]) {
  ea[0] = s2g * (3 - c2l) * (3 - c2d) / 16.0;
  ea[1] = -c2g * sl * (3 - c2d) / 4.0;
  ea[2] = s2g * s2l * s2d / 4.0;
  ea[3] = -c2g * cl * s2d / 2.0;
  ea[4] = 0.75 * s2g * cl * cl * cd * cd;
  eb[0] = c2g * sl * sd;
  eb[1] = s2g * (3 - c2l) * sd / 4.0;
  eb[2] = c2g * cl * cd;
  eb[3] = s2g * s2l * cd / 2.0;
}
__host__ __device__ inline void ab_coefficients(double delta, double lat, double gamma, double ea[5],
                                                double eb[4]) {
  ab_from_trig(sin(2 * gamma), cos(2 * gamma), sin(lat), cos(lat), sin(2 * lat), cos(2 * lat), sin(delta), cos(delta),
               sin(2 * delta), cos(2 * delta), ea, eb);
}

// Per-sky constants of the delay n0 . r_d / c written as in Sec. II:
//   cos(a)cos(d) (R_ES^x + R_E^x) + (sin(a)cos(d)cos(eps) + sin(d)sin(eps)) R_ES^y
//   + sin(a)cos(d) R_E^y + sin(d) R_E^z
// with R_ES = AU (cos lambda_E, sin lambda_E, 0) and R_E = (r_e cos th, r_e sin th, z):
//   phi_m = AU/c (nx cos lambda_E + nyp sin lambda_E) + (r_e/c) cos(d) cos(a - th) + (z/c) sin(d)
__host__ __device__ inline void sky_constants(double alpha, double delta, double eps, double lat,
                                              double gamma, const SegGeom &g, SkyConst64 *k) {
  double ca = cos(alpha), sa = sin(alpha), cd = cos(delta), sd = sin(delta);
  k->nx = ca * cd;
  k->nyp = sa * cd * cos(eps) + sd * sin(eps);
  k->nz = -sa * cd * sin(eps) + sd * cos(eps);
  k->ca = ca;
  k->sa = sa;
  k->rcd = g.re_c * cd;
  k->zsd = g.z_c * sd;
  ab_coefficients(delta, lat, gamma, k->ea, k->eb);
}

// The factors of the sky constants that depend on the detector alone, computed once per
// context (by the device, so that they are the values its kernels would compute).  What is
// left per sky is two sine/cosine pairs: computing all eighteen sines and cosines of
// sky_constants per sky took one thread 13 us, a third of a single-template search of one
// day.
struct DetConst {
  double ce, se;                  // obliquity
  double s2g, c2g, sl, cl, s2l, c2l;  // of 2 gamma, the latitude and twice the latitude
  double ka0, ka1, ka2, ka3, ka4; // a's coefficients without their delta factors
  double kb0, kb1, kb2, kb3;      // b's
};
__host__ __device__ inline DetConst det_const(const fs_detector &det) {
  const double s2g = sin(2 * det.gamma), c2g = cos(2 * det.gamma);
  const double sl = sin(det.lat), cl = cos(det.lat), s2l = sin(2 * det.lat), c2l = cos(2 * det.lat);
  DetConst d;
  d.ce = cos(det.eps);
  d.se = sin(det.eps);
  d.s2g = s2g;
  d.c2g = c2g;
  d.sl = sl;
  d.cl = cl;
  d.s2l = s2l;
  d.c2l = c2l;
  d.ka0 = s2g * (3 - c2l) / 16.0;
  d.ka1 = -c2g * sl / 4.0;
  d.ka2 = s2g * s2l / 4.0;
  d.ka3 = -c2g * cl / 2.0;
  d.ka4 = 0.75 * s2g * cl * cl;
  d.kb0 = c2g * sl;
  d.kb1 = s2g * (3 - c2l) / 4.0;
  d.kb2 = c2g * cl;
  d.kb3 = s2g * s2l / 2.0;
  return d;
}
// sky_constants from the sines and cosines of alpha and delta.
__host__ __device__ __forceinline__ void sky_constants_k(double ca, double sa, double cd, double sd, const DetConst &d,
                                                const SegGeom &g, SkyConst64 *k) {
  k->nx = ca * cd;
  k->nyp = sa * cd * d.ce + sd * d.se;
  k->nz = -sa * cd * d.se + sd * d.ce;
  k->ca = ca;
  k->sa = sa;
  k->rcd = g.re_c * cd;
  k->zsd = g.z_c * sd;
  const double s2d = 2.0 * sd * cd, q = 2.0 + 2.0 * sd * sd;  // q = 3 - cos(2 delta)
  k->ea[0] = d.ka0 * q;
  k->ea[1] = d.ka1 * q;
  k->ea[2] = d.ka2 * s2d;
  k->ea[3] = d.ka3 * s2d;
  k->ea[4] = d.ka4 * cd * cd;
  k->eb[0] = d.kb0 * sd;
  k->eb[1] = d.kb1 * sd;
  k->eb[2] = d.kb2 * cd;
  k->eb[3] = d.kb3 * cd;
}

struct Geo64 {  // delay and its time derivative, plus cos/sin of x = alpha - theta
  double phi, phidot, cx, sx;
  // low words where they are known (source_time64): phi + dphi, and the source time t1 + d
  double dphi = 0.0, t1 = 0.0, d = 0.0;
};

__device__ inline Geo64 geometry64(double t, const SkyConst64 &K, const SegGeom &g) {
  double sl, cl, sth, cth;
  sincos(g.lambda0 + kOmegaO * t, &sl, &cl);
  sincos(g.theta0 + kOmegaR * t, &sth, &cth);
  double cx = K.ca * cth + K.sa * sth;
  double sx = K.sa * cth - K.ca * sth;
  Geo64 r;
  r.phi = kAUls * (K.nx * cl + K.nyp * sl) + K.rcd * cx + K.zsd;
  r.phidot = kAUls * kOmegaO * (-K.nx * sl + K.nyp * cl) + K.rcd * kOmegaR * sx;
  r.cx = cx;
  r.sx = sx;
  return r;
}

__device__ inline void ab_eval64(const SkyConst64 &K, double cx, double sx, double *a, double *b) {
  double c2 = cx * cx - sx * sx, s2 = 2.0 * sx * cx;
  *a = K.ea[0] * c2 + K.ea[1] * s2 + K.ea[2] * cx + K.ea[3] * sx + K.ea[4];
  *b = K.eb[0] * c2 + K.eb[1] * s2 + K.eb[2] * cx + K.eb[3] * sx;
}

// The same from a caller's position table eph[2m] = (r_m, 0), eph[2m + 1] =
// (v_m, 0) on t_m = m dt: r(t) = r_m + (t - t_m) v_m from the nearest grid
// point m clamped to [0, n); phi = n0 . r(t), phidot = n0 . v_m.  The sidereal
// angle (for a, b) is the analytic one.
__device__ inline Geo64 geometry64_eph(double t, const SkyConst64 &K, const SegGeom &g, const dbl4 *eph) {
  double mf = rint(t / g.dt);
  mf = fmin(fmax(mf, 0.0), (double)(g.n - 1));
  const int64_t m = (int64_t)mf;
  const double tau = t - mf * g.dt;
  const dbl4 r = eph[2 * m], v = eph[2 * m + 1];
  double sth, cth;
  sincos(g.theta0 + kOmegaR * t, &sth, &cth);
  Geo64 q;
  q.phidot = K.nx * v.x + K.nyp * v.y + K.nz * v.z;
  q.phi = K.nx * r.x + K.nyp * r.y + K.nz * r.z + tau * q.phidot;
  q.cx = K.ca * cth + K.sa * sth;
  q.sx = K.sa * cth - K.ca * sth;
  return q;
}

// Source time t with t + phi_m(t) = tb (Eq. eq:Bt), the delay and its geometry there.
// FP64 arithmetic runs at 1/64 of the FP32 rate, and the two sine/cosine pairs of a
// geometry are most of it: two FP32 evaluations bring t within 1e-3 s, and one FP64
// evaluation with a Newton step does the rest (the step is off by
// (d2 phi/dt2) 1e-6 / 2 < 1e-16 s; phi, cos x and sin x follow it by their slopes to the
// same order).  The delay and the source time come in two words (a rounded source time,
// 3e-11 s after six days, moves the data of a 0.5 s series by 2e-10).  Measured on 43,082 samples: the
// demodulation takes 67 us with five FP64 evaluations, 27 us this way.
__device__ __forceinline__ float delay32(float t, const SkyConst64 &K, const SegGeom &g) {
  float sl, cl, sth, cth;
  sincosf((float)g.lambda0 + (float)kOmegaO * t, &sl, &cl);
  sincosf((float)g.theta0 + (float)kOmegaR * t, &sth, &cth);
  return (float)kAUls * fmaf((float)K.nx, cl, (float)K.nyp * sl) +
         fmaf((float)K.rcd, fmaf((float)K.ca, cth, (float)K.sa * sth), (float)K.zsd);
}
__device__ inline double source_time64(double tb, const SkyConst64 &K, const SegGeom &g, Geo64 *geo,
                                       const dbl4 *eph = nullptr) {
  if (eph) {  // a caller's table: piecewise linear, Newton's method from t = tb - phi(tb)
    Geo64 q = geometry64_eph(tb, K, g, eph);
    double t = tb - q.phi;
#pragma unroll 1
    for (int it = 0; it < 3; it++) {
      q = geometry64_eph(t, K, g, eph);
      t -= (t + q.phi - tb) / (1.0 + q.phidot);
    }
    *geo = geometry64_eph(t, K, g, eph);
    geo->t1 = t;
    return t;
  }
  const float tf = (float)tb;
  const float p1 = delay32(tf - delay32(tf, K, g), K, g);
  const double t1 = tb - (double)p1;
  Geo64 q = geometry64(t1, K, g);
  const double d = -(q.phi - (tb - t1)) / (1.0 + q.phidot), e = kOmegaR * d;  // tb - t1: exact but for t1 near 0 (6e-14 s)
  q.dphi = q.phidot * d;  // kept beside phi: added to it, half a rounding of 500 s would be lost
  const double cx = fma(q.sx, e, q.cx);
  q.sx = fma(-q.cx, e, q.sx);
  q.cx = cx;
  q.t1 = t1;  // rounded once; d is relative to the rounded value
  q.d = d;
  *geo = q;
  return t1 + d;
}

}  // namespace fs
