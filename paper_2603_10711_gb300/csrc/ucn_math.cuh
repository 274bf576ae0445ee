// Scalar types, dynamics models, RK4 and projections for the device path.
//
// The dynamics are written once over a scalar type S that is float, double
// or a forward-mode dual number Dual<T>; the Jacobians A_i, B_i of the RK4
// map (Sec. III-A, Eq. (2b)) are obtained by pushing one tangent direction
// at a time through the four RK4 stages.
#pragma once
#include <cuda_runtime.h>
#include <math.h>

#include <type_traits>

#include "ucn_df.cuh"

namespace ucn {

// ------------------------------------------------------------------ dual numbers
template <class T>
struct Dual {
  T v, d;
};

template <class S> struct BaseOf { typedef S type; };
template <class T> struct BaseOf<Dual<T>> { typedef T type; };

template <class T> __device__ __forceinline__ Dual<T> operator+(Dual<T> a, Dual<T> b) { return {a.v + b.v, a.d + b.d}; }
template <class T> __device__ __forceinline__ Dual<T> operator-(Dual<T> a, Dual<T> b) { return {a.v - b.v, a.d - b.d}; }
template <class T> __device__ __forceinline__ Dual<T> operator-(Dual<T> a) { return {-a.v, -a.d}; }
template <class T> __device__ __forceinline__ Dual<T> operator*(Dual<T> a, Dual<T> b) { return {a.v * b.v, a.d * b.v + a.v * b.d}; }
// a / b from b's correctly rounded reciprocal r: a r corrected by its exact residue
// is the correctly rounded quotient (Markstein 1990), at three instructions instead
// of a division's chain.
__device__ __forceinline__ double quot_(double a, double b, double r) {
  const double q = a * r;
  return fma(fma(-q, b, a), r, q);
}
__device__ __forceinline__ float quot_(float a, float b, float r) {
  const float q = a * r;
  return fmaf(fmaf(-q, b, a), r, q);
}
__device__ __forceinline__ DF quot_(DF a, DF, DF r) { return df_mul(a, r); }
// Duals divide through one reciprocal (the Jacobian passes' latency is the chain
// of divisions): FP32 by products with it, FP64 by correctly rounded quotients.
__device__ __forceinline__ Dual<float> operator/(Dual<float> a, Dual<float> b) {
  const float r = __frcp_rn(b.v), q = a.v * r;
  return {q, (a.d - q * b.d) * r};
}
__device__ __forceinline__ Dual<float> operator/(float a, Dual<float> b) {
  const float r = __frcp_rn(b.v), q = a * r;
  return {q, -q * b.d * r};
}
template <class T> __device__ __forceinline__ Dual<T> operator/(Dual<T> a, Dual<T> b) {
  const T r = T(1) / b.v, q = quot_(a.v, b.v, r);
  return {q, quot_(a.d - q * b.d, b.v, r)};
}
template <class T> __device__ __forceinline__ Dual<T> quot_(Dual<T> a, T b, T r) { return {quot_(a.v, b, r), quot_(a.d, b, r)}; }
template <class T> __device__ __forceinline__ Dual<T> operator+(Dual<T> a, T b) { return {a.v + b, a.d}; }
template <class T> __device__ __forceinline__ Dual<T> operator+(T b, Dual<T> a) { return {a.v + b, a.d}; }
template <class T> __device__ __forceinline__ Dual<T> operator-(Dual<T> a, T b) { return {a.v - b, a.d}; }
template <class T> __device__ __forceinline__ Dual<T> operator-(T b, Dual<T> a) { return {b - a.v, -a.d}; }
template <class T> __device__ __forceinline__ Dual<T> operator*(Dual<T> a, T b) { return {a.v * b, a.d * b}; }
template <class T> __device__ __forceinline__ Dual<T> operator*(T b, Dual<T> a) { return {a.v * b, a.d * b}; }
template <class T> __device__ __forceinline__ Dual<T> operator/(Dual<T> a, T b) { return {a.v / b, a.d / b}; }
template <class T> __device__ __forceinline__ Dual<T> operator/(T a, Dual<T> b) {
  const T r = T(1) / b.v, q = quot_(a, b.v, r);
  return {q, quot_(-q * b.d, b.v, r)};
}

// K tangent directions on one value (the Jacobian passes of the FP32 path): the
// value is computed once for all K; each tangent takes exactly the operations
// of Dual<T>, so the columns are those of K single-tangent passes.
template <class T, int K>
struct DualN {
  T v, d[K];
};
template <class T, int K> struct BaseOf<DualN<T, K>> { typedef T type; };
template <class T, int K> __device__ __forceinline__ DualN<T, K> operator+(DualN<T, K> a, DualN<T, K> b) {
  DualN<T, K> r;
  r.v = a.v + b.v;
#pragma unroll
  for (int q = 0; q < K; ++q) r.d[q] = a.d[q] + b.d[q];
  return r;
}
template <class T, int K> __device__ __forceinline__ DualN<T, K> operator-(DualN<T, K> a, DualN<T, K> b) {
  DualN<T, K> r;
  r.v = a.v - b.v;
#pragma unroll
  for (int q = 0; q < K; ++q) r.d[q] = a.d[q] - b.d[q];
  return r;
}
template <class T, int K> __device__ __forceinline__ DualN<T, K> operator-(DualN<T, K> a) {
  DualN<T, K> r;
  r.v = -a.v;
#pragma unroll
  for (int q = 0; q < K; ++q) r.d[q] = -a.d[q];
  return r;
}
template <class T, int K> __device__ __forceinline__ DualN<T, K> operator*(DualN<T, K> a, DualN<T, K> b) {
  DualN<T, K> r;
  r.v = a.v * b.v;
#pragma unroll
  for (int q = 0; q < K; ++q) r.d[q] = a.d[q] * b.v + a.v * b.d[q];
  return r;
}
template <class T, int K> __device__ __forceinline__ DualN<T, K> operator+(DualN<T, K> a, T b) { a.v = a.v + b; return a; }
template <class T, int K> __device__ __forceinline__ DualN<T, K> operator+(T b, DualN<T, K> a) { a.v = a.v + b; return a; }
template <class T, int K> __device__ __forceinline__ DualN<T, K> operator-(DualN<T, K> a, T b) { a.v = a.v - b; return a; }
template <class T, int K> __device__ __forceinline__ DualN<T, K> operator-(T b, DualN<T, K> a) {
  DualN<T, K> r;
  r.v = b - a.v;
#pragma unroll
  for (int q = 0; q < K; ++q) r.d[q] = -a.d[q];
  return r;
}
template <class T, int K> __device__ __forceinline__ DualN<T, K> operator*(DualN<T, K> a, T b) {
  DualN<T, K> r;
  r.v = a.v * b;
#pragma unroll
  for (int q = 0; q < K; ++q) r.d[q] = a.d[q] * b;
  return r;
}
template <class T, int K> __device__ __forceinline__ DualN<T, K> operator*(T b, DualN<T, K> a) { return a * b; }
template <class T, int K> __device__ __forceinline__ DualN<T, K> operator/(DualN<T, K> a, T b) {
  DualN<T, K> r;
  r.v = a.v / b;
#pragma unroll
  for (int q = 0; q < K; ++q) r.d[q] = a.d[q] / b;
  return r;
}

__device__ __forceinline__ float sqrt_(float a) { return sqrtf(a); }
__device__ __forceinline__ double sqrt_(double a) { return sqrt(a); }
// 1 / sqrt(a) of a Cholesky pivot: FP64 correctly rounded; FP32 by the hardware
// reciprocal square root and one Newton-Raphson step y (3 - a y^2) / 2 (within
// about one ulp; the factor feeds a refined solve), which replaces a rounded
// square root followed by a rounded divide on the factorisation's serial chain.
__device__ __forceinline__ double inv_sqrt_(double a) { return 1.0 / sqrt(a); }
__device__ __forceinline__ float inv_sqrt_(float a) {
  const float y = rsqrtf(a);
  return y * fmaf(-0.5f * a * y, y, 1.5f);
}
// Double-float: the root by one corrected step.
__device__ __forceinline__ DF sqrt_(DF a) { return df_sqrt(a); }
template <class T> __device__ __forceinline__ Dual<T> sqrt_(Dual<T> a) {
  T s = sqrt_(a.v);
  return {s, s > T(0) ? a.d / (T(2) * s) : T(0)};
}
// DualN as Dual per tangent (one reciprocal per division)
template <int K> __device__ __forceinline__ DualN<double, K> operator/(DualN<double, K> a, DualN<double, K> b) {
  const double rr = 1.0 / b.v;
  DualN<double, K> r;
  r.v = quot_(a.v, b.v, rr);
#pragma unroll
  for (int q = 0; q < K; ++q) r.d[q] = quot_(a.d[q] - r.v * b.d[q], b.v, rr);
  return r;
}
template <int K> __device__ __forceinline__ DualN<double, K> operator/(double a, DualN<double, K> b) {
  const double rr = 1.0 / b.v;
  DualN<double, K> r;
  r.v = quot_(a, b.v, rr);
#pragma unroll
  for (int q = 0; q < K; ++q) r.d[q] = quot_(-r.v * b.d[q], b.v, rr);
  return r;
}
template <class T, int K> __device__ __forceinline__ DualN<T, K> quot_(DualN<T, K> a, T b, T r) {
  DualN<T, K> c;
  c.v = quot_(a.v, b, r);
#pragma unroll
  for (int q = 0; q < K; ++q) c.d[q] = quot_(a.d[q], b, r);
  return c;
}
template <int K> __device__ __forceinline__ DualN<float, K> operator/(DualN<float, K> a, DualN<float, K> b) {
  const float rr = __frcp_rn(b.v);
  DualN<float, K> r;
  r.v = a.v * rr;
#pragma unroll
  for (int q = 0; q < K; ++q) r.d[q] = (a.d[q] - r.v * b.d[q]) * rr;
  return r;
}
template <int K> __device__ __forceinline__ DualN<float, K> operator/(float a, DualN<float, K> b) {
  const float rr = __frcp_rn(b.v);
  DualN<float, K> r;
  r.v = a * rr;
#pragma unroll
  for (int q = 0; q < K; ++q) r.d[q] = -r.v * b.d[q] * rr;
  return r;
}
template <class T, int K> __device__ __forceinline__ DualN<T, K> sqrt_(DualN<T, K> a) {
  DualN<T, K> r;
  r.v = sqrt_(a.v);
#pragma unroll
  for (int q = 0; q < K; ++q) r.d[q] = r.v > T(0) ? a.d[q] / (T(2) * r.v) : T(0);
  return r;
}

// Sine and cosine together: one range reduction for the two.
__device__ __forceinline__ void sincos_(float a, float& s, float& c) { sincosf(a, &s, &c); }
__device__ __forceinline__ void sincos_(double a, double& s, double& c) { sincos(a, &s, &c); }
__device__ __forceinline__ void sincos_(DF a, DF& s, DF& c) { df_sincos(a, s, c); }
template <class T> __device__ __forceinline__ void sincos_(Dual<T> a, Dual<T>& s, Dual<T>& c) {
  T sv, cv;
  sincos_(a.v, sv, cv);
  s = {sv, cv * a.d};
  c = {cv, -sv * a.d};
}
template <class T, int K> __device__ __forceinline__ void sincos_(DualN<T, K> a, DualN<T, K>& s, DualN<T, K>& c) {
  sincos_(a.v, s.v, c.v);
#pragma unroll
  for (int q = 0; q < K; ++q) {
    s.d[q] = c.v * a.d[q];
    c.d[q] = -s.v * a.d[q];
  }
}

// ------------------------------------------------------------------ models
// A model's constants as the dynamics read them: PRM values, the problem's
// eight (model_params) and reciprocals and differences of them, formed once per
// instance in FP64 (derived_param) and rounded to the arithmetic's type -- a
// division costs ~25 dependent FP64 instructions, or ~40 FP32 ones in double-float,
// and the RK4 map has nine of them at every stage of every tangent.
constexpr int PRM = 16;

// What an RK4 step holds constant: the control enters through a few combined
// quantities (Held), formed once per step; f is the dynamics given them.

// Quadrotor, 12 states (position, velocity, ZYX Euler angles phi/theta/psi,
// body rates), 4 rotor thrusts in a "+" layout.
// prm: m, Jx, Jy, Jz, arm, km (yaw moment per unit thrust), drag, g | 1/m, 1/Jx,
// 1/Jy, 1/Jz, drag/m, Jz-Jy, Jx-Jz, Jy-Jx.  The quotients by m and J are taken at
// every stage: one rounding of a held quotient would be the same in all four, and
// add up where four of their own average out.
struct Quad12 {
  static constexpr int NX = 12, NU = 4;
  __host__ __device__ static double derived(const double* p, int k) {
    const double m = p[0], Jx = p[1], Jy = p[2], Jz = p[3];
    switch (k) {
      case 8: return 1.0 / m;
      case 9: return 1.0 / Jx;
      case 10: return 1.0 / Jy;
      case 11: return 1.0 / Jz;
      case 12: return p[6] / m;
      case 13: return Jz - Jy;
      case 14: return Jx - Jz;
      default: return Jy - Jx;
    }
  }
  template <class S> struct Held { S F, tx, ty, tz; };
  template <class S, class P>
  __device__ static __forceinline__ Held<S> hold(const P* prm, const S* u) {
    typedef typename BaseOf<S>::type R;
    const R arm = (R)prm[4], km = (R)prm[5];
    Held<S> H;
    H.F = u[0] + u[1] + u[2] + u[3];
    H.tx = arm * (u[1] - u[3]);
    H.ty = arm * (u[2] - u[0]);
    H.tz = km * (u[0] - u[1] + u[2] - u[3]);
    return H;
  }
  template <class S, class P>
  __device__ static __forceinline__ void f(const P* prm, const S* x, const Held<S>& H, S* xd) {
    typedef typename BaseOf<S>::type R;
    const R m = (R)prm[0], rm = (R)prm[8], g = (R)prm[7], cdm = (R)prm[12];
    S sph, cph, sth, cth, sps, cps;
    sincos_(x[6], sph, cph);
    sincos_(x[7], sth, cth);
    sincos_(x[8], sps, cps);
    // third column of R = Rz(psi) Ry(theta) Rx(phi): the body thrust axis in the world frame
    const S cs = cph * sth;
    xd[0] = x[3];
    xd[1] = x[4];
    xd[2] = x[5];
    xd[3] = quot_((cs * cps + sph * sps) * H.F, m, rm) - cdm * x[3];
    xd[4] = quot_((cs * sps - sph * cps) * H.F, m, rm) - cdm * x[4];
    xd[5] = quot_((cph * cth) * H.F, m, rm) - g - cdm * x[5];
    const S wx = x[9], wy = x[10], wz = x[11];
    // Euler-angle rates from body rates (ZYX kinematics)
    const S w = (sph * wy + cph * wz) / cth;
    xd[6] = wx + sth * w;
    xd[7] = cph * wy - sph * wz;
    xd[8] = w;
    // rigid-body rotation: J w' = tau - w x (J w)
    xd[9] = quot_(H.tx - (R)prm[13] * wy * wz, (R)prm[1], (R)prm[9]);
    xd[10] = quot_(H.ty - (R)prm[14] * wz * wx, (R)prm[2], (R)prm[10]);
    xd[11] = quot_(H.tz - (R)prm[15] * wx * wy, (R)prm[3], (R)prm[11]);
  }
};

// Quadrotor, 13 states (position, velocity, quaternion body-to-world scalar
// first, body rates); control = total thrust along the body z axis and three
// body torques (Sec. IV-A1).  prm as Quad12 (arm and km unused).
struct Quat13 {
  static constexpr int NX = 13, NU = 4;
  __host__ __device__ static double derived(const double* p, int k) { return Quad12::derived(p, k); }
  template <class S> struct Held { S Tm, tx, ty, tz; };
  template <class S, class P>
  __device__ static __forceinline__ Held<S> hold(const P* prm, const S* u) {
    typedef typename BaseOf<S>::type R;
    Held<S> H;
    H.Tm = quot_(u[0], (R)prm[0], (R)prm[8]);
    H.tx = u[1];
    H.ty = u[2];
    H.tz = u[3];
    return H;
  }
  template <class S, class P>
  __device__ static __forceinline__ void f(const P* prm, const S* x, const Held<S>& H, S* xd) {
    typedef typename BaseOf<S>::type R;
    const R g = (R)prm[7], cdm = (R)prm[12];
    const S qw = x[6], qx = x[7], qy = x[8], qz = x[9];
    const S wx = x[10], wy = x[11], wz = x[12];
    // body z axis in the world frame, R(q) e3 (quadratic form, exact for unit q)
    const S a0 = R(2) * (qx * qz + qw * qy);
    const S a1 = R(2) * (qy * qz - qw * qx);
    const S a2 = qw * qw - qx * qx - qy * qy + qz * qz;
    xd[0] = x[3];
    xd[1] = x[4];
    xd[2] = x[5];
    xd[3] = a0 * H.Tm - cdm * x[3];
    xd[4] = a1 * H.Tm - cdm * x[4];
    xd[5] = a2 * H.Tm - g - cdm * x[5];
    // q' = q (x) (0, w) / 2
    xd[6] = R(0.5) * (-(qx * wx) - qy * wy - qz * wz);
    xd[7] = R(0.5) * (qw * wx + qy * wz - qz * wy);
    xd[8] = R(0.5) * (qw * wy - qx * wz + qz * wx);
    xd[9] = R(0.5) * (qw * wz + qx * wy - qy * wx);
    xd[10] = quot_(H.tx - (R)prm[13] * wy * wz, (R)prm[1], (R)prm[9]);
    xd[11] = quot_(H.ty - (R)prm[14] * wz * wx, (R)prm[2], (R)prm[10]);
    xd[12] = quot_(H.tz - (R)prm[15] * wx * wy, (R)prm[3], (R)prm[11]);
  }
};

// Mars powered descent, 7 states: position (Up-East-North), velocity, mass;
// control = thrust vector.  prm: g (acting along -Up), alpha (mass flow per
// unit thrust), non-dimensional units.
struct Mars7 {
  static constexpr int NX = 7, NU = 3;
  __host__ __device__ static double derived(const double*, int) { return 0.0; }
  // the mass rate -alpha |T| depends on the control alone
  template <class S> struct Held { S u0, u1, u2, mdot; };
  template <class S, class P>
  __device__ static __forceinline__ Held<S> hold(const P* prm, const S* u) {
    typedef typename BaseOf<S>::type R;
    const S Tn = sqrt_(u[0] * u[0] + u[1] * u[1] + u[2] * u[2]);
    return {u[0], u[1], u[2], -((R)prm[1] * Tn)};
  }
  template <class S, class P>
  __device__ static __forceinline__ void f(const P* prm, const S* x, const Held<S>& H, S* xd) {
    typedef typename BaseOf<S>::type R;
    const R g = (R)prm[0];
    const S im = R(1) / x[6];   // one division per evaluation (GB300's FP64 divide is costly)
    xd[0] = x[3];
    xd[1] = x[4];
    xd[2] = x[5];
    xd[3] = H.u0 * im - g;
    xd[4] = H.u1 * im;
    xd[5] = H.u2 * im;
    xd[6] = H.mdot;
  }
};

// Mars powered descent, 6-DOF, 14 states (Sec. IV-B1): mass, position
// (Up-East-North), velocity, quaternion body-to-world scalar first, body rates;
// control = thrust in the body frame (body x = thrust axis).  prm: alpha (mass
// flow per unit thrust), g (along -Up), Jx, Jy, Jz, l (the thrust acts at
// -l e_x in the body).  Non-dimensional units.  No Held: rk4h takes its stages as
// they stand here.
struct Mars14 {
  static constexpr int NX = 14, NU = 3;
  __host__ __device__ static double derived(const double*, int) { return 0.0; }
  template <class S, class P>
  __device__ static void f(const P* prm, const S* x, const S* u, S* xd) {
    typedef typename BaseOf<S>::type R;
    const R alpha = (R)prm[0], g = (R)prm[1], Jx = (R)prm[2], Jy = (R)prm[3], Jz = (R)prm[4], l = (R)prm[5];
    const S qw = x[7], qx = x[8], qy = x[9], qz = x[10];
    const S wx = x[11], wy = x[12], wz = x[13];
    const S Tn = sqrt_(u[0] * u[0] + u[1] * u[1] + u[2] * u[2]);
    const S im = R(1) / x[0];
    // rotation body -> world (quadratic form), applied to the body thrust
    const S c00 = qw * qw + qx * qx - qy * qy - qz * qz, c01 = R(2) * (qx * qy - qw * qz), c02 = R(2) * (qx * qz + qw * qy);
    const S c10 = R(2) * (qx * qy + qw * qz), c11 = qw * qw - qx * qx + qy * qy - qz * qz, c12 = R(2) * (qy * qz - qw * qx);
    const S c20 = R(2) * (qx * qz - qw * qy), c21 = R(2) * (qy * qz + qw * qx), c22 = qw * qw - qx * qx - qy * qy + qz * qz;
    xd[0] = -(alpha * Tn);
    xd[1] = x[4];
    xd[2] = x[5];
    xd[3] = x[6];
    xd[4] = (c00 * u[0] + c01 * u[1] + c02 * u[2]) * im - g;
    xd[5] = (c10 * u[0] + c11 * u[1] + c12 * u[2]) * im;
    xd[6] = (c20 * u[0] + c21 * u[1] + c22 * u[2]) * im;
    xd[7] = R(0.5) * (-(qx * wx) - qy * wy - qz * wz);
    xd[8] = R(0.5) * (qw * wx + qy * wz - qz * wy);
    xd[9] = R(0.5) * (qw * wy - qx * wz + qz * wx);
    xd[10] = R(0.5) * (qw * wz + qx * wy - qy * wx);
    // J w' = r_T x T - w x (J w), r_T = (-l, 0, 0): r_T x T = (0, l T_z, -l T_y)
    xd[11] = (-((Jz - Jy) * wy * wz)) / Jx;
    xd[12] = (l * u[2] - (Jx - Jz) * wz * wx) / Jy;
    xd[13] = (-(l * u[1]) - (Jy - Jx) * wx * wy) / Jz;
  }
};

// Entry k of a model's constants from the problem's eight.
template <class M>
__host__ __device__ inline double derived_param(const double* p, int k) {
  return k < 8 ? p[k] : M::derived(p, k);
}

// a + b c in the type of a and c (one fused pass for double-float).
template <class S, class R> __device__ __forceinline__ S fma_(S a, R b, S c) { return a + b * c; }
__device__ __forceinline__ DF fma_(DF a, DF b, DF c) { return df_fma(a, b, c); }

// Classical fourth-order Runge-Kutta step (Eq. (1b)) with the step h and its
// multiples h/2, h/6 given in the base type R of S.  The four stages are one
// loop: unrolled, a step of the larger models is 30 to 180 KB of code that runs
// once per SCP iteration, and the instruction fetch is what it waits for.  The
// 3-DOF Mars model's step is small outside double-float; rolled, its kernels
// spill in the ADMM loop.  The quaternion quadrotor's in FP64 waits for the FP64
// pipe instead, and a loop's frame costs its one-thread kernel more (152 of 50
// nodes, 4 x 100 iterations: 22.72 ms rolled, 22.16 straight).  The 6-DOF
// lander's stays straight-line with quotients and held terms in every stage: its
// FP32 solves meet decisions that a last bit turns (one batch of 1000 in sixteen:
// up to 5e-5 normwise), so their results are only as constant as this rounding.
template <class M, class S, class P, class R>
__device__ __forceinline__ void rk4h(const P* prm, R h, R hh, R h6, const S* x, const S* u, S* xn) {
  constexpr int NX = M::NX;
  S k[NX], t[NX], acc[NX];
  if constexpr (std::is_same<M, Mars14>::value) {
    M::f(prm, x, u, k);
#pragma unroll
    for (int j = 0; j < NX; ++j) { acc[j] = k[j]; t[j] = fma_(x[j], hh, k[j]); }
    M::f(prm, t, u, k);
#pragma unroll
    for (int j = 0; j < NX; ++j) { acc[j] = fma_(acc[j], R(2), k[j]); t[j] = fma_(x[j], hh, k[j]); }
    M::f(prm, t, u, k);
#pragma unroll
    for (int j = 0; j < NX; ++j) { acc[j] = fma_(acc[j], R(2), k[j]); t[j] = fma_(x[j], h, k[j]); }
    M::f(prm, t, u, k);
  } else {
  const typename M::template Held<S> H = M::template hold<S, P>(prm, u);
#pragma unroll
  for (int j = 0; j < NX; ++j) t[j] = x[j];
#pragma unroll ((M::NX == 7 && !std::is_same<S, DF>::value) || (M::NX == 13 && std::is_same<R, double>::value) ? 4 : 1)
  for (int s = 0; s < 4; ++s) {
    M::template f<S, P>(prm, t, H, k);
    if (s == 3) break;
    const R w = s == 2 ? h : hh;
    if (s == 0) {
#pragma unroll
      for (int j = 0; j < NX; ++j) acc[j] = k[j];
    } else {
#pragma unroll
      for (int j = 0; j < NX; ++j) acc[j] = fma_(acc[j], R(2), k[j]);
    }
#pragma unroll
    for (int j = 0; j < NX; ++j) t[j] = fma_(x[j], w, k[j]);
  }
  }
#pragma unroll
  for (int j = 0; j < NX; ++j) xn[j] = fma_(x[j], h6, acc[j] + k[j]);
}

template <class M, class S, class P>
__device__ __forceinline__ void rk4(const P* prm, double h_, const S* x, const S* u, S* xn) {
  typedef typename BaseOf<S>::type R;
  rk4h<M, S, P, R>(prm, (R)h_, (R)(0.5 * h_), (R)(h_ / 6.0), x, u, xn);
}

// The RK4 step h and its multiples h/2, h/6 in the arithmetic type R, rounded
// once from the FP64 step (the values rk4 forms on every call).
template <class R>
struct Step3 {
  R h, hh, h6;
};
template <class R>
__device__ __forceinline__ Step3<R> step_of(double h) {
  return {(R)h, (R)(0.5 * h), (R)(h / 6.0)};
}

// Column `dir` of [A B] = d RK4 / d(x, u) at (x, u), by one forward-mode pass.
template <class M, class T, class X, class P>
__device__ __forceinline__ void rk4_jvp(const P* prm, const Step3<T>& hs, const X* x, const X* u, int dir, T* col) {
  constexpr int NX = M::NX, NU = M::NU;
  Dual<T> xd[NX], ud[NU], out[NX];
#pragma unroll
  for (int j = 0; j < NX; ++j) xd[j] = {(T)x[j], (T)(dir == j ? 1 : 0)};
#pragma unroll
  for (int j = 0; j < NU; ++j) ud[j] = {(T)u[j], (T)(dir == NX + j ? 1 : 0)};
  rk4h<M, Dual<T>, P, T>(prm, hs.h, hs.hh, hs.h6, xd, ud, out);
#pragma unroll
  for (int j = 0; j < NX; ++j) col[j] = out[j].d;
}

// Columns dir0, dir0 + stride, ..., dir0 + (K - 1) stride of [A B] in one
// forward-mode pass (K tangents); cols[q] receives column dir0 + q stride.
template <class M, class T, int K, class X, class P>
__device__ __forceinline__ void rk4_jvpn(const P* prm, const Step3<T>& hs, const X* x, const X* u, int dir0, int stride,
                                         T (*cols)[M::NX]) {
  constexpr int NX = M::NX, NU = M::NU;
  DualN<T, K> xd[NX], ud[NU], out[NX];
#pragma unroll
  for (int j = 0; j < NX; ++j) {
    xd[j].v = (T)x[j];
#pragma unroll
    for (int q = 0; q < K; ++q) xd[j].d[q] = (T)(dir0 + q * stride == j ? 1 : 0);
  }
#pragma unroll
  for (int j = 0; j < NU; ++j) {
    ud[j].v = (T)u[j];
#pragma unroll
    for (int q = 0; q < K; ++q) ud[j].d[q] = (T)(dir0 + q * stride == NX + j ? 1 : 0);
  }
  rk4h<M, DualN<T, K>, P, T>(prm, hs.h, hs.hh, hs.h6, xd, ud, out);
#pragma unroll
  for (int j = 0; j < NX; ++j)
#pragma unroll
    for (int q = 0; q < K; ++q) cols[q][j] = out[j].d[q];
}

// ------------------------------------------------------------------ projections
// Ball {|y| <= R}: vector scaling, the test on squares: a node inside its set
// -- the most, so that whole warps skip -- takes no square root and no division
// (in FP64 some 55 instructions of a 1/64-rate pipe).  FP32: the scale from one
// reciprocal square root.
template <class T>
__device__ __forceinline__ void proj_ball3(T* y, T R) {
  if constexpr (std::is_same<T, float>::value) {
    const float n2 = y[0] * y[0] + y[1] * y[1] + y[2] * y[2];
    if (n2 > R * R) {
      const float s = R * rsqrtf(n2);
      y[0] *= s; y[1] *= s; y[2] *= s;
    }
  } else {
    const T n2 = y[0] * y[0] + y[1] * y[1] + y[2] * y[2];
    if (n2 > R * R) {
      const T s = R / sqrt_(n2);
      y[0] *= s; y[1] *= s; y[2] *= s;
    }
  }
}

// Lorentz cone {(t, y1, y2) : |y| <= tau t}, tau >= 0: inside -> unchanged;
// inside the polar cone (tau |y| <= -t) -> 0; otherwise onto the boundary ray.
// Both tests on squares; ca, sa the cosine and sine of the half-angle.
template <class T>
__device__ __forceinline__ void proj_cone3c(T* v, T tau, T ca, T sa) {
  const T t = v[0], s2 = v[1] * v[1] + v[2] * v[2], t2 = t * t, tau2 = tau * tau;
  if (t >= T(0) && s2 <= tau2 * t2) return;                                     // inside
  if (t <= T(0) && tau2 * s2 <= t2) { v[0] = v[1] = v[2] = T(0); return; }      // polar cone
  T s, r;   // s2 > 0 here
  if constexpr (std::is_same<T, float>::value) {
    const float rs = rsqrtf(s2);
    s = s2 * rs;
    r = (t * ca + s * sa) * sa * rs;
  } else {
    s = sqrt_(s2);
    r = (t * ca + s * sa) * sa / s;
  }
  v[0] = (t * ca + s * sa) * ca;
  v[1] *= r;
  v[2] *= r;
}

// The FP32 forms of both by selection instead of branches (the same numbers).
__device__ __forceinline__ void proj_ball3s(float* y, float R) {
  const float n2 = y[0] * y[0] + y[1] * y[1] + y[2] * y[2];
  const float s = n2 > R * R ? R * rsqrtf(n2) : 1.0f;
  y[0] *= s; y[1] *= s; y[2] *= s;
}
__device__ __forceinline__ void proj_cone3s(float* v, float tau, float ca, float sa) {
  const float t = v[0], s2 = v[1] * v[1] + v[2] * v[2], t2 = t * t, tau2 = tau * tau;
  const bool in = t >= 0.0f && s2 <= tau2 * t2, polar = t <= 0.0f && tau2 * s2 <= t2;
  const float rs = rsqrtf(s2), c = t * ca + s2 * rs * sa;   // (not used where s2 = 0: in or polar)
  v[0] = in ? t : polar ? 0.0f : c * ca;
  const float r = in ? 1.0f : polar ? 0.0f : c * sa * rs;
  v[1] *= r;
  v[2] *= r;
}

template <class T> __device__ __forceinline__ T clampv(T v, T lo, T hi) { return fmin(fmax(v, lo), hi); }
// max / |.| in the type of the arguments (never promoted to FP64 for floats)
__device__ __forceinline__ float maxv(float a, float b) { return fmaxf(a, b); }
__device__ __forceinline__ double maxv(double a, double b) { return fmax(a, b); }
__device__ __forceinline__ float absv(float a) { return fabsf(a); }
__device__ __forceinline__ double absv(double a) { return fabs(a); }
__device__ __forceinline__ float clampv(float v, float lo, float hi) { return fminf(fmaxf(v, lo), hi); }

// ------------------------------------------------------------------ warp reductions (FP64)
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ double warp_max(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

// ------------------------------------------------------------------ thread-block clusters
__device__ __forceinline__ unsigned cluster_size() {
  unsigned r;
  asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
  return r;
}
// Cluster barrier (release on arrive, acquire on wait); every thread of every
// CTA of the cluster executes the same sequence of them.
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
}
// A double from the shared memory of CTA `rank` of this cluster, at the
// address that `local` has in this CTA (distributed shared memory).
__device__ __forceinline__ double ld_cluster(const double* local, unsigned rank) {
  const unsigned a = (unsigned)__cvta_generic_to_shared(local);
  unsigned r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
  double v;
  asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(r) : "memory");
  return v;
}

// Stores to the same shared-memory location of another CTA of the cluster.
__device__ __forceinline__ unsigned cluster_addr(const void* local, unsigned rank) {
  unsigned r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"((unsigned)__cvta_generic_to_shared(local)), "r"(rank));
  return r;
}
__device__ __forceinline__ void st_cluster(const float* local, unsigned rank, float v) {
  asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(cluster_addr(local, rank)), "f"(v) : "memory");
}
__device__ __forceinline__ void st_cluster(const double* local, unsigned rank, double v) {
  asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(cluster_addr(local, rank)), "d"(v) : "memory");
}
__device__ __forceinline__ void st_cluster(const int* local, unsigned rank, int v) {
  asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(cluster_addr(local, rank)), "r"(v) : "memory");
}
__device__ __forceinline__ void st_cluster(const DF* local, unsigned rank, DF v) {
  st_cluster(&local->hi, rank, v.hi);
  st_cluster(&local->lo, rank, v.lo);
}

// Point-to-point exchange within a cluster: the receiver's mbarrier counts the
// bytes that its peers' asynchronous stores bring.  A phase completes when its
// owner has armed it (one arrival, `bytes` expected) and all have come, in either
// order.
__device__ __forceinline__ void tx_init(unsigned long long* bar) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"((unsigned)__cvta_generic_to_shared(bar)) : "memory");
}
__device__ __forceinline__ void tx_arm(unsigned long long* bar, unsigned bytes) {
  asm volatile("{\n .reg .b64 st;\n mbarrier.arrive.expect_tx.shared::cta.b64 st, [%0], %1;\n}" ::"r"(
                   (unsigned)__cvta_generic_to_shared(bar)), "r"(bytes) : "memory");
}
// Waits for the phase of this parity; false when it gave up (bounded).
__device__ __forceinline__ bool tx_wait(unsigned long long* bar, unsigned parity) {
  const unsigned a = (unsigned)__cvta_generic_to_shared(bar);
  for (int it = 0; it < (1 << 20); ++it) {
    unsigned done;
    asm volatile("{\n .reg .pred p;\n mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
                 : "=r"(done) : "r"(a), "r"(parity) : "memory");
    if (done) return true;
  }
  return false;
}
// v to the place of `local` in CTA `rank`, counted by its mbarrier at `bar`'s place.
__device__ __forceinline__ void st_async(const float* local, unsigned rank, float v, const unsigned long long* bar) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];" ::"r"(cluster_addr(local, rank)),
               "r"(__float_as_int(v)), "r"(cluster_addr(bar, rank)) : "memory");
}
__device__ __forceinline__ void st_async(const double* local, unsigned rank, double v, const unsigned long long* bar) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.b64 [%0], %1, [%2];" ::"r"(cluster_addr(local, rank)),
               "l"(__double_as_longlong(v)), "r"(cluster_addr(bar, rank)) : "memory");
}

__device__ __forceinline__ unsigned long long globaltimer_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

}  // namespace ucn
