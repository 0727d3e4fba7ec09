// Device-side building blocks of the TMOP element kernels (sm_103a).
//
//  * Dual<R>: forward-mode dual numbers. The Hessian action needs
//    d^2mu/dT^2 : dT (Section 3.4); evaluating the first derivative P(T) on
//    T + eps dT in dual arithmetic yields exactly that directional derivative
//    (mu302 and mu98 in the FP32 kernels; MetricLin, MetricAct and Metric302
//    write it out).
//  * metric_P: mu and P = dmu/dT for the Table 3.1 / Section 3.2 metrics in
//    the invariants I1 = |T|^2, tau = det T, C = cof T.
//  * fwd2/fwd3, adj2/adj3: sum-factorised tensor-product contractions of one
//    element, executed by one warp in shared memory. Forward: nodal values
//    X[c][l][j][i] -> A[c][b](q) = sum_i X_i d phi_i / d xi_b (eq. (2.2)).
//    Adjoint: per-point matrices R[c][b](q) -> Y[c][i] = sum_q R[c][b](q)
//    d phi_i / d xi_b (the transposed contraction of the gradient formula).
#pragma once
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "tmop_kparams.h"

namespace tmop {



// ---------------------------------------------------------------- scalars
template <class R>
struct Dual {
  R v, d;
};

template <class R> __device__ __forceinline__ Dual<R> operator+(Dual<R> a, Dual<R> b) { return {a.v + b.v, a.d + b.d}; }
template <class R> __device__ __forceinline__ Dual<R> operator-(Dual<R> a, Dual<R> b) { return {a.v - b.v, a.d - b.d}; }
template <class R> __device__ __forceinline__ Dual<R> operator-(Dual<R> a) { return {-a.v, -a.d}; }
template <class R> __device__ __forceinline__ Dual<R> operator*(Dual<R> a, Dual<R> b) {
  return {a.v * b.v, fma(a.v, b.d, a.d * b.v)};
}
template <class R> __device__ __forceinline__ Dual<R> operator*(R s, Dual<R> a) { return {s * a.v, s * a.d}; }
template <class R> __device__ __forceinline__ Dual<R> operator*(Dual<R> a, R s) { return {s * a.v, s * a.d}; }
template <class R> __device__ __forceinline__ Dual<R> operator+(Dual<R> a, R s) { return {a.v + s, a.d}; }
template <class R> __device__ __forceinline__ Dual<R> operator-(Dual<R> a, R s) { return {a.v - s, a.d}; }

__device__ __forceinline__ double value(double a) { return a; }
__device__ __forceinline__ float value(float a) { return a; }
template <class R> __device__ __forceinline__ R value(Dual<R> a) { return a.v; }

__device__ __forceinline__ double recip(double a) { return 1.0 / a; }
__device__ __forceinline__ float recip(float a) { return 1.0f / a; }
template <class R> __device__ __forceinline__ Dual<R> recip(Dual<R> a) {
  R r = R(1) / a.v;
  return {r, -a.d * r * r};
}
// tau^{-1/3}. In FP64 from the FP32 estimate y by one third-order step
// (the cube of the start's ~1e-7 relative error is below FP64 rounding: a
// few ulp) with 6 FP64 operations, on GB300's narrow FP64 pipe the cheaper
// route. Outside
// [2^-120, 2^120] (where the FP32 start would over- or underflow) and for
// non-finite input it defers to rcbrt.
__device__ __forceinline__ double rcbrt_nr(double a);
__device__ __forceinline__ double rcbrt_(double a) { return rcbrt_nr(a); }
__device__ __forceinline__ float rcbrt_(float a) { return rcbrtf(a); }
template <class R> __device__ __forceinline__ Dual<R> rcbrt_(Dual<R> a) {
  R r = rcbrt_(a.v);
  // d(tau^{-1/3}) = -(1/3) tau^{-4/3} dtau
  return {r, R(-1) / R(3) * r / a.v * a.d};
}

// Constants enter the metric formulas as plain reals, so that a dual number
// times a constant costs two multiplications, not a full dual product.
template <class S> struct base_of { using type = S; };
template <class R> struct base_of<Dual<R>> { using type = R; };
template <class S> __device__ __forceinline__ typename base_of<S>::type sc(double c) {
  return typename base_of<S>::type(c);
}

// ---------------------------------------------------------------- node numbering
// Global node ids of the nodes of an element. A structured order-(N-1) grid
// of sx x sy (x sz) elements is numbered lexicographically, x fastest, on a
// (k sx + 1) x (k sy + 1) (x (k sz + 1)) node lattice: the first node of
// element e is found once per element (the divisions by the run-time grid
// sizes are the costly part; GB300 runs their conversions on its narrow FP64
// pipe), and local node t = i + N j + N^2 l adds compile-time digits times
// the lattice strides. Unstructured meshes read the connectivity table.
// zplanes: lattice planes per element layer along the last index, N - 1 in
// 3D; in 2D, 1: a 2D "stack" of sz grids (elements e = ex + sx (ey + sy b),
// grid b's nodes after those of grids 0..b-1), so that many equal meshes
// form one structured problem.
template <int N>
struct NodeMap {
  const int32_t* conn;
  int sx, sy, Nx, NxNy, zplanes, base;
  const int32_t* row;
  __device__ __forceinline__ NodeMap(const int32_t* elem_nodes, int sx_, int sy_, int zplanes_ = N - 1)
      : conn(elem_nodes), sx(sx_), sy(sy_), Nx((N - 1) * sx_ + 1), NxNy(((N - 1) * sx_ + 1) * ((N - 1) * sy_ + 1)),
        zplanes(zplanes_), base(0), row(nullptr) {}
  __device__ __forceinline__ void element(int e, int ndof) {
    if (sx > 0) {
      const int exy = sx * sy, ez = e / exy, r = e - ez * exy, ey = r / sx, ex = r - ey * sx;
      base = ez * zplanes * NxNy + (N - 1) * (ey * Nx + ex);
    } else {
      row = conn + (size_t)e * ndof;
    }
  }
  __device__ __forceinline__ int operator()(int t) const {
    if (sx > 0) {
      const int i = t % N, j = (t / N) % N, l = t / (N * N);
      return base + l * NxNy + j * Nx + i;
    }
    return __ldg(row + t);
  }
};

// ---------------------------------------------------------------- precision conversions
// IEEE binary64 <-> binary32 with integer operations. The FP32 kernels
// convert every gathered FP64 value of v (and x) and every FP32 contribution
// they add into an FP64 output; done with F2F instructions these run on
// GB300's narrow FP64 pipe, here on the integer pipes. f64_to_f32 rounds to
// nearest even, as a cast does, except that results below the smallest
// normal float (|d| < 2^-126) become a signed zero; f32_to_f64 is exact, with
// subnormal inputs read as zero. Infinities and NaNs are kept.
__device__ __forceinline__ float f64_to_f32(double d) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(d);
  const unsigned hi = (unsigned)(b >> 32), lo = (unsigned)b;
  const unsigned sign = hi & 0x80000000u;
  const int e = (int)((hi >> 20) & 0x7FFu);
  if (e == 0x7FF) return __uint_as_float(sign | 0x7F800000u | (((hi & 0xFFFFFu) | lo) ? 0x400000u : 0u));
  const int fe = e - 1023 + 127;
  if (fe <= 0) return __uint_as_float(sign);
  unsigned m = ((hi & 0xFFFFFu) << 3) | (lo >> 29);   // the top 23 of the 52 mantissa bits
  const unsigned rem = lo & 0x1FFFFFFFu, half = 0x10000000u;
  m += (rem > half || (rem == half && (m & 1u))) ? 1u : 0u;
  unsigned r = ((unsigned)fe << 23) + m;              // a carry out of m steps the exponent
  if (fe >= 255 || r >= 0x7F800000u) r = 0x7F800000u;
  return __uint_as_float(sign | r);
}

__device__ __forceinline__ double f32_to_f64(float f) {
  const unsigned u = __float_as_uint(f);
  const unsigned sign = u & 0x80000000u, e = (u >> 23) & 0xFFu, m = u & 0x7FFFFFu;
  if (e == 0) return __longlong_as_double((long long)((unsigned long long)sign << 32));
  const unsigned hi = sign | (e == 0xFFu ? 0x7FF00000u : ((e + (1023u - 127u)) << 20)) | (m >> 3);
  const unsigned lo = m << 29;
  return __longlong_as_double((long long)(((unsigned long long)hi << 32) | lo));
}

__device__ __forceinline__ double rcbrt_nr(double a) {
  if (!(a >= 0x1p-120 && a <= 0x1p120)) return rcbrt(a);
  // one step of the series y (1 + e)^(-1/3) = y (1 - e/3 + 2 e^2 / 9 - ...)
  // with e = a y^3 - 1: the FP32 start has |e| < ~1e-6, so the dropped
  // O(e^3) term is far below FP64 rounding
  const double y = f32_to_f64(rcbrtf(f64_to_f32(a)));
  const double e = fma(a, y * y * y, -1.0);
  return fma(y, e * fma(e, 2.0 / 9.0, -1.0 / 3.0), y);
}

// FP64 value -> the kernel's arithmetic type, and back
template <class R> __device__ __forceinline__ R from_f64(double d) { return R(d); }
template <> __device__ __forceinline__ float from_f64<float>(double d) { return f64_to_f32(d); }
__device__ __forceinline__ double to_f64(double v) { return v; }
__device__ __forceinline__ double to_f64(float v) { return f32_to_f64(v); }

// ---------------------------------------------------------------- matrices
template <int D, class S>
__device__ __forceinline__ S det_m(const S* M) {
  if constexpr (D == 2) {
    return M[0] * M[3] - M[1] * M[2];
  } else {
    return M[0] * (M[4] * M[8] - M[5] * M[7]) - M[1] * (M[3] * M[8] - M[5] * M[6]) +
           M[2] * (M[3] * M[7] - M[4] * M[6]);
  }
}

// cof(M) = det(M) M^{-T}: the derivative of det M with respect to M
template <int D, class S>
__device__ __forceinline__ void cof_m(const S* M, S* C) {
  if constexpr (D == 2) {
    C[0] = M[3]; C[1] = -M[2]; C[2] = -M[1]; C[3] = M[0];
  } else {
    C[0] = M[4] * M[8] - M[5] * M[7];
    C[1] = M[5] * M[6] - M[3] * M[8];
    C[2] = M[3] * M[7] - M[4] * M[6];
    C[3] = M[2] * M[7] - M[1] * M[8];
    C[4] = M[0] * M[8] - M[2] * M[6];
    C[5] = M[1] * M[6] - M[0] * M[7];
    C[6] = M[1] * M[5] - M[2] * M[4];
    C[7] = M[2] * M[3] - M[0] * M[5];
    C[8] = M[0] * M[4] - M[1] * M[3];
  }
}

// ---------------------------------------------------------------- metrics
// mu(T) and P = dmu/dT. Returns false when a barrier metric meets
// tau <= 0 (mu is +inf there, P is left unset).
//
// metric_P(id, T, mu, P, s) returns s P instead (mu unscaled): the factor
// joins the one or two scalars P is built from, so the caller's weight
// w det W costs no multiply per entry of P.
template <int D, class S>
__device__ __forceinline__ bool metric_P(int id, const S* T, S& mu, S* P, typename base_of<S>::type s) {
  using B = typename base_of<S>::type;
  constexpr int DD = D * D;
  S I1 = T[0] * T[0];
#pragma unroll
  for (int i = 1; i < DD; ++i) I1 = I1 + T[i] * T[i];
  if (id == 1) {  // |T|^2
    mu = I1;
    const B c = sc<S>(2.0) * s;
#pragma unroll
    for (int i = 0; i < DD; ++i) P[i] = c * T[i];
    return true;
  }
  if (id == 14) {  // |T - I|^2
    const B c = sc<S>(2.0) * s;
    S e0 = T[0] - sc<S>(1.0);
    S acc = e0 * e0;
    P[0] = c * e0;
#pragma unroll
    for (int i = 1; i < DD; ++i) {
      S e = (i % (D + 1) == 0) ? T[i] - sc<S>(1.0) : T[i];
      acc = acc + e * e;
      P[i] = c * e;
    }
    mu = acc;
    return true;
  }
  // det T by expansion along the first row, from the cofactors P needs anyway
  S C[DD];
  cof_m<D>(T, C);
  S tau = T[0] * C[0];
#pragma unroll
  for (int j = 1; j < D; ++j) tau = tau + T[j] * C[j];
  if (!(value(tau) > 0)) return false;
  if (id == 98) {  // |T - I|^2 / tau (Section 4.3.2); P = (2 (T - I) - mu C) / tau
    S it = recip(tau);
    S E[DD];
#pragma unroll
    for (int i = 0; i < DD; ++i) E[i] = (i % (D + 1) == 0) ? T[i] - sc<S>(1.0) : T[i];
    S acc = E[0] * E[0];
#pragma unroll
    for (int i = 1; i < DD; ++i) acc = acc + E[i] * E[i];
    mu = acc * it;
    const S its = it * s;
#pragma unroll
    for (int i = 0; i < DD; ++i) P[i] = its * (sc<S>(2.0) * E[i] - mu * C[i]);
    return true;
  }
  if constexpr (D == 2) {
    S it = recip(tau);
    if (id == 2) {  // |T|^2 / (2 tau) - 1
      mu = sc<S>(0.5) * I1 * it - sc<S>(1.0);
      S a = it * s, b = (sc<S>(0.5) * s) * I1 * it * it;
#pragma unroll
      for (int i = 0; i < 4; ++i) P[i] = a * T[i] - b * C[i];
      return true;
    }
    S it2 = it * it;
    if (id == 7) {  // |T - T^-t|^2 = I1 (1 + tau^-2) - 4
      mu = I1 * (it2 + sc<S>(1.0)) - sc<S>(4.0);
      S a = (sc<S>(2.0) * s) * (it2 + sc<S>(1.0)), b = (sc<S>(2.0) * s) * I1 * it2 * it;
#pragma unroll
      for (int i = 0; i < 4; ++i) P[i] = a * T[i] - b * C[i];
      return true;
    }
    if (id == 9) {  // tau |T - T^-t|^2 = tau I1 + I1 / tau - 4 tau
      mu = tau * I1 + I1 * it - sc<S>(4.0) * tau;
      S a = (sc<S>(2.0) * s) * (tau + it), b = (I1 - I1 * it2 - sc<S>(4.0)) * s;
#pragma unroll
      for (int i = 0; i < 4; ++i) P[i] = a * T[i] + b * C[i];
      return true;
    }
    if (id == 77) {  // (tau - 1/tau)^2 / 2
      S d = tau - it;
      mu = sc<S>(0.5) * d * d;
      S a = d * (it2 + sc<S>(1.0)) * s;
#pragma unroll
      for (int i = 0; i < 4; ++i) P[i] = a * C[i];
      return true;
    }
  } else {
    if (id == 303) {  // |T|^2 / (3 tau^{2/3}) - 1; 1 / tau = (tau^{-1/3})^3, no division
      S r = rcbrt_(tau);
      S r2 = r * r;
      S it = r2 * r;
      mu = sc<S>(1.0 / 3.0) * I1 * r2 - sc<S>(1.0);
      S a = (sc<S>(2.0 / 3.0) * s) * r2, b = a * ((sc<S>(1.0 / 3.0) * I1) * it);   // b = 2/9 s I1 r^5
#pragma unroll
      for (int i = 0; i < 9; ++i) P[i] = a * T[i] - b * C[i];
      return true;
    }
    if (id == 302) {  // |T|^2 |T^-1|^2 / 9 - 1 = I1 K / (9 tau^2) - 1, K = |cof T|^2
      S it = recip(tau);
      S K = C[0] * C[0];
#pragma unroll
      for (int i = 1; i < 9; ++i) K = K + C[i] * C[i];
      // dK/dT = 2 (I1 T - T T^t T)
      S TtT[9];
#pragma unroll
      for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) TtT[i * 3 + j] = T[i] * T[j] + T[3 + i] * T[3 + j] + T[6 + i] * T[6 + j];
      S a = sc<S>(1.0 / 9.0) * it * it;
      mu = a * I1 * K - sc<S>(1.0);
      S c = sc<S>(2.0) * a * I1 * K * it;
      S as = a * s, cs = c * s;
#pragma unroll
      for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) {
          S M = T[i * 3 + 0] * TtT[0 * 3 + j] + T[i * 3 + 1] * TtT[1 * 3 + j] + T[i * 3 + 2] * TtT[2 * 3 + j];
          S Kp = sc<S>(2.0) * (I1 * T[i * 3 + j] - M);
          P[i * 3 + j] = as * (I1 * Kp + sc<S>(2.0) * K * T[i * 3 + j]) - cs * C[i * 3 + j];
        }
      return true;
    }
  }
  return false;
}

template <int D, class S>
__device__ __forceinline__ bool metric_P(int id, const S* T, S& mu, S* P) {
  return metric_P<D, S>(id, T, mu, P, typename base_of<S>::type(1));
}

// ---------------------------------------------------------------- linearised metric
// For metrics written in I1 = |T|^2 (mu98: |T - I|^2, with X = T - I for T
// in P and in the first and second term of dP) and tau = det T (all but mu302), the
// first derivative is P = 2 mu_1 T + mu_t C and, with dI1 = 2 T:dT and
// dtau = C:dT (C = cof T, the derivative of det),
//   dP = 2 mu_1 dT + 2 (mu_11 dI1 + mu_1t dtau) T + (mu_1t dI1 + mu_tt dtau) C + mu_t dC,
// where dC is the directional derivative of the cofactor matrix (product rule
// on its 2x2 minors in 3D; linear in 2D). MetricLin holds everything that
// depends on T only, so one point can be differentiated in many directions.
template <int D, class R>
struct MetricLin {
  static constexpr int DD = D * D;
  R T[DD], C[DD];
  R X[D];   // diagonal of the matrix I1 is the norm of: T, or T - I (mu98)
  R m1, mt, m11, m1t, mtt;
  bool ok;

  __device__ __forceinline__ R x(int i) const { return i % (D + 1) == 0 ? X[i / (D + 1)] : T[i]; }

  __device__ __forceinline__ bool init(int id, const R* Tin) {
#pragma unroll
    for (int i = 0; i < DD; ++i) T[i] = Tin[i];
#pragma unroll
    for (int d = 0; d < D; ++d) X[d] = T[d * (D + 1)];
    if (sizeof(R) == 8 && id == 98) {
#pragma unroll
      for (int d = 0; d < D; ++d) X[d] -= R(1);
    }
    R I1 = R(0);
#pragma unroll
    for (int i = 0; i < DD; ++i) I1 = fma(x(i), x(i), I1);
    cof_m<D>(T, C);
    R tau = R(0);
#pragma unroll
    for (int j = 0; j < D; ++j) tau = fma(T[j], C[j], tau);   // expansion along the first row
    m1 = R(0); mt = R(0); m11 = R(0); m1t = R(0); mtt = R(0);
    if (id == 1 || id == 14) { m1 = R(1); ok = true; return true; }
    ok = tau > R(0);
    if (!ok) return false;
    if (id == 303) {          // I1 tau^{-2/3} / 3 - 1 (3D); 1 / tau = (tau^{-1/3})^3, no division
      const R r = rcbrt_(tau), r2 = r * r, it = r2 * r, t53 = r2 * it;
      m1 = r2 * R(1.0 / 3.0); mt = R(-2.0 / 9.0) * I1 * t53; m1t = R(-2.0 / 9.0) * t53;
      mtt = R(10.0 / 27.0) * I1 * t53 * it;
      return ok;
    }
    const R it = R(1) / tau, it2 = it * it;
    if (id == 2) {            // I1 / (2 tau) - 1
      m1 = R(0.5) * it; mt = R(-0.5) * I1 * it2; m1t = R(-0.5) * it2; mtt = I1 * it2 * it;
    } else if (id == 7) {     // I1 (1 + tau^-2) - 4 (2D)
      m1 = R(1) + it2; mt = R(-2) * I1 * it2 * it; m1t = R(-2) * it2 * it; mtt = R(6) * I1 * it2 * it2;
    } else if (id == 9) {     // tau I1 + I1 / tau - 4 tau (2D)
      m1 = tau + it; mt = I1 - I1 * it2 - R(4); m1t = R(1) - it2; mtt = R(2) * I1 * it2 * it;
    } else if (sizeof(R) == 8 && id == 98) {    // |T - I|^2 / tau = I1 / tau with I1 = |T - I|^2
      m1 = it; mt = -I1 * it2; m1t = -it2; mtt = R(2) * I1 * it2 * it;
    } else if (id == 77) {    // (tau - 1/tau)^2 / 2
      const R sdiff = tau - it, ds = R(1) + it2;
      mt = sdiff * ds; mtt = ds * ds - R(2) * sdiff * it2 * it;
    } else {
      ok = false;
    }
    return ok;
  }

  // dP for one direction dT
  __device__ __forceinline__ void dP(const R* dT, R* out) const {
    R dI1 = R(0), dtau = R(0);
#pragma unroll
    for (int i = 0; i < DD; ++i) {
      dI1 = fma(x(i), dT[i], dI1);
      dtau = fma(C[i], dT[i], dtau);
    }
    dI1 *= R(2);
    const R a = R(2) * m1;
    const R bT = R(2) * (m11 * dI1 + m1t * dtau);
    const R bC = m1t * dI1 + mtt * dtau;
    R mdC[DD];  // mu_t dC
    if constexpr (D == 2) {
      mdC[0] = mt * dT[3]; mdC[1] = -mt * dT[2]; mdC[2] = -mt * dT[1]; mdC[3] = mt * dT[0];
    } else {
      // each entry of dC is the derivative of a 2x2 minor, dT_a T_b + T_a dT_b
      // - dT_c T_e - T_c dT_e; with U = mu_t T the factor mu_t costs no
      // multiply per entry
      R U[DD];
#pragma unroll
      for (int i = 0; i < DD; ++i) U[i] = mt * T[i];
#define TMOP_DMINOR(a_, b_, c_, e_) fma(dT[a_], U[b_], fma(U[a_], dT[b_], -fma(dT[c_], U[e_], U[c_] * dT[e_])))
      mdC[0] = TMOP_DMINOR(4, 8, 5, 7);
      mdC[1] = TMOP_DMINOR(5, 6, 3, 8);
      mdC[2] = TMOP_DMINOR(3, 7, 4, 6);
      mdC[3] = TMOP_DMINOR(2, 7, 1, 8);
      mdC[4] = TMOP_DMINOR(0, 8, 2, 6);
      mdC[5] = TMOP_DMINOR(1, 6, 0, 7);
      mdC[6] = TMOP_DMINOR(1, 5, 2, 4);
      mdC[7] = TMOP_DMINOR(2, 3, 0, 5);
      mdC[8] = TMOP_DMINOR(0, 4, 1, 3);
#undef TMOP_DMINOR
    }
#pragma unroll
    for (int i = 0; i < DD; ++i) out[i] = fma(a, dT[i], fma(bT, x(i), fma(bC, C[i], mdC[i])));
  }
};

// The same second derivative for a matrix-free Hessian action, with the
// point's weight s = w det W and the constant factors folded into five
// coefficients when T is set, so that dP costs ~10 multiplies fewer per
// point (GB300 issues only two FP64 operations per SM and clock):
//   s dP = cA dT + (c11 t + c1t d) T + (c1t t + ctt d) C + s mu_t dC,
// with t = T:dT, d = C:dT, cA = 2 s mu_1, c11 = 4 s mu_11, c1t = 2 s mu_1t,
// ctt = s mu_tt.
template <int D, class R>
struct MetricAct {
  static constexpr int DD = D * D;
  R T[DD], C[DD];
  R X[D];   // as MetricLin's
  R cA, c11, c1t, ctt, ct;

  __device__ __forceinline__ R x(int i) const { return i % (D + 1) == 0 ? X[i / (D + 1)] : T[i]; }

  __device__ __forceinline__ bool init(int id, const R* Tin, R s) {
    if constexpr (D == 3) {
      if (id == 303) {  // I1 tau^{-2/3} / 3 - 1: mu_11 = 0
#pragma unroll
        for (int i = 0; i < DD; ++i) T[i] = Tin[i];
#pragma unroll
        for (int d = 0; d < D; ++d) X[d] = T[d * (D + 1)];
        R I1 = R(0);
#pragma unroll
        for (int i = 0; i < DD; ++i) I1 = fma(T[i], T[i], I1);
        cof_m<D>(T, C);
        R tau = R(0);
#pragma unroll
        for (int j = 0; j < D; ++j) tau = fma(T[j], C[j], tau);
        if (!(tau > R(0))) return false;
        // mu_1 = r^2 / 3, mu_1t = -2/9 r^5 = -2/3 mu_1 r^3, mu_t = I1 mu_1t,
        // mu_tt = -5/3 mu_t r^3 (r = tau^{-1/3})
        const R r = rcbrt_(tau), r2 = r * r, it = r2 * r;
        cA = (R(2.0 / 3.0) * s) * r2;
        c11 = R(0);
        c1t = cA * (R(-2.0 / 3.0) * it);
        ct = c1t * (R(0.5) * I1);
        ctt = (ct * it) * R(-5.0 / 3.0);
        return true;
      }
    }
    MetricLin<D, R> L;
    if (!L.init(id, Tin)) return false;
#pragma unroll
    for (int i = 0; i < DD; ++i) {
      T[i] = L.T[i];
      C[i] = L.C[i];
    }
#pragma unroll
    for (int d = 0; d < D; ++d) X[d] = L.X[d];
    const R s2 = R(2) * s;
    cA = s2 * L.m1;
    c11 = (R(2) * s2) * L.m11;
    c1t = s2 * L.m1t;
    ctt = s * L.mtt;
    ct = s * L.mt;
    return true;
  }

  __device__ __forceinline__ void dP(const R* dT, R* out) const {
    R t = R(0), d = R(0);
#pragma unroll
    for (int i = 0; i < DD; ++i) {
      t = fma(x(i), dT[i], t);
      d = fma(C[i], dT[i], d);
    }
    const R bT = fma(c11, t, c1t * d);
    const R bC = fma(c1t, t, ctt * d);
    R mdC[DD];  // s mu_t dC
    if constexpr (D == 2) {
      mdC[0] = ct * dT[3]; mdC[1] = -ct * dT[2]; mdC[2] = -ct * dT[1]; mdC[3] = ct * dT[0];
    } else {
      R U[DD];
#pragma unroll
      for (int i = 0; i < DD; ++i) U[i] = ct * T[i];
#define TMOP_DMINOR(a_, b_, c_, e_) fma(dT[a_], U[b_], fma(U[a_], dT[b_], -fma(dT[c_], U[e_], U[c_] * dT[e_])))
      mdC[0] = TMOP_DMINOR(4, 8, 5, 7);
      mdC[1] = TMOP_DMINOR(5, 6, 3, 8);
      mdC[2] = TMOP_DMINOR(3, 7, 4, 6);
      mdC[3] = TMOP_DMINOR(2, 7, 1, 8);
      mdC[4] = TMOP_DMINOR(0, 8, 2, 6);
      mdC[5] = TMOP_DMINOR(1, 6, 0, 7);
      mdC[6] = TMOP_DMINOR(1, 5, 2, 4);
      mdC[7] = TMOP_DMINOR(2, 3, 0, 5);
      mdC[8] = TMOP_DMINOR(0, 4, 1, 3);
#undef TMOP_DMINOR
    }
#pragma unroll
    for (int i = 0; i < DD; ++i) out[i] = fma(cA, dT[i], fma(bT, x(i), fma(bC, C[i], mdC[i])));
  }
};

// mu302 = I1 K / (9 tau^2) - 1 (3D), K = |C|^2, C = cof T: with the
// symmetric bilinear form cof'(A)[B] (the derivative of the cofactor matrix at A
// in direction B) dK/dT = 2 N, N = cof'(T)[C], and
//   P = a T + b N - c C,  a = 2 K / (9 tau^2), b = 2 I1 / (9 tau^2), c = 2 I1 K / (9 tau^3),
//   dP = a dT + b dN - c dC + da T + db N - dc C,
//   dC = cof'(T)[dT], dN = cof'(dT)[C] + cof'(T)[dC].
// s scales P and dP.
template <class R>
struct Metric302 {
  R T[9], C[9], N[9], I1, K, it, a, b, c, f;

  // out += cof'(A)[B]
  static __device__ __forceinline__ void dcof(const R* A, const R* B, R* out) {
#pragma unroll
    for (int i = 0; i < 9; ++i) {
      const int r1 = 3 * ((i / 3 + 1) % 3), r2 = 3 * ((i / 3 + 2) % 3), c1 = (i % 3 + 1) % 3, c2 = (i % 3 + 2) % 3;
      out[i] = fma(A[r1 + c1], B[r2 + c2], out[i]);
      out[i] = fma(B[r1 + c1], A[r2 + c2], out[i]);
      out[i] = fma(-A[r1 + c2], B[r2 + c1], out[i]);
      out[i] = fma(-B[r1 + c2], A[r2 + c1], out[i]);
    }
  }
  __device__ __forceinline__ bool init(const R* Tin, R s) {
    I1 = R(0);
    K = R(0);
    R tau = R(0);
#pragma unroll
    for (int i = 0; i < 9; ++i) {
      T[i] = Tin[i];
      N[i] = R(0);
    }
    cof_m<3>(T, C);
#pragma unroll
    for (int i = 0; i < 9; ++i) {
      I1 = fma(T[i], T[i], I1);
      K = fma(C[i], C[i], K);
      if (i < 3) tau = fma(T[i], C[i], tau);
    }
    if (!(tau > R(0))) return false;
    dcof(T, C, N);
    it = R(1) / tau;
    f = R(2.0 / 9.0) * s * it * it;
    a = f * K;
    b = f * I1;
    c = a * I1 * it;
    return true;
  }
  __device__ __forceinline__ R P(int i) const { return fma(a, T[i], fma(b, N[i], -c * C[i])); }
  __device__ __forceinline__ void dP(const R* dT, R* out) const {
    R t = R(0), n = R(0), d = R(0);   // dI1 / 2, dK / 2, dtau
    R dC[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) {
      t = fma(T[i], dT[i], t);
      n = fma(N[i], dT[i], n);
      d = fma(C[i], dT[i], d);
      dC[i] = R(0);
      out[i] = R(0);
    }
    const R dt = R(2) * it * d;   // 2 dtau / tau
    const R da = fma(R(2) * f, n, -a * dt), db = fma(R(2) * f, t, -b * dt);
    const R dc = it * fma(R(2), fma(a, t, b * n), -R(3) * c * d);
    dcof(T, dT, dC);
    dcof(dT, C, out);
    dcof(T, dC, out);
#pragma unroll
    for (int i = 0; i < 9; ++i)
      out[i] = fma(b, out[i], fma(a, dT[i], fma(-c, dC[i], fma(da, T[i], fma(db, N[i], -dc * C[i])))));
  }
};

// ---------------------------------------------------------------- contractions
// Tables in shared memory: B[q][i] = phi_i(xi_q), G[q][i] = phi_i'(xi_q).

// 2D forward. P0: X[NC][N][N] -> (P1: S[NC][2][N][Q]) -> P0: A[NC][2][Q][Q]
template <int N, int Q1, int NC, class R>
__device__ __forceinline__ void fwd2(const R* __restrict__ B, const R* __restrict__ G, R* P0, R* P1, int lane) {
  for (int t = lane; t < NC * N * Q1; t += 32) {
    const int q0 = t % Q1, j = (t / Q1) % N, c = t / (Q1 * N);
    const R* xr = P0 + (c * N + j) * N;
    R sb = R(0), sg = R(0);
#pragma unroll
    for (int i = 0; i < N; ++i) {
      const R xv = xr[i];
      sb = fma(xv, B[q0 * N + i], sb);
      sg = fma(xv, G[q0 * N + i], sg);
    }
    P1[((c * 2 + 0) * N + j) * Q1 + q0] = sb;
    P1[((c * 2 + 1) * N + j) * Q1 + q0] = sg;
  }
  __syncwarp();
  for (int t = lane; t < NC * Q1 * Q1; t += 32) {
    const int q0 = t % Q1, q1 = (t / Q1) % Q1, c = t / (Q1 * Q1);
    const R* sB = P1 + (c * 2 + 0) * N * Q1 + q0;
    const R* sG = P1 + (c * 2 + 1) * N * Q1 + q0;
    R a0 = R(0), a1 = R(0);
#pragma unroll
    for (int j = 0; j < N; ++j) {
      a0 = fma(sG[j * Q1], B[q1 * N + j], a0);  // d/dxi_0: G in x, B in y
      a1 = fma(sB[j * Q1], G[q1 * N + j], a1);  // d/dxi_1: B in x, G in y
    }
    P0[(c * 2 + 0) * Q1 * Q1 + q1 * Q1 + q0] = a0;
    P0[(c * 2 + 1) * Q1 * Q1 + q1 * Q1 + q0] = a1;
  }
  __syncwarp();
}

// 2D adjoint. P0: R[NC][2][Q][Q] -> (P1: U[NC][2][N][Q]) -> P0: Y[NC][N][N]
template <int N, int Q1, int NC, class R>
__device__ __forceinline__ void adj2(const R* __restrict__ B, const R* __restrict__ G, R* P0, R* P1, int lane) {
  for (int t = lane; t < NC * N * Q1; t += 32) {
    const int q0 = t % Q1, j = (t / Q1) % N, c = t / (Q1 * N);
    const R* r0 = P0 + (c * 2 + 0) * Q1 * Q1 + q0;
    const R* r1 = P0 + (c * 2 + 1) * Q1 * Q1 + q0;
    R u0 = R(0), u1 = R(0);
#pragma unroll
    for (int q1 = 0; q1 < Q1; ++q1) {
      u0 = fma(r0[q1 * Q1], B[q1 * N + j], u0);
      u1 = fma(r1[q1 * Q1], G[q1 * N + j], u1);
    }
    P1[((c * 2 + 0) * N + j) * Q1 + q0] = u0;  // pairs with G in x
    P1[((c * 2 + 1) * N + j) * Q1 + q0] = u1;  // pairs with B in x
  }
  __syncwarp();
  for (int t = lane; t < NC * N * N; t += 32) {
    const int i = t % N, j = (t / N) % N, c = t / (N * N);
    const R* u0 = P1 + ((c * 2 + 0) * N + j) * Q1;
    const R* u1 = P1 + ((c * 2 + 1) * N + j) * Q1;
    R y = R(0);
#pragma unroll
    for (int q0 = 0; q0 < Q1; ++q0) y = fma(u0[q0], G[q0 * N + i], fma(u1[q0], B[q0 * N + i], y));
    P0[(c * N + j) * N + i] = y;
  }
  __syncwarp();
}

// ---------------------------------------------------------------- register-blocked 3D contractions
// Same maps as fwd3/adj3 with the same buffer layouts, but each lane owns a
// whole row of outputs: it loads the row's inputs once into registers and
// takes the 1D tables from registers (tB/tG: [Q1][N], compile-time indexed),
// so a stage issues ~4x fewer shared-memory instructions. Used by the FP32
// kernels, whose throughput the shared-memory pipe otherwise bounds. Each
// loop over lanes runs its compile-time number of passes, so the index
// arithmetic folds into straight-line code.
template <int N, int Q1, int NC, class R>
__device__ __forceinline__ void fwd3_rb(const R (&tB)[Q1 * N], const R (&tG)[Q1 * N], R* P0, R* P1, int lane) {
  constexpr int NNQ = N * N * Q1, NQQ = N * Q1 * Q1, QQ = Q1 * Q1, QQQ = Q1 * Q1 * Q1;
  #pragma unroll
  for (int k = 0; k < (NC * N * N + 31) / 32; ++k) {           // (c, l, j) rows of x
    const int t = lane + 32 * k;
    if (t >= NC * N * N) break;
    const int c = t / (N * N), lj = t % (N * N);
    R xv[N];
#pragma unroll
    for (int i = 0; i < N; ++i) xv[i] = P0[t * N + i];
#pragma unroll
    for (int q0 = 0; q0 < Q1; ++q0) {
      R sb = R(0), sg = R(0);
#pragma unroll
      for (int i = 0; i < N; ++i) {
        sb = fma(xv[i], tB[q0 * N + i], sb);
        sg = fma(xv[i], tG[q0 * N + i], sg);
      }
      P1[(c * 2 + 0) * NNQ + lj * Q1 + q0] = sb;
      P1[(c * 2 + 1) * NNQ + lj * Q1 + q0] = sg;
    }
  }
  __syncwarp();
  #pragma unroll
  for (int k = 0; k < (NC * N * Q1 + 31) / 32; ++k) {          // (c, l, q0)
    const int t = lane + 32 * k;
    if (t >= NC * N * Q1) break;
    const int q0 = t % Q1, l = (t / Q1) % N, c = t / (Q1 * N);
    R xb[N], xg[N];
#pragma unroll
    for (int j = 0; j < N; ++j) {
      xb[j] = P1[(c * 2 + 0) * NNQ + (l * N + j) * Q1 + q0];
      xg[j] = P1[(c * 2 + 1) * NNQ + (l * N + j) * Q1 + q0];
    }
#pragma unroll
    for (int q1 = 0; q1 < Q1; ++q1) {
      R bb = R(0), bg = R(0), gb = R(0);
#pragma unroll
      for (int j = 0; j < N; ++j) {
        bb = fma(xb[j], tB[q1 * N + j], bb);
        bg = fma(xb[j], tG[q1 * N + j], bg);
        gb = fma(xg[j], tB[q1 * N + j], gb);
      }
      const int o = l * QQ + q1 * Q1 + q0;
      P0[(c * 3 + 0) * NQQ + o] = bb;
      P0[(c * 3 + 1) * NQQ + o] = bg;
      P0[(c * 3 + 2) * NQQ + o] = gb;
    }
  }
  __syncwarp();
  #pragma unroll
  for (int k = 0; k < (NC * QQ + 31) / 32; ++k) {              // (c, q1, q0) columns
    const int t = lane + 32 * k;
    if (t >= NC * QQ) break;
    const int c = t / QQ, q01 = t % QQ;
    R sbb[N], sbg[N], sgb[N];
#pragma unroll
    for (int l = 0; l < N; ++l) {
      sbb[l] = P0[(c * 3 + 0) * NQQ + l * QQ + q01];
      sbg[l] = P0[(c * 3 + 1) * NQQ + l * QQ + q01];
      sgb[l] = P0[(c * 3 + 2) * NQQ + l * QQ + q01];
    }
#pragma unroll
    for (int q2 = 0; q2 < Q1; ++q2) {
      R a0 = R(0), a1 = R(0), a2 = R(0);
#pragma unroll
      for (int l = 0; l < N; ++l) {
        a0 = fma(sgb[l], tB[q2 * N + l], a0);
        a1 = fma(sbg[l], tB[q2 * N + l], a1);
        a2 = fma(sbb[l], tG[q2 * N + l], a2);
      }
      const int o = q2 * QQ + q01;
      P1[(c * 3 + 0) * QQQ + o] = a0;
      P1[(c * 3 + 1) * QQQ + o] = a1;
      P1[(c * 3 + 2) * QQQ + o] = a2;
    }
  }
  __syncwarp();
}

template <int N, int Q1, int NC, class R>
__device__ __forceinline__ void adj3_rb(const R (&tB)[Q1 * N], const R (&tG)[Q1 * N], R* P0, R* P1, int lane) {
  constexpr int NNQ = N * N * Q1, NQQ = N * Q1 * Q1, QQ = Q1 * Q1, QQQ = Q1 * Q1 * Q1;
  #pragma unroll
  for (int k = 0; k < (NC * QQ + 31) / 32; ++k) {              // (c, q1, q0) columns of R
    const int t = lane + 32 * k;
    if (t >= NC * QQ) break;
    const int c = t / QQ, q01 = t % QQ;
    R r0[Q1], r1[Q1], r2[Q1];
#pragma unroll
    for (int q2 = 0; q2 < Q1; ++q2) {
      r0[q2] = P1[(c * 3 + 0) * QQQ + q2 * QQ + q01];
      r1[q2] = P1[(c * 3 + 1) * QQQ + q2 * QQ + q01];
      r2[q2] = P1[(c * 3 + 2) * QQQ + q2 * QQ + q01];
    }
#pragma unroll
    for (int l = 0; l < N; ++l) {
      R u0 = R(0), u1 = R(0), u2 = R(0);
#pragma unroll
      for (int q2 = 0; q2 < Q1; ++q2) {
        u0 = fma(r0[q2], tB[q2 * N + l], u0);
        u1 = fma(r1[q2], tB[q2 * N + l], u1);
        u2 = fma(r2[q2], tG[q2 * N + l], u2);
      }
      const int o = l * QQ + q01;
      P0[(c * 3 + 0) * NQQ + o] = u0;
      P0[(c * 3 + 1) * NQQ + o] = u1;
      P0[(c * 3 + 2) * NQQ + o] = u2;
    }
  }
  __syncwarp();
  #pragma unroll
  for (int k = 0; k < (NC * N * Q1 + 31) / 32; ++k) {          // (c, l, q0)
    const int t = lane + 32 * k;
    if (t >= NC * N * Q1) break;
    const int q0 = t % Q1, l = (t / Q1) % N, c = t / (Q1 * N);
    R u0[Q1], u1[Q1], u2[Q1];
#pragma unroll
    for (int q1 = 0; q1 < Q1; ++q1) {
      u0[q1] = P0[(c * 3 + 0) * NQQ + l * QQ + q1 * Q1 + q0];
      u1[q1] = P0[(c * 3 + 1) * NQQ + l * QQ + q1 * Q1 + q0];
      u2[q1] = P0[(c * 3 + 2) * NQQ + l * QQ + q1 * Q1 + q0];
    }
#pragma unroll
    for (int j = 0; j < N; ++j) {
      R vg = R(0), vb = R(0);
#pragma unroll
      for (int q1 = 0; q1 < Q1; ++q1) {
        vg = fma(u0[q1], tB[q1 * N + j], vg);
        vb = fma(u1[q1], tG[q1 * N + j], fma(u2[q1], tB[q1 * N + j], vb));
      }
      const int o = (l * N + j) * Q1 + q0;
      P1[(c * 2 + 0) * NNQ + o] = vg;
      P1[(c * 2 + 1) * NNQ + o] = vb;
    }
  }
  __syncwarp();
  #pragma unroll
  for (int k = 0; k < (NC * N * N + 31) / 32; ++k) {           // (c, l, j) rows of y
    const int t = lane + 32 * k;
    if (t >= NC * N * N) break;
    const int c = t / (N * N), lj = t % (N * N);
    R vg[Q1], vb[Q1];
#pragma unroll
    for (int q0 = 0; q0 < Q1; ++q0) {
      vg[q0] = P1[(c * 2 + 0) * NNQ + lj * Q1 + q0];
      vb[q0] = P1[(c * 2 + 1) * NNQ + lj * Q1 + q0];
    }
#pragma unroll
    for (int i = 0; i < N; ++i) {
      R y = R(0);
#pragma unroll
      for (int q0 = 0; q0 < Q1; ++q0) y = fma(vg[q0], tG[q0 * N + i], fma(vb[q0], tB[q0 * N + i], y));
      P0[t * N + i] = y;
    }
  }
  __syncwarp();
}

}  // namespace tmop
