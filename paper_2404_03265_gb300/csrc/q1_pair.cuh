// Arithmetic shared by the Q1 cell kernels: packed pairs (the two members are two
// cells), the Q1 field of a cell at the 2x2 Gauss points and the test of fluxes and
// values against the cell's basis.  Every operation is an explicit intrinsic, so
// kernels that call these functions round the same expressions.
#pragma once

#include "kernels.cuh"

namespace pff {

template <typename T> struct VT;
template <> struct VT<float> { using T2 = float2; using T4 = float4; };
template <> struct VT<double> { using T2 = double2; using T4 = dbl4; };

// 2-point Gauss rule on [0, 1]
constexpr double GA = 0.21132486540518711775;
constexpr double GB = 0.78867513459481288225;

// ---- one cell (a scalar) or two (a packed pair; FP32: Blackwell paired instructions).
// Products and sums are single rounded operations that the compiler does not contract.
template <typename P> struct Elem;   // element type of a scalar or pair
template <> struct Elem<float> { using T = float; };
template <> struct Elem<double> { using T = double; };
template <> struct Elem<float2> { using T = float; };
template <> struct Elem<double2> { using T = double; };
__device__ __forceinline__ float pfma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ float padd(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float pmul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double pfma(double a, double b, double c) { return __fma_rn(a, b, c); }
__device__ __forceinline__ double padd(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ double pmul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float2 pfma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 padd(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 pmul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ double2 pfma(double2 a, double2 b, double2 c) {
  return make_double2(__fma_rn(a.x, b.x, c.x), __fma_rn(a.y, b.y, c.y));
}
__device__ __forceinline__ double2 padd(double2 a, double2 b) {
  return make_double2(__dadd_rn(a.x, b.x), __dadd_rn(a.y, b.y));
}
__device__ __forceinline__ double2 pmul(double2 a, double2 b) {
  return make_double2(__dmul_rn(a.x, b.x), __dmul_rn(a.y, b.y));
}
// s in every member of a P
template <typename P>
__device__ __forceinline__ P bc(typename Elem<P>::T s) {
  if constexpr (sizeof(P) == sizeof(s)) return s; else return P{s, s};
}
__device__ __forceinline__ float2 pbc(float s) { return make_float2(s, s); }
__device__ __forceinline__ double2 pbc(double s) { return make_double2(s, s); }
template <typename P>
__device__ __forceinline__ P psub(P a, P b) { return pfma(b, bc<P>(typename Elem<P>::T(-1)), a); }  // a - b, exact sign flip

// Q1 field on a cell (pair): reference derivatives at the Gauss points.
//   dxi[q2] = dv/dxi at eta = g_q2, deta[q1] = dv/deta at xi = g_q1.
template <typename P>
struct PField {
  P dxi[2], deta[2];
  P dx0, dy0, X;
  // b, t: values at the cell's lower-left and upper-left nodes; hb, ht: the
  // right node minus the left node along the lower and upper edge
  __device__ __forceinline__ void init(P b, P hb, P t, P ht) {
    using T = typename Elem<P>::T;
    dx0 = hb;
    dy0 = psub(t, b);
    X = psub(ht, hb);
    dxi[0] = pfma(bc<P>(T(GA)), X, dx0);
    dxi[1] = pfma(bc<P>(T(GB)), X, dx0);
    deta[0] = pfma(bc<P>(T(GA)), X, dy0);
    deta[1] = pfma(bc<P>(T(GB)), X, dy0);
  }
  // values at (xi_q1, eta_q2) given v0
  __device__ __forceinline__ void values(P v0, P val[2][2]) const {
    using T = typename Elem<P>::T;
    const P vb0 = pfma(bc<P>(T(GA)), dx0, v0), vb1 = pfma(bc<P>(T(GB)), dx0, v0);
    val[0][0] = pfma(bc<P>(T(GA)), deta[0], vb0);
    val[0][1] = pfma(bc<P>(T(GB)), deta[0], vb0);
    val[1][0] = pfma(bc<P>(T(GA)), deta[1], vb1);
    val[1][1] = pfma(bc<P>(T(GB)), deta[1], vb1);
  }
};

// Test a gradient flux fx (coefficient of dN/dxi), fy (of dN/deta) given per
// Gauss point, with weights wx, wy (nwx = -wx, nwy = -wy), into r[0..3].
//   dN/dxi: N0 -(1-eta), N1 (1-eta), N2 -eta, N3 eta
//   dN/deta: N0 -(1-xi), N1 -xi, N2 (1-xi), N3 xi
template <typename P>
__device__ __forceinline__ void ptest_grad(P sx0, P sx1, P sy0, P sy1, P wx, P wy, P nwx, P nwy, P r[4]) {
  using T = typename Elem<P>::T;
  const P px = pfma(bc<P>(T(GA)), sx0, pmul(bc<P>(T(GB)), sx1));
  const P qx = psub(padd(sx0, sx1), px);
  const P py = pfma(bc<P>(T(GA)), sy0, pmul(bc<P>(T(GB)), sy1));
  const P qy = psub(padd(sy0, sy1), py);
  r[0] = pfma(nwx, qx, pfma(nwy, qy, r[0]));
  r[1] = pfma(wx, qx, pfma(nwy, py, r[1]));
  r[2] = pfma(nwx, px, pfma(wy, qy, r[2]));
  r[3] = pfma(wx, px, pfma(wy, py, r[3]));
}

// Test a value f given per Gauss point [q1][q2] against N_A = L_a(xi) L_b(eta), into r[0..3].
template <typename P>
__device__ __forceinline__ void ptest_value(const P fv[2][2], P jxw, P r[4]) {
  using T = typename Elem<P>::T;
  const P s0 = padd(fv[0][0], fv[0][1]), s1 = padd(fv[1][0], fv[1][1]);
  const P t0 = pfma(bc<P>(T(GA)), fv[0][0], pmul(bc<P>(T(GB)), fv[0][1]));
  const P t1 = pfma(bc<P>(T(GA)), fv[1][0], pmul(bc<P>(T(GB)), fv[1][1]));
  const P b0 = psub(s0, t0), b1 = psub(s1, t1);
  const P pb = pfma(bc<P>(T(GA)), b0, pmul(bc<P>(T(GB)), b1));
  const P pt = pfma(bc<P>(T(GA)), t0, pmul(bc<P>(T(GB)), t1));
  r[0] = pfma(jxw, psub(padd(b0, b1), pb), r[0]);
  r[1] = pfma(jxw, pb, r[1]);
  r[2] = pfma(jxw, psub(padd(t0, t1), pt), r[2]);
  r[3] = pfma(jxw, pt, r[3]);
}

}  // namespace pff
