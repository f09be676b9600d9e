// The Q2 leaf operators on one cell: Jacobian, its transpose and the residual (Sec. 3.1
// and Problem 2 of Kolditz & Wick, arXiv 2404.03265) with the 3x3 Gauss rule.
//
// Sum factorisation with the symmetry of the 1D rule: its points are -s, 0, s about the
// middle node, so with d = v2 - v0 and c = v0 - 2 v1 + v2 a quadratic is v1 + t d + 2 t^2 c
// and its derivative d + 4 t c; the middle point costs nothing (value) or one operation
// (derivative).  Geometry, Gauss weights and elastic constants are folded into per-cell
// constants that multiply reference derivatives.  About 1,000 operations a cell against
// about 2,400 for the plain 3-term contractions with scalings at every point.
// Fields that take the same contractions travel as pairs (u_x with u_y; the input dphi
// with phi), one paired instruction for both in FP32.
#pragma once

#include "q1_cell.cuh"

namespace pff {

// 1D values and derivatives at the Gauss points of a quadratic with nodal values v
template <typename P>
__device__ __forceinline__ void q2_even_odd(P v0, P v1, P v2, P& d, P& c) {
  using T = typename Elem<P>::T;
  d = psub(v2, v0);
  c = pfma(bc<P>(T(-2)), v1, padd(v0, v2));
}
constexpr double kQ2S = 0.38729833462074168852;   // half the distance of the outer points, sqrt(15) / 10
template <typename P>
__device__ __forceinline__ void q2_values(P v1, P d, P c, P out[3]) {
  using T = typename Elem<P>::T;
  const P e = pfma(bc<P>(T(0.3)), c, v1);
  out[0] = pfma(bc<P>(T(-kQ2S)), d, e);
  out[1] = v1;
  out[2] = pfma(bc<P>(T(kQ2S)), d, e);
}
template <typename P>
__device__ __forceinline__ void q2_derivs(P d, P c, P out[3]) {
  using T = typename Elem<P>::T;
  out[0] = pfma(bc<P>(T(-4.0 * kQ2S)), c, d);
  out[1] = d;
  out[2] = pfma(bc<P>(T(4.0 * kQ2S)), c, d);
}
// transposes: nodal tests of point values f against the basis and against its derivative
template <typename P>
__device__ __forceinline__ void q2_test_value(const P f[3], P r[3]) {
  using T = typename Elem<P>::T;
  const P s = padd(f[0], f[2]), d = psub(f[2], f[0]), s3 = pmul(bc<P>(T(0.3)), s);
  r[0] = pfma(bc<P>(T(-kQ2S)), d, s3);
  r[1] = pfma(bc<P>(T(0.4)), s, f[1]);
  r[2] = pfma(bc<P>(T(kQ2S)), d, s3);
}
template <typename P>
__device__ __forceinline__ void q2_test_deriv(const P f[3], P r[3]) {
  using T = typename Elem<P>::T;
  const P t = padd(padd(f[0], f[1]), f[2]), h = pmul(bc<P>(T(4.0 * kQ2S)), psub(f[2], f[0]));
  r[0] = psub(h, t);
  r[1] = pmul(bc<P>(T(-2)), h);
  r[2] = padd(h, t);
}
// A Gauss row eta = t.  RowAt<T, Q>: known when compiled (the middle row costs next to
// nothing); RowVar: at run time, so that a loop over the rows keeps only one of them in
// registers.
template <typename T, int Q>
struct RowAt {
  static constexpr double t = (Q - 1) * kQ2S;
  // value and derivative along eta of a column (v0, v1, v2)
  template <typename P>
  __device__ __forceinline__ void column(P v0, P v1, P v2, P& V, P& E) const {
    if constexpr (Q == 1) {
      V = v1;
      E = psub(v2, v0);
    } else {
      P d, c;
      q2_even_odd(v0, v1, v2, d, c);
      V = pfma(bc<P>(T(t)), d, pfma(bc<P>(T(0.3)), c, v1));
      E = pfma(bc<P>(T(4.0 * t)), c, d);
    }
  }
  template <typename P>
  __device__ __forceinline__ P value(P v0, P v1, P v2) const {
    if constexpr (Q == 1) return v1;
    else return pfma(bc<P>(T(2 * t * t + t)), v2, pfma(bc<P>(T(1 - 4 * t * t)), v1, pmul(bc<P>(T(2 * t * t - t)), v0)));
  }
  // r[a + 3 b] += l_b(t) V[a] + l_b'(t) E[a]
  template <typename P>
  __device__ __forceinline__ void scatter(const P V[3], const P E[3], P r[9]) const {
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      if constexpr (Q == 1) {
        r[a] = psub(r[a], E[a]);
        r[a + 3] = padd(r[a + 3], V[a]);
        r[a + 6] = padd(r[a + 6], E[a]);
      } else {
        r[a] = pfma(bc<P>(T(2 * t * t - t)), V[a], pfma(bc<P>(T(4 * t - 1)), E[a], r[a]));
        r[a + 3] = pfma(bc<P>(T(1 - 4 * t * t)), V[a], pfma(bc<P>(T(-8 * t)), E[a], r[a + 3]));
        r[a + 6] = pfma(bc<P>(T(2 * t * t + t)), V[a], pfma(bc<P>(T(4 * t + 1)), E[a], r[a + 6]));
      }
    }
  }
  __device__ __forceinline__ int weight_class(int i) const { return (i == 1) + (Q == 1); }
  __device__ __forceinline__ T weight(int i) const {
    constexpr double w1[3] = {5.0 / 18.0, 8.0 / 18.0, 5.0 / 18.0};
    return T(w1[i] * w1[Q]);
  }
};

template <typename T>
struct RowVar {
  T t;
  bool mid;
  __device__ __forceinline__ explicit RowVar(int q) : t(T(kQ2S) * T(q - 1)), mid(q == 1) {}
  template <typename P>
  __device__ __forceinline__ void column(P v0, P v1, P v2, P& V, P& E) const {
    P d, c;
    q2_even_odd(v0, v1, v2, d, c);
    V = pfma(bc<P>(t), d, pfma(bc<P>(mid ? T(0) : T(0.3)), c, v1));
    E = pfma(bc<P>(T(4) * t), c, d);
  }
  template <typename P>
  __device__ __forceinline__ P value(P v0, P v1, P v2) const {
    const T h = mid ? T(0) : T(0.3);
    return pfma(bc<P>(h + t), v2, pfma(bc<P>(T(1) - T(2) * h), v1, pmul(bc<P>(h - t), v0)));
  }
  template <typename P>
  __device__ __forceinline__ void scatter(const P V[3], const P E[3], P r[9]) const {
    const T h = mid ? T(0) : T(0.3);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      r[a] = pfma(bc<P>(h - t), V[a], pfma(bc<P>(T(4) * t - T(1)), E[a], r[a]));
      r[a + 3] = pfma(bc<P>(T(1) - T(2) * h), V[a], pfma(bc<P>(T(-8) * t), E[a], r[a + 3]));
      r[a + 6] = pfma(bc<P>(h + t), V[a], pfma(bc<P>(T(4) * t + T(1)), E[a], r[a + 6]));
    }
  }
  __device__ __forceinline__ int weight_class(int i) const { return (i == 1) + (mid ? 1 : 0); }
  __device__ __forceinline__ T weight(int i) const {
    return (i == 1 ? T(8.0 / 18.0) : T(5.0 / 18.0)) * (mid ? T(8.0 / 18.0) : T(5.0 / 18.0));
  }
};

// The cell's own constants beside Q2Mat (kernels.cuh): p hy, p hx, G_c/l times the area, modulus
template <typename T>
struct Q2Own {
  T px, py, gcl, ec;
  __device__ __forceinline__ Q2Own(const MatConst<T>& m, const LevGeom<T>& g, T e) {
    const T area = T(4) * g.jxw;   // hx hy
    px = m.p * (g.ihx * area);
    py = m.p * (g.ihy * area);
    gcl = m.gcl * area;
    ec = e;
  }
};

// One Gauss row: ld(k, a, b) is field pair k at the cell's node (a, b): 0 the input
// (u_x, u_y), 1 the linearisation's (u_x, u_y), 2 (input dphi, phi), 3 (phi_tilde, -).
// MOD: the cell has a modulus of its own (o.ec; the constants are those of unit E).
template <typename T, int OP, bool MOD, class Row, class Load>
__device__ __forceinline__ void q2_jac_row(const Row& row, const Load& ld, const Q2Mat<T>& k, const Q2Own<T>& o,
                                           typename VT<T>::T2 ru[9], T rp[9]) {
  using P = typename VT<T>::T2;
  constexpr bool RES = OP == OP_RESID;
  // (the residual is R = -A)
  // ---- fields at the row's three points: reference derivatives and values
  P xdx[3], xdy[3], ldx[3], ldy[3], val[3];   // (u_x, u_y) of input and linearisation; (dphi, phi)
  T pdx[3], pdy[3], pt[3];                    // gradient of dphi (residual: of phi), phi_tilde
  {
    P V[3], E[3], d, c;
    if constexpr (!RES) {
#pragma unroll
      for (int a = 0; a < 3; ++a) row.column(ld(0, a, 0), ld(0, a, 1), ld(0, a, 2), V[a], E[a]);
      q2_even_odd(V[0], V[1], V[2], d, c);
      q2_derivs(d, c, xdx);
      q2_even_odd(E[0], E[1], E[2], d, c);
      q2_values(E[1], d, c, xdy);
    }
#pragma unroll
    for (int a = 0; a < 3; ++a) row.column(ld(1, a, 0), ld(1, a, 1), ld(1, a, 2), V[a], E[a]);
    q2_even_odd(V[0], V[1], V[2], d, c);
    q2_derivs(d, c, ldx);
    q2_even_odd(E[0], E[1], E[2], d, c);
    q2_values(E[1], d, c, ldy);
    T Es[3], Vs[3], ds, cs;
    if constexpr (RES) {
#pragma unroll
      for (int a = 0; a < 3; ++a) row.column(ld(2, a, 0).y, ld(2, a, 1).y, ld(2, a, 2).y, Vs[a], Es[a]);
      T v[3];
      q2_even_odd(Vs[0], Vs[1], Vs[2], ds, cs);
      q2_values(Vs[1], ds, cs, v);
      q2_derivs(ds, cs, pdx);
#pragma unroll
      for (int i = 0; i < 3; ++i) val[i] = P{T(0), v[i]};
    } else {
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        const P v0 = ld(2, a, 0), v1 = ld(2, a, 1), v2 = ld(2, a, 2);
        V[a] = row.value(v0, v1, v2);
        T unused;
        row.column(v0.x, v1.x, v2.x, unused, Es[a]);
      }
      q2_even_odd(V[0], V[1], V[2], d, c);
      q2_values(V[1], d, c, val);
      q2_derivs(d.x, c.x, pdx);
    }
    q2_even_odd(Es[0], Es[1], Es[2], ds, cs);
    q2_values(Es[1], ds, cs, pdy);
#pragma unroll
    for (int a = 0; a < 3; ++a) Vs[a] = row.value(ld(3, a, 0).x, ld(3, a, 1).x, ld(3, a, 2).x);
    q2_even_odd(Vs[0], Vs[1], Vs[2], ds, cs);
    q2_values(Vs[1], ds, cs, pt);
  }
  // ---- fluxes: Fx tests d/dxi, Fy d/deta (pairs: u_x and u_y rows), f0 the value of psi_phi
  P Fx[3], Fy[3];
  T f0[3], gx[3], gy[3];
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const T W = RES ? -row.weight(i) : row.weight(i);
    const T a = ldx[i].x, b = ldy[i].x, c = ldx[i].y, d = ldy[i].y;   // u_x,xi u_x,eta u_y,xi u_y,eta
    const int wi = row.weight_class(i);   // corner, edge, centre
    T g = pfma(k.omkw[wi], pmul(pt[i], pt[i]), k.kapw[wi]);   // signed weight times g(phi~)
    if (RES) g = -g;
    T q11 = pfma(k.oal, a, pmul(k.obe, d)), q22 = pfma(k.obe, a, pmul(k.oalt, d));
    T t1 = pfma(k.oga, b, pmul(k.ode, c)), t2 = pfma(k.ode, b, pmul(k.ogat, c));
    if constexpr (MOD) {
      g = pmul(g, o.ec);
      t1 = pmul(t1, o.ec);
      t2 = pmul(t2, o.ec);
      q11 = RES ? pmul(q11, o.ec) : pfma(o.ec, q11, o.px);
      q22 = RES ? pmul(q22, o.ec) : pfma(o.ec, q22, o.py);
    } else if constexpr (!RES) {
      q11 = padd(q11, o.px);
      q22 = padd(q22, o.py);
    }
    // (1 - kappa) sigma(u):e(u), in the Jacobian with p div u once
    const T se = pfma(q11, a, pfma(q22, d, pfma(t1, b, pmul(t2, c))));
    const T ph = val[i].y;
    if constexpr (RES) {
      const T pp = pmul(W, pmul(pt[i], pt[i]));
      Fx[i].x = pfma(g, pfma(k.al, a, pmul(k.be, d)), pmul(o.px, pp));
      Fy[i].x = pmul(g, pfma(k.ga, b, pmul(k.de, c)));
      Fx[i].y = pmul(g, pfma(k.de, b, pmul(k.gat, c)));
      Fy[i].y = pfma(g, pfma(k.be, a, pmul(k.alt, d)), pmul(o.py, pp));
      const T dv = pfma(o.px, a, pmul(o.py, d));
      f0[i] = pmul(W, pfma(ph, pfma(T(2), dv, se), pmul(o.gcl, psub(ph, T(1)))));
    } else {
      const T A = xdx[i].x, B = xdy[i].x, C = xdx[i].y, D = xdy[i].y, xp = val[i].x;
      const T m = pfma(o.px, a, pfma(o.py, d, padd(se, o.gcl)));
      Fx[i].x = pmul(g, pfma(k.al, A, pmul(k.be, D)));
      Fy[i].x = pmul(g, pfma(k.ga, B, pmul(k.de, C)));
      Fx[i].y = pmul(g, pfma(k.de, B, pmul(k.gat, C)));
      Fy[i].y = pmul(g, pfma(k.be, A, pmul(k.alt, D)));
      if constexpr (OP == OP_FULL) {
        const T w = pfma(q11, A, pfma(q22, D, pfma(t1, B, pmul(t2, C))));
        f0[i] = pmul(W, pfma(padd(ph, ph), w, pmul(m, xp)));
      } else {
        const T z = pmul(pmul(T(2) * W, ph), xp);
        Fx[i].x = pfma(z, q11, Fx[i].x);
        Fy[i].x = pfma(z, t1, Fy[i].x);
        Fx[i].y = pfma(z, t2, Fx[i].y);
        Fy[i].y = pfma(z, q22, Fy[i].y);
        f0[i] = pmul(W, pmul(m, xp));
      }
    }
    gx[i] = pmul(RES ? -k.gxxw[wi] : k.gxxw[wi], pdx[i]);
    gy[i] = pmul(RES ? -k.gyyw[wi] : k.gyyw[wi], pdy[i]);
  }
  // ---- tests
  {
    P V[3], E[3];
    q2_test_deriv(Fx, V);
    q2_test_value(Fy, E);
    row.scatter(V, E, ru);
  }
  {
    T V[3], E[3], V0[3];
    q2_test_deriv(gx, V);
    q2_test_value(f0, V0);
#pragma unroll
    for (int a = 0; a < 3; ++a) V[a] = padd(V[a], V0[a]);
    q2_test_value(gy, E);
    row.scatter(V, E, rp);
  }
}

// Contributions of one cell to its node a + 3 b: ru (u_x, u_y), rp (phi).  OP: OP_FULL,
// OP_FULL_T or OP_RESID.
template <typename T, int OP, bool MOD, class Load>
__device__ __forceinline__ void q2_jac(const Load& ld, const Q2Mat<T>& k, const Q2Own<T>& o,
                                       typename VT<T>::T2 ru[9], T rp[9]) {
  using P = typename VT<T>::T2;
#pragma unroll
  for (int i = 0; i < 9; ++i) {
    ru[i] = P{T(0), T(0)};
    rp[i] = T(0);
  }
  if constexpr (sizeof(T) == 8) {
    // FP64: each row from zero, then (row 0 + row 1) + row 2, the bits of the kernel that
    // gives a row to a warp (leaf_cells_q2.cu)
    q2_jac_row<T, OP, MOD>(RowAt<T, 0>(), ld, k, o, ru, rp);
    P u[9];
    T p[9];
    auto add = [&](const auto& row) {
#pragma unroll
      for (int i = 0; i < 9; ++i) {
        u[i] = P{T(0), T(0)};
        p[i] = T(0);
      }
      q2_jac_row<T, OP, MOD>(row, ld, k, o, u, p);
#pragma unroll
      for (int i = 0; i < 9; ++i) {
        ru[i] = padd(ru[i], u[i]);
        rp[i] = padd(rp[i], p[i]);
      }
    };
    add(RowAt<T, 1>());
    add(RowAt<T, 2>());
  } else {
#pragma unroll 1
    for (int q = 0; q < 3; ++q) q2_jac_row<T, OP, MOD>(RowVar<T>(q), ld, k, o, ru, rp);
  }
}

}  // namespace pff
