// FP32 cell arithmetic of the tiled Q1 level kernels: a level block (u-u or phi-phi) on a
// pair of cells whose nodes lie in a window of NW x NW nodes in shared memory.  The
// expressions are those of q1_cell for OP_UU and OP_PP, split into the factors that do not
// depend on the input and the apply.
#pragma once

#include "q1_pair.cuh"

namespace pff {
namespace tile {

using P = float2;

// components of a block's node value: UU two (u_x, u_y), PP one
template <int OP> struct Comp;
template <> struct Comp<OP_UU> { static constexpr int NC = 2; using V = float2; };
template <> struct Comp<OP_PP> { static constexpr int NC = 1; using V = float; };

__device__ __forceinline__ float& comp(float2& v, int c) { return c ? v.y : v.x; }
__device__ __forceinline__ float comp(const float2& v, int c) { return c ? v.y : v.x; }
__device__ __forceinline__ float& comp(float& v, int) { return v; }
__device__ __forceinline__ float comp(const float& v, int) { return v; }

// component c of window nodes a, b as a pair
template <typename V>
__device__ __forceinline__ P two(const V* s, int a, int b, int c) {
  return make_float2(comp(s[a], c), comp(s[b], c));
}

// The x-independent Gauss-point factors of a cell pair: UU g(phi~), PP the mass coefficient.
// sv: window node values, UU phi~ in .x; PP (u_x, u_y).
template <int OP, int NW, typename V>
__device__ __forceinline__ void cell_coef(const V* sv, int a, int b, const MatConst<float>& m,
                                          const LevGeom<float>& g, P ec, P q[2][2]) {
  const P omk = pbc(m.omk);
  auto init = [&](PField<P>& f, int c, P& b0) {
    b0 = two(sv, a, b, c);
    const P t0 = two(sv, a + NW, b + NW, c);
    f.init(b0, psub(two(sv, a + 1, b + 1, c), b0), t0, psub(two(sv, a + NW + 1, b + NW + 1, c), t0));
  };
  if constexpr (OP == OP_UU) {
    PField<P> f;
    P b0, v[2][2];
    init(f, 0, b0);
    f.values(b0, v);
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int j = 0; j < 2; ++j) q[i][j] = pfma(omk, pmul(v[i][j], v[i][j]), pbc(m.kap));
  } else {
    const P ihx = pbc(g.ihx), ihy = pbc(g.ihy), pp = pbc(m.p);
    const P oc2ml = pmul(omk, pmul(pbc(m.c2ml), ec)), ocl = pmul(omk, pmul(pbc(m.cl), ec)),
            ocm = pmul(omk, pmul(pbc(m.cm), ec));
    PField<P> fx, fy;
    P b0, e11[2], e22[2], uyx[2], uxy[2];
    init(fx, 0, b0);
    init(fy, 1, b0);
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      e11[i] = pmul(fx.dxi[i], ihx);
      uyx[i] = pmul(fy.dxi[i], ihx);
      e22[i] = pmul(fy.deta[i], ihy);
      uxy[i] = pmul(fx.deta[i], ihy);
    }
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const P ge12 = padd(uxy[i], uyx[j]);
        const P q11 = pfma(oc2ml, e11[j], pfma(ocl, e22[i], pp));
        const P q22 = pfma(ocl, e11[j], pfma(oc2ml, e22[i], pp));
        const P q12 = pmul(ocm, ge12);
        q[i][j] = pfma(q11, e11[j],
                       pfma(q22, e22[i], pfma(q12, ge12, pfma(pp, padd(e11[j], e22[i]), pbc(m.gcl)))));
      }
  }
}

// Cell contributions r[component][corner] of a cell pair (corners 0 (0,0), 1 (1,0), 2 (0,1), 3 (1,1)).
template <int OP, int NW, typename V>
__device__ __forceinline__ void cell_apply(const V* xs, int a, int b, const MatConst<float>& m,
                                           const LevGeom<float>& g, P ec, const P q[2][2],
                                           P r[Comp<OP>::NC][4]) {
  const P zero = pbc(0.f);
#pragma unroll
  for (int c = 0; c < Comp<OP>::NC; ++c)
#pragma unroll
    for (int k = 0; k < 4; ++k) r[c][k] = zero;
  auto init = [&](PField<P>& f, int c, P& b0) {
    b0 = two(xs, a, b, c);
    const P t0 = two(xs, a + NW, b + NW, c);
    f.init(b0, psub(two(xs, a + 1, b + 1, c), b0), t0, psub(two(xs, a + NW + 1, b + NW + 1, c), t0));
  };
  if constexpr (OP == OP_UU) {
    const P ihx = pbc(g.ihx), ihy = pbc(g.ihy);
    const P c2ml = pmul(pbc(m.c2ml), ec), cl = pmul(pbc(m.cl), ec), cm = pmul(pbc(m.cm), ec);
    PField<P> fx, fy;
    P b0, ax[2], dy[2], bxy[2], cyx[2], S11[2][2], S12[2][2], S22[2][2];
    init(fx, 0, b0);
    init(fy, 1, b0);
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      ax[i] = pmul(fx.dxi[i], ihx);
      cyx[i] = pmul(fy.dxi[i], ihx);
      dy[i] = pmul(fy.deta[i], ihy);
      bxy[i] = pmul(fx.deta[i], ihy);
    }
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const P bc = padd(bxy[i], cyx[j]);
        S11[i][j] = pmul(q[i][j], pfma(c2ml, ax[j], pmul(cl, dy[i])));
        S22[i][j] = pmul(q[i][j], pfma(cl, ax[j], pmul(c2ml, dy[i])));
        S12[i][j] = pmul(q[i][j], pmul(cm, bc));
      }
    const P wx = pbc(g.wx), wy = pbc(g.wy), nwx = pbc(-g.wx), nwy = pbc(-g.wy);
    ptest_grad(padd(S11[0][0], S11[1][0]), padd(S11[0][1], S11[1][1]), padd(S12[0][0], S12[0][1]),
               padd(S12[1][0], S12[1][1]), wx, wy, nwx, nwy, r[0]);
    ptest_grad(padd(S12[0][0], S12[1][0]), padd(S12[0][1], S12[1][1]), padd(S22[0][0], S22[0][1]),
               padd(S22[1][0], S22[1][1]), wx, wy, nwx, nwy, r[1]);
  } else {
    PField<P> f;
    P b0, v[2][2], fv[2][2];
    init(f, 0, b0);
    f.values(b0, v);
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int j = 0; j < 2; ++j) fv[i][j] = pmul(q[i][j], v[i][j]);
    ptest_value(fv, pbc(g.jxw), r[0]);
    ptest_grad(f.dxi[0], f.dxi[1], f.deta[0], f.deta[1], pbc(g.wpx), pbc(g.wpy), pbc(-g.wpx), pbc(-g.wpy), r[0]);
  }
}

}  // namespace tile
}  // namespace pff
