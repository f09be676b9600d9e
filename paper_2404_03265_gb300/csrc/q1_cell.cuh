// The operators of the Q1 cell kernels on one cell or a pair of cells: Jacobian and
// transpose, level blocks and their diagonals, residual, lumped mass, crack volume and
// its gradient, parameter and phi_tilde derivatives.
#pragma once

#include "q1_pair.cuh"

namespace pff {

// Which node fields an operator reads.
template <int OP> struct Needs {
  static constexpr bool xu = (OP == OP_FULL || OP == OP_FULL_T || OP == OP_UU || OP == OP_VJP || OP == OP_PHIT_VJP);
  static constexpr bool xp = (OP == OP_FULL || OP == OP_FULL_T || OP == OP_PP || OP == OP_VJP);
  static constexpr bool linU = (OP == OP_FULL || OP == OP_FULL_T || OP == OP_PP || OP == OP_PP_DIAG ||
                                OP == OP_RESID || OP == OP_TCV || OP == OP_TCV_GRAD || OP == OP_VJP ||
                                OP == OP_PHIT_VJP);
  static constexpr bool phi = (OP == OP_FULL || OP == OP_FULL_T || OP == OP_RESID || OP == OP_TCV ||
                               OP == OP_TCV_GRAD || OP == OP_VJP);
  static constexpr bool phit = (OP == OP_FULL || OP == OP_FULL_T || OP == OP_UU || OP == OP_UU_DIAG ||
                                OP == OP_RESID || OP == OP_VJP || OP == OP_PHIT_VJP);
};

// Node fields of one node of a cell (pair), in registers.
template <typename P>
struct NodePair {
  P x0, x1, xp, lx, ly, lz, lw;
};

// One Q1 cell, or two at once (the members of every pair).  b: fields at the cells'
// lower-left nodes (0,0), hb: node (1,0) minus node (0,0); t: fields at the
// upper-left nodes (0,1), ht: node (1,1) minus node (0,1).  out[3*N + c]:
// contribution to node N (0 = (0,0), 1 = (1,0), 2 = (0,1), 3 = (1,1)) of
// component c (0 u_x, 1 u_y, 2 phi), as a pair over the two cells.  ec: the
// cells' moduli E_K (the elastic constants in m are then those of unit E), or 1.
// OP_VJP returns its three per-cell values in out[0..2].
template <typename P, int OP>
__device__ __forceinline__ void q1_cell(const NodePair<P>& b, const NodePair<P>& hb, const NodePair<P>& t,
                                        const NodePair<P>& ht, const MatConst<typename Elem<P>::T>& m,
                                        const LevGeom<typename Elem<P>::T>& g, P ec, P out[12]) {
  using N = Needs<OP>;
  using T = typename Elem<P>::T;
  const P zero = bc<P>(T(0));
  P rux[4] = {zero, zero, zero, zero}, ruy[4] = {zero, zero, zero, zero}, rp[4] = {zero, zero, zero, zero};
  const P ihx = bc<P>(g.ihx), ihy = bc<P>(g.ihy);
  const P c2ml = pmul(bc<P>(m.c2ml), ec), cl = pmul(bc<P>(m.cl), ec), cm = pmul(bc<P>(m.cm), ec), omk = bc<P>(m.omk);
  // du_x/dy + du_y/dx at a Gauss point.  FP64's rate is the limit: here, and in the
  // sums of two products below, the first product is formed inside the sum (always
  // this one, so that every path over the cells gives the same bits).  FP32 rounds
  // both, as the level operators' V-cycles do.
  constexpr bool f64 = sizeof(T) == 8;
  auto shear = [&](const PField<P>& f, int q1, const P* xy, P yx) {
    return f64 ? pfma(f.deta[q1], ihy, yx) : padd(xy[q1], yx);
  };
  // ---- linearisation
  PField<P> fux, fuy, fphi, fphit;
  P e11[2], e22[2], uyx[2], uxy[2];
  if (N::linU) {
    fux.init(b.lx, hb.lx, t.lx, ht.lx);
    fuy.init(b.ly, hb.ly, t.ly, ht.ly);
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      e11[q] = pmul(fux.dxi[q], ihx);    // du_x/dx at eta_q
      uyx[q] = pmul(fuy.dxi[q], ihx);    // du_y/dx at eta_q
      e22[q] = pmul(fuy.deta[q], ihy);   // du_y/dy at xi_q
      uxy[q] = pmul(fux.deta[q], ihy);   // du_x/dy at xi_q
    }
  }
  P phiq[2][2], phitq[2][2];
  if (N::phi) { fphi.init(b.lz, hb.lz, t.lz, ht.lz); fphi.values(b.lz, phiq); }
  if (N::phit) { fphit.init(b.lw, hb.lw, t.lw, ht.lw); fphit.values(b.lw, phitq); }
  // ---- input
  PField<P> fxu, fxv, fxp;
  P ax[2], dy[2], bxy[2], cyx[2], xpq[2][2];
  if (N::xu) {
    fxu.init(b.x0, hb.x0, t.x0, ht.x0);
    fxv.init(b.x1, hb.x1, t.x1, ht.x1);
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      ax[q] = pmul(fxu.dxi[q], ihx);     // d du_x/dx at eta_q
      cyx[q] = pmul(fxv.dxi[q], ihx);    // d du_y/dx at eta_q
      dy[q] = pmul(fxv.deta[q], ihy);    // d du_y/dy at xi_q
      bxy[q] = pmul(fxu.deta[q], ihy);   // d du_x/dy at xi_q
    }
  }
  if (N::xp) { fxp.init(b.xp, hb.xp, t.xp, ht.xp); fxp.values(b.xp, xpq); }
  if (OP == OP_MASS) {
    // (1, psi): the test below of f = 1 gives every node jxw, exactly
    static_assert(GA + GB == 1.0, "");
#pragma unroll
    for (int A = 0; A < 4; ++A) rp[A] = bc<P>(g.jxw);
  } else if (OP == OP_RESID || OP == OP_TCV) {
    // R = -A(U)(psi), Problem 2 with sigma^+ read as sigma:
    //   A_u(psi)   = (g(phi~) sigma(u), e(psi)) + (phi~^2 p, div psi)
    //   A_phi(psi) = ((1-kappa) phi sigma(u):e(u) + 2 p phi div u - G_c/l (1 - phi), psi)
    //                + G_c l (grad phi, grad psi)
    // TCV: (u . grad phi, psi)
    P S11[2][2], S12[2][2], S22[2][2], fv[2][2], G[2][2], U12[2][2];
    P uxq[2][2], uyq[2][2];
    if (OP == OP_TCV) { fux.values(b.lx, uxq); fuy.values(b.ly, uyq); }
#pragma unroll
    for (int q1 = 0; q1 < 2; ++q1)
#pragma unroll
      for (int q2 = 0; q2 < 2; ++q2) {
        if (OP == OP_TCV) {
          // u . grad phi, grad phi from the reference derivatives of phi
          const P gpx = pmul(fphi.dxi[q2], ihx), gpy = pmul(fphi.deta[q1], ihy);
          fv[q1][q2] = pfma(uxq[q1][q2], gpx, pmul(uyq[q1][q2], gpy));
          continue;
        }
        const P gq = pfma(omk, pmul(phitq[q1][q2], phitq[q1][q2]), bc<P>(m.kap));
        const P ge12 = shear(fux, q1, uxy, uyx[q2]);
        const P s11 = pfma(c2ml, e11[q2], pmul(cl, e22[q1]));
        const P s22 = pfma(cl, e11[q2], pmul(c2ml, e22[q1]));
        const P s12 = pmul(cm, ge12);
        const P pt2 = pmul(bc<P>(m.p), pmul(phitq[q1][q2], phitq[q1][q2]));
        S11[q1][q2] = pfma(gq, s11, pt2);
        S22[q1][q2] = pfma(gq, s22, pt2);
        S12[q1][q2] = pmul(gq, s12);
        G[q1][q2] = gq; U12[q1][q2] = s12;
        const P se = pfma(s11, e11[q2], pfma(s22, e22[q1], pmul(s12, ge12)));
        const P ph = phiq[q1][q2];
        // (1-kappa) phi se + 2 p phi div u - G_c/l (1 - phi)
        const P a1 = pfma(pmul(omk, ph), se, pmul(pmul(bc<P>(m.p2), ph), padd(e11[q2], e22[q1])));
        fv[q1][q2] = pfma(bc<P>(m.gcl), psub(ph, bc<P>(T(1))), a1);
      }
    const P wx = bc<P>(g.wx), wy = bc<P>(g.wy), nwx = bc<P>(-g.wx), nwy = bc<P>(-g.wy);
    if (OP == OP_RESID) {
      auto sum = [&](int a, int b, int c, int d) {
        return f64 ? pfma(G[a][b], U12[a][b], S12[c][d]) : padd(S12[a][b], S12[c][d]);
      };
      ptest_grad(padd(S11[0][0], S11[1][0]), padd(S11[0][1], S11[1][1]), sum(0, 0, 0, 1), sum(1, 1, 1, 0), wx, wy, nwx,
                 nwy, rux);
      ptest_grad(sum(0, 0, 1, 0), sum(0, 1, 1, 1),
                 padd(S22[0][0], S22[0][1]), padd(S22[1][0], S22[1][1]), wx, wy, nwx, nwy, ruy);
      ptest_grad(fphi.dxi[0], fphi.dxi[1], fphi.deta[0], fphi.deta[1], bc<P>(g.wpx), bc<P>(g.wpy), bc<P>(-g.wpx),
                 bc<P>(-g.wpy), rp);
    }
    {
      const P jxw = bc<P>(g.jxw);
      const P s0 = padd(fv[0][0], fv[0][1]), s1 = padd(fv[1][0], fv[1][1]);
      const P t0 = pfma(bc<P>(T(GA)), fv[0][0], pmul(bc<P>(T(GB)), fv[0][1]));
      const P t1 = pfma(bc<P>(T(GA)), fv[1][0], pmul(bc<P>(T(GB)), fv[1][1]));
      const P b0 = psub(s0, t0), b1 = psub(s1, t1);
      const P pb = pfma(bc<P>(T(GA)), b0, pmul(bc<P>(T(GB)), b1));
      const P pt = pfma(bc<P>(T(GA)), t0, pmul(bc<P>(T(GB)), t1));
      rp[0] = pfma(jxw, psub(padd(b0, b1), pb), rp[0]);
      rp[1] = pfma(jxw, pb, rp[1]);
      rp[2] = pfma(jxw, psub(padd(t0, t1), pt), rp[2]);
      rp[3] = pfma(jxw, pt, rp[3]);
    }
    if (OP == OP_RESID) {
      const P neg = bc<P>(T(-1));
#pragma unroll
      for (int A = 0; A < 4; ++A) { rux[A] = pmul(rux[A], neg); ruy[A] = pmul(ruy[A], neg); rp[A] = pmul(rp[A], neg); }
    }
  } else if (OP == OP_TCV_GRAD) {
    // J = integral of u . grad phi:  dJ/du_(A,i) = (dphi/dx_i, N_A),  dJ/dphi_A = (u, grad N_A)
    P uxq[2][2], uyq[2][2], gpx[2][2], gpy[2][2];
    fux.values(b.lx, uxq);
    fuy.values(b.ly, uyq);
#pragma unroll
    for (int q1 = 0; q1 < 2; ++q1)
#pragma unroll
      for (int q2 = 0; q2 < 2; ++q2) {
        gpx[q1][q2] = pmul(fphi.dxi[q2], ihx);
        gpy[q1][q2] = pmul(fphi.deta[q1], ihy);
      }
    const P jxw = bc<P>(g.jxw);
    ptest_value(gpx, jxw, rux);
    ptest_value(gpy, jxw, ruy);
    ptest_grad(padd(uxq[0][0], uxq[1][0]), padd(uxq[0][1], uxq[1][1]), padd(uyq[0][0], uyq[0][1]),
               padd(uyq[1][0], uyq[1][1]), bc<P>(g.wx), bc<P>(g.wy), bc<P>(-g.wx), bc<P>(-g.wy), rp);
  } else if (OP == OP_VJP) {
    // x . dR/dtheta per cell (R = -A, Problem 2; x = (w_u, w_phi) after constraints):
    //   E_K: -[(g(phi~) sigma_1(u), e(w_u)) + (1-kappa)(phi sigma_1(u):e(u), w_phi)]_K
    //   p:   -[(phi~^2, div w_u) + 2 (phi div u, w_phi)]_K
    //   G_c: -[-(1/l)(1 - phi, w_phi) + l (grad phi, grad w_phi)]_K
    // sigma_1: stress of unit modulus (m holds unit-E constants for this operator)
    const P uc2ml = bc<P>(m.c2ml), ucl = bc<P>(m.cl), ucm = bc<P>(m.cm);
    const T ihx2 = g.ihx * g.ihx, ihy2 = g.ihy * g.ihy;
    P sE = zero, sP = zero, sG = zero;
#pragma unroll
    for (int q1 = 0; q1 < 2; ++q1)
#pragma unroll
      for (int q2 = 0; q2 < 2; ++q2) {
        const P pt2 = pmul(phitq[q1][q2], phitq[q1][q2]);
        const P gq = pfma(omk, pt2, bc<P>(m.kap));
        const P ge12 = shear(fux, q1, uxy, uyx[q2]);
        const P s11 = pfma(uc2ml, e11[q2], pmul(ucl, e22[q1]));
        const P s22 = pfma(ucl, e11[q2], pmul(uc2ml, e22[q1]));
        const P s12 = pmul(ucm, ge12);
        const P se = pfma(s11, e11[q2], pfma(s22, e22[q1], pmul(s12, ge12)));
        const P gxy = shear(fxu, q1, bxy, cyx[q2]);
        const P sw = pfma(s11, ax[q2], pfma(s22, dy[q1], pmul(s12, gxy)));
        const P ph = phiq[q1][q2], wp = xpq[q1][q2];
        sE = padd(sE, pfma(gq, sw, pmul(pmul(omk, ph), pmul(se, wp))));
        sP = padd(sP, pfma(pt2, padd(ax[q2], dy[q1]), pmul(padd(ph, ph), pmul(padd(e11[q2], e22[q1]), wp))));
        const P gg = pfma(pmul(fphi.dxi[q2], fxp.dxi[q2]), bc<P>(ihx2),
                          pmul(pmul(fphi.deta[q1], fxp.deta[q1]), bc<P>(ihy2)));
        sG = padd(sG, pfma(bc<P>(m.l), gg, pmul(bc<P>(-m.il), pmul(psub(bc<P>(T(1)), ph), wp))));
      }
    const P njxw = bc<P>(-g.jxw);
    rux[0] = pmul(njxw, sE);
    ruy[0] = pmul(njxw, sP);
    rp[0] = pmul(njxw, sG);
  } else if (OP == OP_PHIT_VJP) {
    // (dA/dphi~)^T x: value test of 2 phi~ [(1-kappa) sigma(u):e(x_u) + p div x_u]
    P fv[2][2];
#pragma unroll
    for (int q1 = 0; q1 < 2; ++q1)
#pragma unroll
      for (int q2 = 0; q2 < 2; ++q2) {
        const P ge12 = shear(fux, q1, uxy, uyx[q2]);
        const P s11 = pfma(c2ml, e11[q2], pmul(cl, e22[q1]));
        const P s22 = pfma(cl, e11[q2], pmul(c2ml, e22[q1]));
        const P s12 = pmul(cm, ge12);
        const P sw = pfma(s11, ax[q2], pfma(s22, dy[q1], pmul(s12, shear(fxu, q1, bxy, cyx[q2]))));
        const P pt = phitq[q1][q2];
        fv[q1][q2] = pmul(padd(pt, pt), pfma(omk, sw, pmul(bc<P>(m.p), padd(ax[q2], dy[q1]))));
      }
    ptest_value(fv, bc<P>(g.jxw), rp);
  } else if (OP == OP_UU_DIAG || OP == OP_PP_DIAG) {
#pragma unroll
    for (int q1 = 0; q1 < 2; ++q1)
#pragma unroll
      for (int q2 = 0; q2 < 2; ++q2) {
        const T xi = q1 ? T(GB) : T(GA), eta = q2 ? T(GB) : T(GA);
        const T dxs[4] = {-(1 - eta), (1 - eta), -eta, eta};
        const T dys[4] = {-(1 - xi), -xi, (1 - xi), xi};
        const T Ns[4] = {(1 - xi) * (1 - eta), xi * (1 - eta), (1 - xi) * eta, xi * eta};
        if (OP == OP_UU_DIAG) {
          const P gq = pfma(omk, pmul(phitq[q1][q2], phitq[q1][q2]), bc<P>(m.kap));
          const P jg = pmul(pmul(bc<P>(g.jxw), gq), ec);
#pragma unroll
          for (int A = 0; A < 4; ++A) {
            const T dx = dxs[A] * g.ihx, dyy = dys[A] * g.ihy;
            rux[A] = pfma(jg, bc<P>(m.c2ml * dx * dx + m.cm * dyy * dyy), rux[A]);
            ruy[A] = pfma(jg, bc<P>(m.cm * dx * dx + m.c2ml * dyy * dyy), ruy[A]);
          }
        } else {
          const P ge12 = shear(fux, q1, uxy, uyx[q2]);
          const P s11 = pfma(c2ml, e11[q2], pmul(cl, e22[q1]));
          const P s22 = pfma(cl, e11[q2], pmul(c2ml, e22[q1]));
          const P s12 = pmul(cm, ge12);
          const P se = pfma(s11, e11[q2], pfma(s22, e22[q1], pmul(s12, ge12)));
          const P mq = pfma(omk, se, pfma(bc<P>(m.p2), padd(e11[q2], e22[q1]), bc<P>(m.gcl)));
#pragma unroll
          for (int A = 0; A < 4; ++A) {
            const T dx = dxs[A] * g.ihx, dyy = dys[A] * g.ihy;
            const P w = pfma(mq, bc<P>(Ns[A] * Ns[A]), bc<P>(m.gcL * (dx * dx + dyy * dyy)));
            rp[A] = f64 ? pfma(bc<P>(g.jxw), w, rp[A]) : padd(rp[A], pmul(bc<P>(g.jxw), w));
          }
        }
      }
  } else {
    P S11[2][2], S12[2][2], S22[2][2], fv[2][2], G[2][2], U11[2][2], U12[2][2], U22[2][2];
    // q = (1-kappa) sigma(u) + p I, so that the phi rows' coefficients are
    //   (1-kappa) sigma(u):e(u) + 2 p div u + G_c/l = q : e(u) + p div u + G_c/l,
    //   2 phi ((1-kappa) sigma(u) + p I) = 2 phi q
    P oc2ml = zero, ocl = zero, ocm = zero;
    if (N::linU) { oc2ml = pmul(omk, c2ml); ocl = pmul(omk, cl); ocm = pmul(omk, cm); }
#pragma unroll
    for (int q1 = 0; q1 < 2; ++q1)
#pragma unroll
      for (int q2 = 0; q2 < 2; ++q2) {
        P gq = zero, T11 = zero, T22 = zero, T12 = zero, mq = zero;
        if (N::phit) gq = pfma(omk, pmul(phitq[q1][q2], phitq[q1][q2]), bc<P>(m.kap));
        if (N::linU) {
          const P pp = bc<P>(m.p);
          const P ge12 = shear(fux, q1, uxy, uyx[q2]);   // 2 e12
          const P q11 = pfma(oc2ml, e11[q2], pfma(ocl, e22[q1], pp));
          const P q22 = pfma(ocl, e11[q2], pfma(oc2ml, e22[q1], pp));
          const P q12 = pmul(ocm, ge12);
          mq = pfma(q11, e11[q2], pfma(q22, e22[q1], pfma(q12, ge12, pfma(pp, padd(e11[q2], e22[q1]), bc<P>(m.gcl)))));
          if (N::phi) {
            const P tp = padd(phiq[q1][q2], phiq[q1][q2]);
            T11 = pmul(tp, q11);
            T22 = pmul(tp, q22);
            T12 = pmul(tp, q12);
          }
        }
        if (N::xu) {
          const P gxy = shear(fxu, q1, bxy, cyx[q2]);
          const P t11 = pfma(c2ml, ax[q2], pmul(cl, dy[q1])), t22 = pfma(cl, ax[q2], pmul(c2ml, dy[q1])), t12 = pmul(cm, gxy);
          P s11 = pmul(gq, t11);
          P s22 = pmul(gq, t22);
          P s12 = pmul(gq, t12);
          G[q1][q2] = gq; U11[q1][q2] = t11; U22[q1][q2] = t22; U12[q1][q2] = t12;
          if (OP == OP_FULL_T) {
            s11 = pfma(xpq[q1][q2], T11, s11);
            s22 = pfma(xpq[q1][q2], T22, s22);
            s12 = pfma(xpq[q1][q2], T12, s12);
          }
          S11[q1][q2] = s11; S12[q1][q2] = s12; S22[q1][q2] = s22;
          if (OP == OP_FULL) fv[q1][q2] = pfma(T11, ax[q2], pfma(T22, dy[q1], pfma(T12, gxy, pmul(mq, xpq[q1][q2]))));
        }
        if (N::xp && OP != OP_FULL) fv[q1][q2] = pmul(mq, xpq[q1][q2]);
      }
    const P wx = bc<P>(g.wx), wy = bc<P>(g.wy), nwx = bc<P>(-g.wx), nwy = bc<P>(-g.wy);
    if (f64 && (OP == OP_FULL || OP == OP_UU)) {
      auto sum = [&](const P (*U)[2], const P (*S)[2], int a, int b, int c, int d) {
        return pfma(G[a][b], U[a][b], S[c][d]);
      };
      ptest_grad(sum(U11, S11, 0, 0, 1, 0), sum(U11, S11, 0, 1, 1, 1), sum(U12, S12, 0, 0, 0, 1),
                 sum(U12, S12, 1, 1, 1, 0), wx, wy, nwx, nwy, rux);
      ptest_grad(sum(U12, S12, 0, 0, 1, 0), sum(U12, S12, 0, 1, 1, 1), sum(U22, S22, 0, 0, 0, 1),
                 sum(U22, S22, 1, 0, 1, 1), wx, wy, nwx, nwy, ruy);
    } else if (N::xu) {
      // u_x test: (S11, S12) . grad psi;  u_y test: (S12, S22) . grad psi
      ptest_grad(padd(S11[0][0], S11[1][0]), padd(S11[0][1], S11[1][1]),
                 padd(S12[0][0], S12[0][1]), padd(S12[1][0], S12[1][1]), wx, wy, nwx, nwy, rux);
      ptest_grad(padd(S12[0][0], S12[1][0]), padd(S12[0][1], S12[1][1]),
                 padd(S22[0][0], S22[0][1]), padd(S22[1][0], S22[1][1]), wx, wy, nwx, nwy, ruy);
    }
    if (N::xp) {
      // value test against N_A = L_a(xi) L_b(eta)
      const P jxw = bc<P>(g.jxw);
      const P s0 = padd(fv[0][0], fv[0][1]), s1 = padd(fv[1][0], fv[1][1]);
      const P t0 = pfma(bc<P>(T(GA)), fv[0][0], pmul(bc<P>(T(GB)), fv[0][1]));
      const P t1 = pfma(bc<P>(T(GA)), fv[1][0], pmul(bc<P>(T(GB)), fv[1][1]));
      const P b0 = psub(s0, t0), b1 = psub(s1, t1);
      const P pb = pfma(bc<P>(T(GA)), b0, pmul(bc<P>(T(GB)), b1));
      const P pt = pfma(bc<P>(T(GA)), t0, pmul(bc<P>(T(GB)), t1));
      rp[0] = pfma(jxw, psub(padd(b0, b1), pb), rp[0]);
      rp[1] = pfma(jxw, pb, rp[1]);
      rp[2] = pfma(jxw, psub(padd(t0, t1), pt), rp[2]);
      rp[3] = pfma(jxw, pt, rp[3]);
      // G_c l (grad dphi, grad psi): the reference d/dxi flux is the same at both
      // xi points, the d/deta flux at both eta points (factor 2 is in wpx, wpy)
      ptest_grad(fxp.dxi[0], fxp.dxi[1], fxp.deta[0], fxp.deta[1], bc<P>(g.wpx), bc<P>(g.wpy), bc<P>(-g.wpx),
                 bc<P>(-g.wpy), rp);
    }
  }
#pragma unroll
  for (int A = 0; A < 4; ++A) {
    out[3 * A + 0] = rux[A];
    out[3 * A + 1] = ruy[A];
    out[3 * A + 2] = rp[A];
  }
}

}  // namespace pff
