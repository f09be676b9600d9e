// Q2 elements (k = 2) on the brick layout: one thread per cell of a brick window.
// Included by apply.cu inside its anonymous namespace (uses its field helpers,
// storage codes and write_node).
//
// Same operators as the Q1 kernel (Sec. 3.1 Jacobian and its transpose, the
// diagonal blocks and their diagonals of Sec. 3.2, the residual of Problem 2,
// lumped mass, TCV and its gradient, the parameter VJP), with the 3x3 Gauss rule.
//
// A brick owns 30 x 30 node slots = 15 x 15 Q2 cells; its window holds the
// 33 x 33 nodes -2..30 and the 16 x 16 cells -1..14 (all cells touching an
// owned node).  A block of 256 threads takes one brick at a time:
//   1. the window's node fields go to shared memory, one plane per field (hanging values
//      from their parents, fixed input components masked, absent nodes zero);
//   2. each thread evaluates one cell, sum-factorised: per Gauss row eta_q2 the
//      3x3 nodal values collapse to three column values, then to the row's
//      three Gauss points; the test runs the same two steps backwards.  Fields
//      that take the same contractions travel as pairs (u_x with u_y of the
//      input and of the linearisation, the input dphi with phi), one paired
//      FP32 instruction for both;
//   3. the cells write their contributions to shared memory, one column per cell, and a
//      thread sums them for the four owned nodes (2i, 2j) .. (2i + 1, 2j + 1): the cells
//      around a node in the order (even column, even row), (odd, even), (even, odd),
//      (odd, odd), so every nodal sum has a fixed order (the FP64 Jacobian: below,
//      below-left, left, own);
//   4. the owned nodes are written (constraint rows, partial sums, holes; pairs of
//      unconstrained nodes of regular bricks as one 8-byte store in FP32), or for the
//      level block operators the fused Chebyshev step of ChebEpi.

// Measured (Jacobian FP32, 16.4M DoFs, the same vectors every call): 212 us with single-value
// copies, colour phases and plain contractions; 176 us in this form (rotating vectors: 204 and
// 158), with half the error against 64 bits.  16 warps
// an SM wait in turn for the window, the barriers and the stores of irregular bricks
// (issue slots 36% busy); the vectors and the linearisation take 32 us at the copy rate.

constexpr int Q2NB = 30;          // owned node slots per side
constexpr int Q2W = 33;           // window nodes per side (-2..30)
constexpr int Q2C = 16;           // window cells per side (-1..14)
constexpr int Q2T = Q2C * Q2C;    // threads per block: one per window cell
constexpr int Q2WW = Q2W * Q2W;

// Field pairs of the window tiles: pair 0 (u_x, u_y of the input), 1 (u_x, u_y
// of the linearisation), 2 (input dphi, phi), 3 (phi_tilde, unused).
constexpr int Q2NP = 4;
__host__ __device__ constexpr int q2_pair(int f) {
  return f == F_XU || f == F_XV ? 0 : f == F_LU || f == F_LV ? 1 : f == F_XP || f == F_LP ? 2 : 3;
}
__host__ __device__ constexpr int q2_half(int f) { return f == F_XV || f == F_LV || f == F_LP ? 1 : 0; }
template <int OP>
__device__ __forceinline__ constexpr bool q2_pair_used(int k) {
  return k == 0 ? field_used<OP>(F_XU) || field_used<OP>(F_XV)
       : k == 1 ? field_used<OP>(F_LU) || field_used<OP>(F_LV)
       : k == 2 ? field_used<OP>(F_XP) || field_used<OP>(F_LP) : field_used<OP>(F_LT);
}

// A plane holds the rows -2..30 of columns 0..29 (the brick's own block and, around it in
// the same row order, the last two rows of the brick below and the first row of the one
// above, 32 values), then columns -2, -1, then column 30.  So a regular brick arrives as
// 16-byte copies of contiguous storage but for the two side halos: 248 + 66 copies per
// field instead of 1,089 single values.
constexpr int Q2ROWS = 992;                          // 33 rows of 30, and 2 values past the last
constexpr int Q2LEFT = Q2ROWS, Q2RIGHT = Q2LEFT + 2 * Q2W;
constexpr int Q2PL = Q2RIGHT + Q2W + 1;
// plane offset of window node (wx, wy), wx, wy = 0..32
__device__ __forceinline__ int q2_at(int wx, int wy) {
  return wx < 2 ? Q2LEFT + 2 * wy + wx : wx == Q2W - 1 ? Q2RIGHT + wy : wx - 2 + Q2NB * wy;
}

// FP32 keeps two window buffers: while a block computes one brick, the window
// of its next brick streams into the other with cp.async.  FP64 (twice the bytes
// per field) keeps one and gathers each brick in turn.
template <typename T>
struct Q2Smem {
  using P = typename VT<T>::T2;
  static constexpr int NBUF = sizeof(T) == 4 ? 2 : 1;
  alignas(16) T f[NBUF][NF][Q2PL];   // node fields of the window
  P conu[9][Q2T];           // contributions of the window's cells by local node: u_x and u_y
  T conp[9][Q2T];           // phi
  // constraint-mask bytes: the plane layout's rows, then the aligned words that hold
  // columns -2, -1 and column 30 of each window row
  alignas(16) uint8_t cm[NBUF][Q2ROWS + 4 * 2 * Q2W];
  alignas(16) int32_t own[NBUF][Q2NB * Q2NB];   // irregular bricks: DevLayout::own of the owned slots
  int32_t nb[3][9];         // storage bases of the 3x3 neighbour bricks of three bricks in turn
};

// Nodes (a, b) of window cell (ci, cj): value pair k (q2_pair) of the fields OP reads.
template <typename T, int OP>
struct Q2Node {
  using P = typename VT<T>::T2;
  const T* pl;
  int o[3], st[3];   // per column a: plane offset of its node (a, 0), and the row stride
  __device__ __forceinline__ void at(int ci, int cj) {
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const int wx = 2 * ci + a;
      o[a] = q2_at(wx, 2 * cj);
      st[a] = wx < 2 ? 2 : wx == Q2W - 1 ? 1 : Q2NB;
    }
  }
  template <int F>
  __device__ __forceinline__ T field(int e) const {
    if constexpr (field_used<OP>(F)) return pl[F * Q2PL + e]; else return T(0);
  }
  __device__ __forceinline__ P operator()(int k, int a, int b) const {
    const int e = o[a] + b * st[a];
    return k == 0 ? P{field<F_XU>(e), field<F_XV>(e)} : k == 1 ? P{field<F_LU>(e), field<F_LV>(e)}
         : k == 2 ? P{field<F_XP>(e), field<F_LP>(e)} : P{field<F_LT>(e), T(0)};
  }
};

// Storage slot of node (n, r) (brick-relative, -2..30) of a brick whose
// neighbour bases are nb; the caller guarantees the neighbour exists.
__device__ __forceinline__ int32_t q2_slot(const int32_t* nb, int n, int r) {
  const int dx = n < 0 ? -1 : (n >= Q2NB ? 1 : 0);
  const int dy = r < 0 ? -1 : (r >= Q2NB ? 1 : 0);
  return nb[(dy + 1) * 3 + dx + 1] + (n - dx * Q2NB) + Q2NB * (r - dy * Q2NB);
}

// Quantities of one Gauss point (only those the operator needs are set).
template <typename T>
struct Q2Point {
  T ux, uy, uxx, uxy, uyx, uyy;   // u and grad u (u_i,j = du_i/dx_j)
  T phi, phix, phiy, phit;        // phi, grad phi, phi_tilde
  T ax, bxy, cyx, dy;             // grad of the input du: du_x,x  du_x,y  du_y,x  du_y,y
  T xp, xpx, xpy;                 // input dphi and its gradient
};

// Test coefficients of one Gauss point: component c gets
//   f0[c] psi + fx[c] dpsi/dx + fy[c] dpsi/dy.
template <typename T>
struct Q2Coef {
  T f0[3], fx[3], fy[3];
};

template <typename T, int OP>
__device__ __forceinline__ void q2_point(const Q2Point<T>& q, const MatConst<T>& m, T c2ml, T cl, T cm,
                                         Q2Coef<T>& c, T cell[3]) {
  using N = Needs<OP>;
#pragma unroll
  for (int k = 0; k < 3; ++k) { c.f0[k] = T(0); c.fx[k] = T(0); c.fy[k] = T(0); }
  T gq = T(0), s11 = T(0), s22 = T(0), s12 = T(0), se = T(0), mq = T(0), ge12 = T(0);
  if (N::phit) gq = m.omk * q.phit * q.phit + m.kap;
  if (N::linU) {
    ge12 = q.uxy + q.uyx;
    s11 = c2ml * q.uxx + cl * q.uyy;
    s22 = cl * q.uxx + c2ml * q.uyy;
    s12 = cm * ge12;
    se = s11 * q.uxx + s22 * q.uyy + s12 * ge12;
    mq = m.omk * se + m.p2 * (q.uxx + q.uyy) + m.gcl;
  }
  if constexpr (OP == OP_UU) {
    const T bc = q.bxy + q.cyx;
    const T S11 = gq * (c2ml * q.ax + cl * q.dy);
    const T S22 = gq * (cl * q.ax + c2ml * q.dy);
    const T S12 = gq * (cm * bc);
    c.fx[0] = S11; c.fy[0] = S12;
    c.fx[1] = S12; c.fy[1] = S22;
  } else if constexpr (OP == OP_PP) {
    c.f0[2] = mq * q.xp;
    c.fx[2] = m.gcL * q.xpx;
    c.fy[2] = m.gcL * q.xpy;
  } else if constexpr (OP == OP_MASS) {
    c.f0[2] = T(1);
  } else if constexpr (OP == OP_TCV) {
    c.f0[2] = q.ux * q.phix + q.uy * q.phiy;
  } else if constexpr (OP == OP_TCV_GRAD) {
    c.f0[0] = q.phix;
    c.f0[1] = q.phiy;
    c.fx[2] = q.ux;
    c.fy[2] = q.uy;
  } else if constexpr (OP == OP_PHIT_VJP) {
    const T sw = s11 * q.ax + s22 * q.dy + s12 * (q.bxy + q.cyx);
    c.f0[2] = T(2) * q.phit * (m.omk * sw + m.p * (q.ax + q.dy));
  } else if constexpr (OP == OP_VJP) {
    // per cell: E_K, p and G_c derivatives of x . R (unit-modulus constants in m)
    const T u11 = m.c2ml * q.uxx + m.cl * q.uyy, u22 = m.cl * q.uxx + m.c2ml * q.uyy, u12 = m.cm * ge12;
    const T use = u11 * q.uxx + u22 * q.uyy + u12 * ge12;
    const T sw = u11 * q.ax + u22 * q.dy + u12 * (q.bxy + q.cyx);
    cell[0] = gq * sw + m.omk * q.phi * use * q.xp;
    cell[1] = q.phit * q.phit * (q.ax + q.dy) + T(2) * q.phi * (q.uxx + q.uyy) * q.xp;
    cell[2] = m.l * (q.phix * q.xpx + q.phiy * q.xpy) - m.il * (T(1) - q.phi) * q.xp;
  }
  (void)se;
}

// One Q2 cell, its node (a, b) (a along x, b along y) read by ld.  Contributions to node
// A = a + 3 b: ru[A] (components u_x, u_y) and rp[A] (phi).  cell[]: per-cell values (OP_VJP).
template <typename T, int OP, class Load>
__device__ __forceinline__ void q2_cell(const Load& ld, const MatConst<T>& m, const LevGeom<T>& g, const Q2Tab<T>& tb, T ec, typename VT<T>::T2 ru[9],
                                        T rp[9], T cell[3]) {
  using N = Needs<OP>;
  using P = typename VT<T>::T2;
  constexpr bool isDiag = (OP == OP_UU_DIAG || OP == OP_PP_DIAG);
  const T c2ml = m.c2ml * ec, cl = m.cl * ec, cm = m.cm * ec;
  const T area = T(4) * g.jxw;   // hx hy
#pragma unroll
  for (int k = 0; k < 9; ++k) { ru[k] = pbc(T(0)); rp[k] = T(0); }
  cell[0] = cell[1] = cell[2] = T(0);
#pragma unroll
  for (int q2 = 0; q2 < 3; ++q2) {
    // collapse every used pair along eta: V[a] = sum_b l_b(eta) v_ab, E[a] = sum_b l_b'(eta) v_ab
    // (pair 3 holds phi_tilde alone, whose value is all the point needs: no E)
    P V[Q2NP][3], E[Q2NP - 1][3];
#pragma unroll
    for (int k = 0; k < Q2NP; ++k) {
      if (!q2_pair_used<OP>(k)) continue;
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        const P v0 = ld(k, a, 0), v1 = ld(k, a, 1), v2 = ld(k, a, 2);
        V[k][a] = pfma(pbc(tb.L[2][q2]), v2, pfma(pbc(tb.L[1][q2]), v1, pmul(pbc(tb.L[0][q2]), v0)));
        if (k < Q2NP - 1)
          E[k][a] = pfma(pbc(tb.D[2][q2]), v2, pfma(pbc(tb.D[1][q2]), v1, pmul(pbc(tb.D[0][q2]), v0)));
      }
    }
    // test sums per node column a: value/x-gradient part and y-gradient part
    P RvU[3], ReU[3];
    T Rvp[3], Rep[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) { RvU[a] = pbc(T(0)); ReU[a] = pbc(T(0)); Rvp[a] = T(0); Rep[a] = T(0); }
#pragma unroll
    for (int q1 = 0; q1 < 3; ++q1) {
      auto val = [&](int k) {
        return pfma(pbc(tb.L[2][q1]), V[k][2], pfma(pbc(tb.L[1][q1]), V[k][1], pmul(pbc(tb.L[0][q1]), V[k][0])));
      };
      auto ddx = [&](int k) {
        return pmul(pfma(pbc(tb.D[2][q1]), V[k][2], pfma(pbc(tb.D[1][q1]), V[k][1], pmul(pbc(tb.D[0][q1]), V[k][0]))),
                    pbc(g.ihx));
      };
      auto ddy = [&](int k) {
        return pmul(pfma(pbc(tb.L[2][q1]), E[k][2], pfma(pbc(tb.L[1][q1]), E[k][1], pmul(pbc(tb.L[0][q1]), E[k][0]))),
                    pbc(g.ihy));
      };
      Q2Point<T> q{};
      if (N::xu) {
        const P dx = ddx(0), dy = ddy(0);
        q.ax = dx.x; q.bxy = dy.x; q.cyx = dx.y; q.dy = dy.y;
      }
      if (N::xp || N::phi) {
        const P v = val(2), dx = ddx(2), dy = ddy(2);
        if (N::xp) { q.xp = v.x; q.xpx = dx.x; q.xpy = dy.x; }
        if (N::phi) { q.phi = v.y; q.phix = dx.y; q.phiy = dy.y; }
      }
      if (N::linU) {
        const P dx = ddx(1), dy = ddy(1);
        q.uxx = dx.x; q.uxy = dy.x; q.uyx = dx.y; q.uyy = dy.y;
        if (OP == OP_TCV || OP == OP_TCV_GRAD) {
          const P v = val(1);
          q.ux = v.x; q.uy = v.y;
        }
      }
      if (N::phit) q.phit = val(3).x;
      const T W = area * tb.w[q1] * tb.w[q2];
      if constexpr (isDiag) {
        // diagonal of the element matrix of the block
        T gq = T(0), mq = T(0);
        if (OP == OP_UU_DIAG) gq = m.omk * q.phit * q.phit + m.kap;
        if (OP == OP_PP_DIAG) {
          const T ge12 = q.uxy + q.uyx;
          const T s11 = c2ml * q.uxx + cl * q.uyy, s22 = cl * q.uxx + c2ml * q.uyy, s12 = cm * ge12;
          mq = m.omk * (s11 * q.uxx + s22 * q.uyy + s12 * ge12) + m.p2 * (q.uxx + q.uyy) + m.gcl;
        }
#pragma unroll
        for (int b = 0; b < 3; ++b)
#pragma unroll
          for (int a = 0; a < 3; ++a) {
            const T Nv = tb.L[a][q1] * tb.L[b][q2];
            const T dxn = tb.D[a][q1] * tb.L[b][q2] * g.ihx, dyn = tb.L[a][q1] * tb.D[b][q2] * g.ihy;
            const int A = a + 3 * b;
            if (OP == OP_UU_DIAG) {
              ru[A].x += W * gq * (c2ml * dxn * dxn + cm * dyn * dyn);
              ru[A].y += W * gq * (cm * dxn * dxn + c2ml * dyn * dyn);
            } else {
              rp[A] += W * (mq * Nv * Nv + m.gcL * (dxn * dxn + dyn * dyn));
            }
          }
      } else if constexpr (OP == OP_VJP) {
        Q2Coef<T> cf;
        T cv[3];
        q2_point<T, OP>(q, m, c2ml, cl, cm, cf, cv);
        cell[0] += W * cv[0];
        cell[1] += W * cv[1];
        cell[2] += W * cv[2];
      } else {
        Q2Coef<T> cf;
        T cv[3];
        q2_point<T, OP>(q, m, c2ml, cl, cm, cf, cv);
        const T wx = W * g.ihx, wy = W * g.ihy;
        P f0u, fxu, fyu;
        f0u.x = W * cf.f0[0]; f0u.y = W * cf.f0[1];
        fxu.x = wx * cf.fx[0]; fxu.y = wx * cf.fx[1];
        fyu.x = wy * cf.fy[0]; fyu.y = wy * cf.fy[1];
        const T f0p = W * cf.f0[2], fxp = wx * cf.fx[2], fyp = wy * cf.fy[2];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
          RvU[a] = pfma(pbc(tb.L[a][q1]), f0u, pfma(pbc(tb.D[a][q1]), fxu, RvU[a]));
          ReU[a] = pfma(pbc(tb.L[a][q1]), fyu, ReU[a]);
          Rvp[a] += tb.L[a][q1] * f0p + tb.D[a][q1] * fxp;
          Rep[a] += tb.L[a][q1] * fyp;
        }
      }
    }
    if constexpr (!isDiag && OP != OP_VJP) {
#pragma unroll
      for (int b = 0; b < 3; ++b)
#pragma unroll
        for (int a = 0; a < 3; ++a) {
          const int A = a + 3 * b;
          ru[A] = pfma(pbc(tb.L[b][q2]), RvU[a], pfma(pbc(tb.D[b][q2]), ReU[a], ru[A]));
          rp[A] += tb.L[b][q2] * Rvp[a] + tb.D[b][q2] * Rep[a];
        }
    }
  }
  if constexpr (OP == OP_VJP) {
    cell[0] = -cell[0]; cell[1] = -cell[1]; cell[2] = -cell[2];
  }
}

template <typename T, int OP>
__global__ void __launch_bounds__(Q2T, sizeof(T) == 4 ? 2 : 1) apply_q2_kernel(const __grid_constant__ BrickArgs<T> a) {
  using P = typename VT<T>::T2;
  constexpr bool isVjp = (OP == OP_VJP);
  constexpr int NBUF = Q2Smem<T>::NBUF;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  Q2Smem<T>& sm = *reinterpret_cast<Q2Smem<T>*>(smem_raw);
  const int tid = threadIdx.x;
  const bool mask = (a.mode & MODE_MASK_INPUT) != 0;
  const MatConst<T>& mc = a.m;
  const Q2Tab<T>& tb = a.q2;
  const int ci = tid % Q2C, cj = tid / Q2C;          // window cell (cell ci - 1, cj - 1)
  Q2Node<T, OP> node;
  node.at(ci, cj);
  const int G = int(gridDim.x);
  constexpr int NWN = (Q2WW + Q2T - 1) / Q2T;   // window nodes per thread
  // Constraint byte of window node (wx, wy) (plane layout of Q2Smem::cm)
  auto cm_at = [&](const uint8_t* cm, int wx, int wy) -> uint32_t {
    if (wx >= 2 && wx < Q2W - 1) return cm[wx - 2 + Q2NB * wy];
    const int r = wy < 2 ? Q2NB - 2 + wy : wy == Q2W - 1 ? 0 : wy - 2;   // brick row of the node's storage
    const int byte = wx < 2 ? (Q2NB * r + Q2NB - 2) % 4 + wx : Q2NB * r % 4;
    return cm[Q2ROWS + 4 * ((wx < 2 ? 0 : Q2W) + wy) + byte];
  };
  // Window of the brick with neighbour bases nb and irregular-table index irn into buffer
  // bu as one group of cp.async; hanging nodes are resolved from their parents, absent
  // ones are zero
  auto prefetch = [&](const int32_t* nb, int irn, int bu) {
    if (irn < 0 && a.wide) {
      constexpr int E = 16 / int(sizeof(T));
      const int32_t below = nb[1], own = nb[4], above = nb[7];
      auto src_of = [&](int v) {
        return v < 2 * Q2NB ? below + Q2NB * (Q2NB - 2) + v
               : v < 2 * Q2NB + Q2NB * Q2NB ? own + v - 2 * Q2NB : above + v - 2 * Q2NB - Q2NB * Q2NB;
      };
      for (int t = tid; t < Q2ROWS / E; t += Q2T) {
        const int32_t src = src_of(t * E);
#pragma unroll
        for (int f = 0; f < NF; ++f)
          if (field_used<OP>(f)) cp_async16(&sm.f[bu][f][t * E], field_ptr<T>(a, f) + src);
      }
      if (tid < Q2ROWS / 4) cp_async4(&sm.cm[bu][4 * tid], a.cmask + src_of(4 * tid));
      // side halos: the fields f = group mod 3, one window row of one side per thread
      const int group = tid / (2 * Q2W), h = tid % (2 * Q2W), wy = h % Q2W, side = h / Q2W;
      const int dy = wy < 2 ? 0 : wy == Q2W - 1 ? 2 : 1, r = wy < 2 ? Q2NB - 2 + wy : wy == Q2W - 1 ? 0 : wy - 2;
      const int32_t src = nb[3 * dy + 2 * side] + Q2NB * r + (side ? 0 : Q2NB - 2);
      if (group < 3) {
#pragma unroll
        for (int f = 0; f < NF; ++f)
          if (field_used<OP>(f) && f % 3 == group) {
            const T* p = field_ptr<T>(a, f) + src;
            if (side) cp_one(&sm.f[bu][f][Q2RIGHT + wy], p);
            else cp_two(&sm.f[bu][f][Q2LEFT + 2 * wy], p);
          }
        if (group == 2) cp_async4(&sm.cm[bu][Q2ROWS + 4 * h], a.cmask + (src & ~3));
      }
      cp_async_commit();
      return;
    }
    if (irn >= 0 && tid < Q2NB * Q2NB / 4)
      cp_async16(&sm.own[bu][4 * tid], a.lay.own + int64_t(irn) * (Q2NB * Q2NB) + 4 * tid);
    int32_t code[NWN];
#pragma unroll
    for (int e = 0; e < NWN; ++e) {
      const int w = tid + Q2T * e;
      code[e] = kAbsent;
      if (w < Q2WW)
        code[e] = irn < 0 ? q2_slot(nb, w % Q2W - 2, w / Q2W - 2) : __ldg(a.lay.win + int64_t(irn) * Q2WW + w);
    }
#pragma unroll
    for (int e = 0; e < NWN; ++e)
      if (code[e] >= 0) {
        const int at = q2_at((tid + Q2T * e) % Q2W, (tid + Q2T * e) / Q2W);
#pragma unroll
        for (int f = 0; f < NF; ++f)
          if (field_used<OP>(f)) cp_one(&sm.f[bu][f][at], field_ptr<T>(a, f) + code[e]);
      }
    uint8_t cm[NWN];
#pragma unroll
    for (int e = 0; e < NWN; ++e) cm[e] = code[e] >= 0 ? __ldg(a.cmask + code[e]) : uint8_t(0);
#pragma unroll
    for (int e = 0; e < NWN; ++e) {
      const int w = tid + Q2T * e;
      if (w >= Q2WW) break;
      const int wx = w % Q2W, wy = w / Q2W;
      if (wx >= 2 && wx < Q2W - 1) {
        sm.cm[bu][wx - 2 + Q2NB * wy] = cm[e];
      } else {
        const int r = wy < 2 ? Q2NB - 2 + wy : wy == Q2W - 1 ? 0 : wy - 2;
        const int byte = wx < 2 ? (Q2NB * r + Q2NB - 2) % 4 + wx : Q2NB * r % 4;
        sm.cm[bu][Q2ROWS + 4 * ((wx < 2 ? 0 : Q2W) + wy) + byte] = cm[e];
      }
      if (code[e] >= 0) continue;
      const int at = q2_at(wx, wy);
      T v[NF];
#pragma unroll
      for (int f = 0; f < NF; ++f) v[f] = T(0);
      if (code[e] != kAbsent) {
        const DevHanging& h = a.hang[-2 - code[e]];
#pragma unroll
        for (int f = F_LU; f < NF; ++f)
          if (field_used<OP>(f)) v[f] = ldg(field_ptr<T>(a, f) + h.slot);
        for (int p = 0; p < 3; ++p) {
          const int ps = h.parent[p];
          const T wgt = T(h.weight[p]);
          const uint8_t pc = mask ? __ldg(a.cmask + ps) : uint8_t(0);
#pragma unroll
          for (int f = F_XU; f <= F_XP; ++f)
            if (field_used<OP>(f) && !(pc & (1 << f))) v[f] += wgt * ldg(field_ptr<T>(a, f) + ps);
        }
      }
#pragma unroll
      for (int f = 0; f < NF; ++f)
        if (field_used<OP>(f)) sm.f[bu][f][at] = v[f];
    }
    cp_async_commit();
  };
  int cur = 0;
  // irregular-table index and level of the current and the next brick: read one brick
  // ahead, so that no block waits for them
  auto desc = [&](int bn) -> int2 {
    if (bn >= a.lay.nbricks) return make_int2(0, 0);
    return make_int2(__ldg(&a.lay.bricks[bn].irr), __ldg(&a.lay.bricks[bn].level));
  };
  int2 dc = desc(blockIdx.x), dn = desc(blockIdx.x + G);
  // neighbour bases: of brick number i of this block in sm.nb[i % 3], two bricks ahead
  auto base_of = [&](int bn) { return tid < 9 && bn < a.lay.nbricks ? __ldg(a.lay.bricks[bn].nbr_base + tid) : 0; };
  if (tid < 9) {
    sm.nb[0][tid] = base_of(blockIdx.x);
    sm.nb[1][tid] = base_of(blockIdx.x + G);
  }
  __syncthreads();
  if (NBUF == 2 && int(blockIdx.x) < a.lay.nbricks) prefetch(sm.nb[0], dc.x, 0);
  int turn = 0;
#pragma unroll 1
  for (int b = blockIdx.x; b < a.lay.nbricks; b += G) {
    const int irr = dc.x, level = dc.y;
    node.pl = &sm.f[cur][0][0];
    const int32_t* nbc = sm.nb[turn];
    __syncthreads();   // the previous brick's tiles are no longer read
    if (NBUF == 1) prefetch(nbc, irr, 0);
    // 1. the window: masked input components
    cp_async_wait<0>();
    const uint8_t* cmw = sm.cm[cur];
    if (mask) {
      __syncthreads();   // the constraint bytes come from other threads
#pragma unroll
      for (int e = 0; e < NWN; ++e) {
        const int w = tid + Q2T * e;
        if (w >= Q2WW) break;
        const uint32_t cm = cm_at(cmw, w % Q2W, w / Q2W);
        if (cm) {
          const int at = q2_at(w % Q2W, w / Q2W);
          if (cm & 1) sm.f[cur][F_XU][at] = T(0);
          if (cm & 2) sm.f[cur][F_XV][at] = T(0);
          if (cm & 4) sm.f[cur][F_XP][at] = T(0);
        }
      }
    }
    __syncthreads();
    // the next brick's window streams in while this one computes
    const int2 dnn = desc(b + 2 * G);
    const int32_t nb2 = base_of(b + 2 * G);
    if (NBUF == 2 && b + G < a.lay.nbricks) prefetch(sm.nb[(turn + 1) % 3], dn.x, cur ^ 1);
    // 2. one cell per thread
    bool act = true;
    if (irr >= 0) {
      const int c = ci + Q2C * cj;
      act = (__ldg(a.lay.cellmask + irr * ((Q2T + 31) / 32) + (c >> 5)) >> (c & 31)) & 1u;
    }
    T ec = T(1);
    if (a.ecell != nullptr && act) ec = ldg(reinterpret_cast<const T*>(a.ecell) + q2_slot(nbc, 2 * ci - 2, 2 * cj - 2));
    P ru[9];
    T rp[9], cell[3];
    if (act) {
      if constexpr (OP == OP_FULL || OP == OP_FULL_T)
        if (a.ecell == nullptr) q2_jac<T, OP, false>(node, a.q2m, Q2Own<T>(mc, a.g[level], T(1)), ru, rp);
        else q2_jac<T, OP, true>(node, a.q2m, Q2Own<T>(mc, a.g[level], ec), ru, rp);
      else
        q2_cell<T, OP>(node, mc, a.g[level], tb, ec, ru, rp, cell);
    }
    if constexpr (isVjp) {
      // the brick owns the cells whose lower-left node it owns (cells 0..14)
      if (act && ci >= 1 && cj >= 1) {
        T* co = reinterpret_cast<T*>(a.cell_out);
        const int64_t s = int64_t(nbc[4]) + 2 * (ci - 1) + Q2NB * 2 * (cj - 1);
#pragma unroll
        for (int q = 0; q < 3; ++q) co[q * a.n_slots + s] = cell[q];
      }
    } else {
      // 3. contributions to shared memory, then the owned nodes' sums
      if (!act) {
#pragma unroll
        for (int e = 0; e < 9; ++e) { ru[e] = pbc(T(0)); rp[e] = T(0); }
      }
      constexpr bool outU = OP != OP_PP && OP != OP_PP_DIAG && OP != OP_MASS && OP != OP_TCV && OP != OP_PHIT_VJP;
      constexpr bool outP = OP != OP_UU && OP != OP_UU_DIAG;
#pragma unroll
      for (int e = 0; e < 9; ++e) {
        if (outU) sm.conu[e][tid] = ru[e];
        if (outP) sm.conp[e][tid] = rp[e];
      }
      __syncthreads();
      const int own_base = nbc[4];
      if (tid < 225) {
        const int i = tid % 15, j = tid / 15;
        const int own = (i + 1) + Q2C * (j + 1);   // the window cell above right of node (2i, 2j)
        const bool ox = (i + 1) & 1, oy = (j + 1) & 1;   // its column, row is odd: its neighbour's comes first
#pragma unroll
        for (int py = 0; py < 2; ++py) {
          T y[2][3];
#pragma unroll
          for (int px = 0; px < 2; ++px) {
            // per direction the even cell (first) and the odd one: offset from own, local node
            const int cx0 = px || !ox ? 0 : -1, ax0 = px ? 1 : (ox ? 2 : 0), cx1 = ox ? 0 : -1, ax1 = ox ? 0 : 2;
            const int cy0 = py || !oy ? 0 : -Q2C, ay0 = py ? 1 : (oy ? 2 : 0), cy1 = oy ? 0 : -Q2C, ay1 = oy ? 0 : 2;
            auto sum = [&](auto (*con)[Q2T]) {
              if constexpr (sizeof(T) == 8 && (OP == OP_FULL || OP == OP_FULL_T)) {
                // the order of the two passes (leaf_cells_q2.cu), which give the same bits
                using V = typename std::remove_reference<decltype(con[0][0])>::type;
                const V none{};
                const V below = py ? none : con[px + 6][own - Q2C], corner = px || py ? none : con[8][own - Q2C - 1],
                        left = px ? none : con[2 + 3 * py][own - 1];
                return padd(padd(padd(below, corner), left), con[px + 3 * py][own]);
              }
              auto v = con[ax0 + 3 * ay0][own + cx0 + cy0];
              if (!px) v = padd(v, con[ax1 + 3 * ay0][own + cx1 + cy0]);
              if (!py) {
                v = padd(v, con[ax0 + 3 * ay1][own + cx0 + cy1]);
                if (!px) v = padd(v, con[ax1 + 3 * ay1][own + cx1 + cy1]);
              }
              return v;
            };
            const P yu = outU ? sum(sm.conu) : P{T(0), T(0)};
            y[px][0] = yu.x;
            y[px][1] = yu.y;
            y[px][2] = outP ? sum(sm.conp) : T(0);
          }
          // 4. owned nodes (level block operators: or the fused Chebyshev store)
          const int oi = 2 * i, oj = 2 * j + py, o = oi + Q2NB * oj;
          const uint8_t cm0 = cmw[oi + Q2NB * (oj + 2)], cm1 = cmw[oi + 1 + Q2NB * (oj + 2)];
          // storage actions and partial sums of irregular bricks
          const uint32_t w0 = irr >= 0 ? uint32_t(sm.own[cur][o]) : uint32_t(kActFinal) << 30,
                         w1 = irr >= 0 ? uint32_t(sm.own[cur][o + 1]) : uint32_t(kActFinal) << 30;
          bool done = false;
          if constexpr (OP == OP_UU || OP == OP_PP) {
            if (a.ch.mode != CHEB_OFF) {
#pragma unroll
              for (int px = 0; px < 2; ++px) {
                const int act_s = int((px ? w1 : w0) >> 30);
                ChebOps<T, OP> co;
                cheb_load<T, OP>(a, own_base + o + px, co);
                cheb_store<T, OP>(a, own_base + o + px, act_s, px ? cm1 : cm0, y[px][0], y[px][1], y[px][2], co);
              }
              done = true;
            }
          }
          if (!done && irr < 0 && (cm0 | cm1) == 0) {
            T* yu = reinterpret_cast<T*>(a.yu) + own_base + o;
            T* yp = reinterpret_cast<T*>(a.yp) + own_base + o;
            if (a.pair_store) {   // even slots of 8-byte (FP64: 16-byte) aligned vectors
              if (outU) {
                *reinterpret_cast<P*>(yu) = P{y[0][0], y[1][0]};
                *reinterpret_cast<P*>(yu + a.n_slots) = P{y[0][1], y[1][1]};
              }
              if (outP) *reinterpret_cast<P*>(yp) = P{y[0][2], y[1][2]};
            } else {
              if (outU) { yu[0] = y[0][0]; yu[1] = y[1][0]; yu[a.n_slots] = y[0][1]; yu[a.n_slots + 1] = y[1][1]; }
              if (outP) { yp[0] = y[0][2]; yp[1] = y[1][2]; }
            }
          } else if (!done) {
            store_owned<T, OP>(a, own_base + o, int(w0 >> 30), int(w0 & 0x3fffffffu) - 1, cm0, y[0][0], y[0][1], y[0][2]);
            store_owned<T, OP>(a, own_base + o + 1, int(w1 >> 30), int(w1 & 0x3fffffffu) - 1, cm1, y[1][0], y[1][1],
                               y[1][2]);
          }
        }
      }
    }
    dc = dn;
    dn = dnn;
    if (tid < 9) sm.nb[(turn + 2) % 3][tid] = nb2;
    turn = (turn + 1) % 3;
    if (NBUF == 2) cur ^= 1;
  }
  cp_async_wait<0>();
}

template <typename T>
cudaError_t launch_apply_q2(const ApplyArgs& a, int op, cudaStream_t s) {
  const size_t smem = sizeof(Q2Smem<T>);
  auto grid_of = [&](const void* fn) -> unsigned {
    const int full = resident_blocks(fn, Q2T, smem);
    return unsigned(a.lay.nbricks < full ? a.lay.nbricks : full);
  };
  const BrickArgs<T> k = brick_args<T>(a);
  auto go = [&](auto fn) {
    fn<<<grid_of(reinterpret_cast<const void*>(fn)), Q2T, smem, s>>>(k);
    return cudaGetLastError();
  };
  if constexpr (sizeof(T) == 8) {   // formed in FP64 only
    switch (op) {
      case OP_UU_DIAG: return go(&apply_q2_kernel<T, OP_UU_DIAG>);
      case OP_PP_DIAG: return go(&apply_q2_kernel<T, OP_PP_DIAG>);
      case OP_MASS: return go(&apply_q2_kernel<T, OP_MASS>);
      case OP_TCV: return go(&apply_q2_kernel<T, OP_TCV>);
      case OP_TCV_GRAD: return go(&apply_q2_kernel<T, OP_TCV_GRAD>);
      case OP_VJP: return go(&apply_q2_kernel<T, OP_VJP>);
      case OP_PHIT_VJP: return go(&apply_q2_kernel<T, OP_PHIT_VJP>);
      default: break;
    }
  }
  switch (op) {
    case OP_FULL: return go(&apply_q2_kernel<T, OP_FULL>);
    case OP_FULL_T: return go(&apply_q2_kernel<T, OP_FULL_T>);
    case OP_UU: return go(&apply_q2_kernel<T, OP_UU>);
    case OP_PP: return go(&apply_q2_kernel<T, OP_PP>);
    default: return cudaErrorInvalidValue;
  }
}
