// Fused level smoothers of the FP32 Q1 V-cycle (Sec. 3.2 of Kolditz & Wick,
// arXiv 2404.03265): a whole smoothing of one level, with its transfer, in one launch.
//
// Down: Chebyshev degree 3 from zero on A x = d, the residual d - A x and its
// restriction into the coarser level.  Up: prolongation of the coarse correction and
// Chebyshev degree 3 on the new residual.  Each does three level applies; a block
// takes a tile of 6, 10 or 15 nodes a side (by the size of the level) and evaluates the
// cells around it that the three applies need (halo 4 down, 3 up), so nothing is
// exchanged between blocks.
//
// Why: level meshes of a crack mesh hold 10^2..10^5 nodes; a launch per apply is a
// chain of ~100 dependent launches of 4-6 us, each a few serial L2 round trips and
// cell rows, with most of the chip idle.  One tile per block needs one round trip
// per level and direction, and the halo's extra cells cost idle issue slots (cells
// evaluated per cell of the tile, down and up: side 15 1.8 and 1.5, side 10 2.3 and 1.7,
// side 6 3.4 and 2.3).  Measured (u block, 1.04M-DoF crack mesh, 13 levels): 101 launches
// and 482 us before; 27 launches (12 down, 12 up, defects, coarse solve, copy out) and
// 135 us with the tiles.
//
// Arithmetic: every cell, nodal sum, smoother step and transfer row is the
// expression and order of sweep_q1_kernel, k_restrict and k_prolong (the transfer
// weights 1, 1/2, 1/4 are exact), so the results are the same bits; cells evaluated
// by two tiles give the same values in both.
//
// Layout in a block: thread t holds the cell pair (i, j), (i, j + CW / 2) as the two
// members of every packed operation, with the pair's Gauss-point coefficients in
// registers for all three applies, and up to NPT window nodes (their defect, inverse
// diagonal and iterates) in registers.  Iterates go through shared memory node by
// node, cell contributions as four corner arrays.
#include "smooth.cuh"

#include "cheb.cuh"
#include "pdl.cuh"
#include "tile_cell.cuh"

namespace pff {

namespace {

using namespace tile;

constexpr int NB = 30;   // node slots per brick side

// TN: nodes per tile side; HW: halo of the window (4 down, 3 up).  Window nodes and
// cells are numbered from the window's corner; cell (i, j) has its lower-left node at
// node (i, j).
template <int OP, bool DOWN, int TN>
struct SmoothSmem {
  static constexpr int HW = DOWN ? 4 : 3;
  static constexpr int NW = TN + 2 * HW;     // window nodes per side
  static constexpr int CW = NW - 1;          // window cells per side
  static constexpr int HC = (CW + 1) / 2;    // cell rows of a pair's first member
  static constexpr int CN = NW / 2 + 2;      // up: coarse nodes under the window, per side
  static constexpr int TPB = (CW * HC + 31) / 32 * 32;
  static constexpr int NPT = (NW * NW + TPB - 1) / TPB;
  static_assert(CN * CN <= TPB && ((TN + 1) / 2) * ((TN + 1) / 2) <= TPB, "one thread per coarse node");
  using V = typename Comp<OP>::V;
  union {
    struct {
      float2 lin[NW * NW];   // UU phi~ in .x, PP u_x, u_y
      float e[NW * NW];      // modulus of the cell whose lower-left node this is
    };
    V con[4][CW * CW];       // cell contributions by corner
  };
  V xs[NW * NW];
  V xc[DOWN ? 1 : CN * CN];
  int32_t tile[20];
  uint8_t cell[NW * NW];     // bit0 the node exists, bit5 the cell whose lower-left node this is exists
};

template <int OP, bool DOWN, int TN>
__global__ void __launch_bounds__(SmoothSmem<OP, DOWN, TN>::TPB, 768 / SmoothSmem<OP, DOWN, TN>::TPB)
smooth_kernel(const __grid_constant__ SmoothArgs a) {
  using S = SmoothSmem<OP, DOWN, TN>;
  using V = typename Comp<OP>::V;
  constexpr int NC = Comp<OP>::NC, HW = S::HW, NW = S::NW, CW = S::CW, NPT = S::NPT, HC = S::HC, TPB = S::TPB;
  constexpr int HB = NB / 2;   // coarse nodes per brick side
  __shared__ S sm;
  const int tid = threadIdx.x;
  if (tid < 20) sm.tile[tid] = __ldg(reinterpret_cast<const int32_t*>(a.tiles + blockIdx.x) + tid);
  __syncthreads();
  const int pos = sm.tile[18];
  const int n0 = TN * (pos & 7) - HW, r0 = TN * ((pos >> 3) & 7) - HW;   // brick position of window node 0
  const int ox = HB * ((pos >> 6) & 1), oy = HB * ((pos >> 7) & 1);      // the brick's corner in its parent brick
  constexpr int fix0 = OP == OP_UU ? 1 : 4;
  // ---- tables and set-up data, which no kernel of the chain writes: window nodes,
  // the cells' factors.  All loads of a thread's nodes are issued together (a position
  // without a brick reads slot 0 and is masked), so a tile pays one round trip.
  int32_t slot[NPT];
  uint32_t cm[NPT];
  V di[NPT];
  {
    uint8_t f[NPT];
    float2 li[NPT];
    float e[NPT];
#pragma unroll
    for (int k = 0; k < NPT; ++k) {
      const int w = tid + TPB * k;
      const int n = n0 + w % NW, r = r0 + w / NW;
      const int dx = n < 0 ? 0 : (n >= NB ? 2 : 1), dy = r < 0 ? 0 : (r >= NB ? 2 : 1);
      const int32_t base = w < NW * NW ? sm.tile[3 * dy + dx] : -1;
      const int32_t s = base < 0 ? 0 : base + (n - NB * (dx - 1)) + NB * (r - NB * (dy - 1));
      f[k] = __ldg(a.flags + s);
      cm[k] = __ldg(a.cmask + s);
#pragma unroll
      for (int c = 0; c < NC; ++c) comp(di[k], c) = __ldg(a.dinv + c * int64_t(a.n) + s);
      li[k] = make_float2(0.f, 0.f);
      if constexpr (OP == OP_UU) {
        li[k].x = __ldg(a.lin + 3 * int64_t(a.n) + s);
      } else {
        li[k].x = __ldg(a.lin + s);
        li[k].y = __ldg(a.lin + int64_t(a.n) + s);
      }
      e[k] = a.ecell != nullptr ? __ldg(a.ecell + s) : 1.f;
      slot[k] = base < 0 ? -1 : s;
    }
#pragma unroll
    for (int k = 0; k < NPT; ++k) {
      const int w = tid + TPB * k;
      if (slot[k] < 0 || !(f[k] & 1)) {
        slot[k] = -1;
        f[k] = 0;
        cm[k] = 0;
        di[k] = V();
        li[k] = make_float2(0.f, 0.f);
      }
      if (w < NW * NW) {
        sm.lin[w] = li[k];
        sm.e[w] = (f[k] & 32) ? e[k] : 1.f;
        sm.cell[w] = f[k] & 33;
      }
    }
  }
  __syncthreads();
  const int ci = tid % CW, cj = tid / CW;
  const bool has = cj < HC;
  const int nA = ci + NW * (has ? cj : 0), nB = has && cj + HC < CW ? nA + NW * HC : nA;   // lower-left nodes of the pair
  const bool hasB = has && cj + HC < CW;
  const bool actA = has && (sm.cell[nA] & 32), actB = hasB && (sm.cell[nB] & 32);
  P q[2][2], ec = pbc(1.f);
  if (actA || actB) {
    if (a.ecell != nullptr) ec = make_float2(sm.e[nA], sm.e[nB]);
    cell_coef<OP, NW>(sm.lin, nA, nB, a.m, a.g, ec, q);
  }
  // ---- level vectors.  The next launch may start once every block is past its wait
  // (the trigger follows it), so a block that runs knows that the launch before the
  // preceding one has completed.  Up: the defect and the pre-smoothed iterate are
  // older than that and are read before the wait, the coarse correction after it.
  V dv[NPT], xv[NPT], xl[NPT];   // defect (then residual), iterate; up: the pre-smoothed iterate
  auto level_loads = [&]() {
#pragma unroll
    for (int k = 0; k < NPT; ++k) {
      const int32_t s = slot[k] < 0 ? 0 : slot[k];
#pragma unroll
      for (int c = 0; c < NC; ++c) comp(dv[k], c) = a.d[c * int64_t(a.n) + s];
      if constexpr (!DOWN) {
#pragma unroll
        for (int c = 0; c < NC; ++c) comp(xl[k], c) = a.x[c * int64_t(a.n) + s];
      }
    }
  };
  if constexpr (!DOWN) level_loads();
  pdl_wait();
  pdl_trigger();
  if constexpr (DOWN) level_loads();
  {
    if constexpr (!DOWN) {
      // the coarse nodes under the window (those without a brick are parents of no window node)
      constexpr int CN = S::CN;
      if (tid < CN * CN) {
        const int gx = (n0 >> 1) + ox + tid % CN, gy = (r0 >> 1) + oy + tid / CN;
        const int dx = gx < 0 ? 0 : (gx >= NB ? 2 : 1), dy = gy < 0 ? 0 : (gy >= NB ? 2 : 1);
        const int32_t base = sm.tile[9 + 3 * dy + dx];
        const int32_t cs = base < 0 ? 0 : base + (gx - NB * (dx - 1)) + NB * (gy - NB * (dy - 1));
        V v;
#pragma unroll
        for (int c = 0; c < NC; ++c) comp(v, c) = a.xc[c * int64_t(a.nc) + cs];
        sm.xc[tid] = v;
      }
      __syncthreads();
    }
#pragma unroll
    for (int k = 0; k < NPT; ++k) {
      const int w = tid + TPB * k;
      const bool node = slot[k] >= 0;
      if (!node) dv[k] = V();
      if constexpr (DOWN) {
#pragma unroll
        for (int c = 0; c < NC; ++c) comp(xv[k], c) = cheb_first_of(a.c0, comp(di[k], c), comp(dv[k], c));
      } else {
        // x + P xc: the row's coarse nodes in ascending (y, x), zero weights left out
        constexpr int CN = S::CN;
        xv[k] = V();
        if (node) {
          const int n = n0 + w % NW, r = r0 + w / NW;
          const int q = (n >> 1) - (n0 >> 1) + CN * ((r >> 1) - (r0 >> 1));
          const bool nx = n & 1, ny = r & 1;
          const float wt = (nx ? 0.5f : 1.f) * (ny ? 0.5f : 1.f);
          const int qx = nx ? q + 1 : q, qy = ny ? q + CN : q;
          const V p0 = sm.xc[q], p1 = sm.xc[qx], p2 = sm.xc[qy], p3 = sm.xc[qx + qy - q];
#pragma unroll
          for (int c = 0; c < NC; ++c) {
            float acc = comp(xl[k], c);
            acc += wt * comp(p0, c);
            if (nx) acc += wt * comp(p1, c);
            if (ny) acc += wt * comp(p2, c);
            if (nx && ny) acc += wt * comp(p3, c);
            comp(xv[k], c) = (cm[k] & (fix0 << c)) ? 0.f : acc;
          }
        }
      }
      if (w < NW * NW) sm.xs[w] = xv[k];
    }
  }
  // Down: the restriction's row of this thread.  P^T of the residual goes onto the
  // coarse nodes at the tile's even positions, one per thread.
  // Rows are summed in ascending storage slot: bricks by (row, column), nodes by
  // (row, column) in each; absent nodes add zero.
  int32_t cs = -1, rw = 0;
  uint32_t cmc = 0;
  V dcv = V();
  if constexpr (DOWN) {
    constexpr int TC = (TN + 1) / 2;
    const int wx = HW + 2 * (tid % TC) + (n0 + HW) % 2, wy = HW + 2 * (tid / TC) + (r0 + HW) % 2;   // even brick positions
    if (tid < TC * TC && wx < HW + TN && wy < HW + TN && (sm.cell[wx + NW * wy] & 1)) {
      rw = wx + NW * wy;
      const int n = n0 + wx, r = r0 + wy;
      cs = sm.tile[9 + 4] + (n >> 1) + ox + NB * ((r >> 1) + oy);
      cmc = __ldg(a.cmask_c + cs);
#pragma unroll
      for (int c = 0; c < NC; ++c) comp(dcv, c) = a.dc[c * int64_t(a.nc) + cs];
    }
  }
  __syncthreads();   // sm.lin and sm.e are no longer read: sm.con takes their place
  V pv[NPT], xf[NPT];   // previous iterate; up: the prolonged x
#pragma unroll
  for (int k = 0; k < NPT; ++k) { pv[k] = V(); xf[k] = xv[k]; }
#pragma unroll
  for (int step = 0; step < 3; ++step) {
    const int R = HW - 1 - step;   // nodes within R of the tile are updated from cells within R + 1
    {
      const int lo = HW - R - 1, hi = HW + TN + R - 1;   // window cells per direction
      const bool cx = ci >= lo && ci <= hi;
      const bool inA = has && cx && cj >= lo && cj <= hi, inB = hasB && cx && cj + HC >= lo && cj + HC <= hi;
      if (inA || inB) {
        P r[NC][4];
        if ((inA && actA) || (inB && actB)) {
          cell_apply<OP, NW>(sm.xs, nA, nB, a.m, a.g, ec, q, r);
        } else {
#pragma unroll
          for (int c = 0; c < NC; ++c)
#pragma unroll
            for (int e = 0; e < 4; ++e) r[c][e] = pbc(0.f);
        }
        const int iA = ci + CW * cj, iB = iA + CW * HC;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          V vA, vB;
#pragma unroll
          for (int c = 0; c < NC; ++c) {
            comp(vA, c) = actA ? r[c][e].x : 0.f;
            comp(vB, c) = actB ? r[c][e].y : 0.f;
          }
          sm.con[e][iA] = vA;
          if (hasB) sm.con[e][iB] = vB;
        }
      }
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < NPT; ++k) {
      const int w = tid + TPB * k;
      const int wx = w % NW, wy = w / NW;
      if (w < NW * NW && wx >= HW - R && wx < HW + TN + R && wy >= HW - R && wy < HW + TN + R) {
        const int i = wx + CW * wy;   // the cell above right of the node
        const V c2 = sm.con[2][i - CW], c3 = sm.con[3][i - CW - 1], c1 = sm.con[1][i - 1], c0 = sm.con[0][i];
        V out;
#pragma unroll
        for (int c = 0; c < NC; ++c) {
          const float y = ((comp(c2, c) + comp(c3, c)) + comp(c1, c)) + comp(c0, c);
          const float ye = (slot[k] < 0 || (cm[k] & (fix0 << c))) ? 0.f : y;
          const float dk = comp(dv[k], c), dik = comp(di[k], c), xk = comp(xv[k], c);
          float o;
          if (DOWN ? step == 2 : step == 0) {
            const float rk = dk - ye;
            if (DOWN) {
              o = rk;   // the residual to restrict
            } else {
              comp(dv[k], c) = rk;
              o = cheb_first_of(a.c0, dik, rk);
              comp(pv[k], c) = 0.f;
              comp(xv[k], c) = o;
            }
          } else {
            const bool second = DOWN ? step == 1 : step == 2;
            o = cheb_next(xk, comp(pv[k], c), dik, dk, ye, second ? a.a2 : a.a1, second ? a.b2 : a.b1);
            comp(pv[k], c) = xk;
            comp(xv[k], c) = o;
          }
          comp(out, c) = o;
        }
        if (DOWN || step < 2) sm.xs[w] = out;
        if (step == (DOWN ? 1 : 2)) {
          // the tile's own nodes
          if (slot[k] >= 0 && wx >= HW && wx < HW + TN && wy >= HW && wy < HW + TN) {
#pragma unroll
            for (int c = 0; c < NC; ++c)
              a.xout[c * int64_t(a.n) + slot[k]] = DOWN ? comp(out, c) : comp(xf[k], c) + comp(out, c);
          }
        }
      }
    }
    if (DOWN || step < 2) __syncthreads();
  }
  if constexpr (DOWN) {
    if (cs >= 0) {
      const int w = rw;
      const bool crossx = n0 + rw % NW == 0, crossy = r0 + rw / NW == 0;
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        float v[3][3];
#pragma unroll
        for (int b = 0; b < 3; ++b)
#pragma unroll
          for (int e = 0; e < 3; ++e)
            v[b][e] = ((b == 1 ? 1.f : 0.5f) * (e == 1 ? 1.f : 0.5f)) * comp(sm.xs[w + (e - 1) + NW * (b - 1)], c);
        float acc = comp(dcv, c);
        acc += v[0][0];
        if (crossx && !crossy) {   // the left brick's column first
          acc += v[1][0];
          acc += v[2][0];
          acc += v[0][1];
          acc += v[0][2];
        } else {
          acc += v[0][1];
          acc += v[0][2];
          acc += v[1][0];
          if (crossx) acc += v[2][0];
        }
        acc += v[1][1];
        acc += v[1][2];
        if (!crossx) acc += v[2][0];
        acc += v[2][1];
        acc += v[2][2];
        a.dc[c * int64_t(a.nc) + cs] = (cmc & (fix0 << c)) ? 0.f : acc;
      }
    }
  }
}

template <bool DOWN, int TN>
cudaError_t launch_tile(const SmoothArgs& a, int op, cudaStream_t s, bool pdl) {
  constexpr unsigned tpb = SmoothSmem<OP_UU, DOWN, TN>::TPB;
  if (op == OP_UU) return launch_ex(pdl, &smooth_kernel<OP_UU, DOWN, TN>, unsigned(a.ntiles), tpb, 0, s, a);
  if (op == OP_PP) return launch_ex(pdl, &smooth_kernel<OP_PP, DOWN, TN>, unsigned(a.ntiles), tpb, 0, s, a);
  return cudaErrorInvalidValue;
}

template <bool DOWN>
cudaError_t launch_smooth(const SmoothArgs& a, int op, cudaStream_t s, bool pdl) {
  if (a.ntiles <= 0) return cudaSuccess;
  switch (a.tile) {
    case 6: return launch_tile<DOWN, 6>(a, op, s, pdl);
    case 10: return launch_tile<DOWN, 10>(a, op, s, pdl);
    case 15: return launch_tile<DOWN, 15>(a, op, s, pdl);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace

cudaError_t launch_smooth_down(const SmoothArgs& a, int op, cudaStream_t s) {
  return launch_smooth<true>(a, op, s, true);
}
cudaError_t launch_smooth_up(const SmoothArgs& a, int op, cudaStream_t s, bool pdl) {
  return launch_smooth<false>(a, op, s, pdl);
}

}  // namespace pff
