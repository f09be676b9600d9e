// Set-up of all levels of the Q1 multigrid in shared launches (Sec. 3.2 of Kolditz & Wick,
// arXiv 2404.03265): inverse diagonals (FP64) and the eigenvalue estimates' CG runs with
// FP32 applies.
//
// Why: each (block, level) is a chain of a diagonal apply and 12 CG steps, small launches
// that depend on each other.  As one branch per level of a graph they were 1,300 nodes,
// and the graph took 2.5 ms on a 13-level crack mesh, about 2 us a node, with the chip
// idle.  The levels do not depend on each other, so a launch takes one stage of all of
// them: 37 launches for a block's CG runs.  Measured: set-up and both first V-cycles on
// that mesh 3.10 -> 2.57 ms, what bounds it being those chains and the coarse inversion's.
//
// A block of the apply takes a tile of 15 x 15 nodes (16 x 16 cells, a pair per thread):
// it forms p = z + beta p_old on the tile and its halo and applies the operator to p
// rounded to FP32 (the sums and order of the column sweep).  The dots keep the partition
// and order that they have in a chain of its own (mg.cu): a run that exhausts the Krylov
// space of a level with few free entries hands the rounding of its dots on to lambda_max,
// so another order would give another estimate there.
#include "cheb.cuh"
#include "pdl.cuh"
#include "q1_cell.cuh"
#include "smooth.cuh"
#include "tile_cell.cuh"

namespace pff {

namespace {

using namespace tile;

constexpr int NB = 30, SLOTS = NB * NB;
constexpr int TN = kSetupTile, NW = TN + 2, CW = TN + 1, HC = CW / 2;   // window nodes and cells per side, rows of a half
constexpr int TPB = CW * HC;                                            // a cell pair per thread
constexpr int NPT = (NW * NW + TPB - 1) / TPB;
static_assert(TPB % 32 == 0, "whole warps");

// Slot (on its level) of window node w of the tile, or -1 without a brick
__device__ __forceinline__ int32_t window_slot(const int32_t* tile, int w) {
  const int pos = tile[18];
  const int n = TN * (pos & 7) - 1 + w % NW, r = TN * ((pos >> 3) & 7) - 1 + w / NW;
  const int dx = n < 0 ? 0 : (n >= NB ? 2 : 1), dy = r < 0 ? 0 : (r >= NB ? 2 : 1);
  const int32_t base = tile[3 * dy + dx];
  return base < 0 ? -1 : base + (n - NB * (dx - 1)) + NB * (r - NB * (dy - 1));
}

// ---- inverse diagonals: 1 / diag on interior entries (node, not fixed, not a refinement
// edge), 0 on the others; all levels
template <int OP>
__global__ void __launch_bounds__(TPB) setup_diag_kernel(const __grid_constant__ SetupArgs a) {
  constexpr int NC = OP == OP_UU ? 2 : 1;
  constexpr int DOP = OP == OP_UU ? OP_UU_DIAG : OP_PP_DIAG;
  struct Smem {
    double2 lin[NW * NW];
    double con[NC][4][CW * CW];
    int32_t tile[20];
    uint8_t flag[NW * NW];
  };
  __shared__ Smem sm;
  pdl_wait();
  pdl_trigger();
  const int tid = threadIdx.x;
  if (tid < 20) sm.tile[tid] = __ldg(reinterpret_cast<const int32_t*>(a.tiles + blockIdx.x) + tid);
  __syncthreads();
  const int l = sm.tile[19];
  const int32_t off = a.off[l], n = a.n[l];
  const double* lin = a.lin64 + 4 * int64_t(off);
#pragma unroll
  for (int k = 0; k < NPT; ++k) {
    const int w = tid + TPB * k;
    if (w >= NW * NW) break;
    const int32_t s = window_slot(sm.tile, w);
    const uint8_t f = s >= 0 ? a.flags[off + s] : uint8_t(0);
    double2 v = make_double2(0.0, 0.0);
    if (f & 1) {
      if (OP == OP_UU) v.x = lin[3 * int64_t(n) + s];
      else v = make_double2(lin[s], lin[int64_t(n) + s]);
    }
    sm.lin[w] = v;
    sm.flag[w] = f;
  }
  __syncthreads();
  const LevGeom<double> g = a.gd[l];
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int ci = tid % CW, cj = tid / CW + HC * h, w = ci + NW * cj;
    double out[12];
    const bool act = sm.flag[w] & 32;
    if (act) {
      NodePair<double> v[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const double2 q = sm.lin[w + (e & 1) + NW * (e >> 1)];
        v[e] = NodePair<double>{};
        if (OP == OP_UU) v[e].lw = q.x;
        else { v[e].lx = q.x; v[e].ly = q.y; }
      }
      auto minus = [](const NodePair<double>& p, const NodePair<double>& q) {
        return NodePair<double>{p.x0 - q.x0, p.x1 - q.x1, p.xp - q.xp, p.lx - q.lx, p.ly - q.ly, p.lz - q.lz, p.lw - q.lw};
      };
      const double ec = a.ecell64 != nullptr ? a.ecell64[off + window_slot(sm.tile, w)] : 1.0;
      q1_cell<double, DOP>(v[0], minus(v[1], v[0]), v[2], minus(v[3], v[2]), a.md, g, ec, out);
    }
#pragma unroll
    for (int e = 0; e < 4; ++e)
#pragma unroll
      for (int c = 0; c < NC; ++c)
        sm.con[c][e][ci + CW * cj] = act ? out[3 * e + (OP == OP_UU ? c : 2)] : 0.0;
  }
  __syncthreads();
  for (int o = tid; o < TN * TN; o += TPB) {
    const int wx = o % TN + 1, wy = o / TN + 1, w = wx + NW * wy;
    const uint8_t f = sm.flag[w];
    if (!(f & 1)) continue;
    const int32_t s = window_slot(sm.tile, w);
    const uint8_t cm = a.cmask[off + s];
    const int i = wx + CW * wy;   // the cell above right of the node
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      const double d = padd(padd(padd(sm.con[c][2][i - CW], sm.con[c][3][i - CW - 1]), sm.con[c][1][i - 1]), sm.con[c][0][i]);
      const int bit = OP == OP_UU ? 1 << c : 4;
      const double v = !(f & 8) && !(cm & bit) && d != 0.0 ? 1.0 / d : 0.0;
      const int64_t at = NC * int64_t(off) + c * int64_t(n) + s;
      a.dinv64[at] = v;
      a.dinv32[at] = float(v);
    }
  }
}

// ---- CG beside the apply: start vector r = 1 + 0.01 (splitmix64((gx << 32) | gy) mod
// 1000) / 1000 on interior entries, z = D^-1 r; p . q; r -= alpha q, z = D^-1 r.  A level
// has min(512, ceil(entries / 256)) blocks; its last block to finish adds their partial
// sums in a fixed order and forms the scalars
//   sc: 0 rz, 1 pq, 2 rz_new, 3 alpha, 4 beta, 5 ok.
__device__ __forceinline__ uint64_t splitmix64(uint64_t x) {
  uint64_t z = x + 0x9E3779B97F4A7C15ull;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

constexpr int RT = 256;
enum Stage : int { START = 0, PQ = 1, RZ = 2 };
template <int OP, int STAGE>
__global__ void __launch_bounds__(RT) setup_dot_kernel(const __grid_constant__ SetupArgs a, int step) {
  constexpr int NC = OP == OP_UU ? 2 : 1;
  __shared__ double sh[RT];
  __shared__ bool last;
  pdl_wait();
  pdl_trigger();
  int l = 1;
  while (int(blockIdx.x) >= a.dot0[l + 1]) ++l;
  const int first = a.dot0[l], nb = a.dot0[l + 1] - first, tid = threadIdx.x;
  const int32_t off = a.off[l], n = a.n[l];
  const int64_t v0 = NC * int64_t(off), nn = NC * int64_t(n);
  double* sc = a.sc + 8 * l;
  const double* p = a.p[step & 1] + v0;
  const double alpha = STAGE == RZ ? sc[3] : 0.0;
  double acc = 0.0;
  for (int64_t i = int64_t(int(blockIdx.x) - first) * RT + tid; i < nn; i += int64_t(nb) * RT) {
    if (STAGE == PQ) {
      const double pi = p[i];   // zero off the interior, where q may hold no value
      acc += pi * double(pi != 0.0 ? a.q[v0 + i] : 0.f);
      continue;
    }
    const double di = a.dinv64[v0 + i];
    double ri;
    if (STAGE == START) {
      ri = 0.0;
      const int32_t s = int32_t(i % n), gx = a.gx[off + s], gy = a.gy[off + s];
      if (gx >= 0 && di != 0.0)
        ri = 1.0 + 0.01 * double(splitmix64((uint64_t(uint32_t(gx)) << 32) | uint64_t(uint32_t(gy))) % 1000ull) / 1000.0;
    } else {
      ri = a.r[v0 + i] - alpha * double(di != 0.0 ? a.q[v0 + i] : 0.f);
    }
    const double zi = di * ri;
    a.r[v0 + i] = ri;
    a.z[v0 + i] = zi;
    acc += ri * zi;
  }
  auto tree = [&]() {
    for (int o = RT / 2; o > 0; o >>= 1) {
      if (tid < o) sh[tid] += sh[tid + o];
      __syncthreads();
    }
  };
  sh[tid] = acc;
  __syncthreads();
  tree();
  if (tid == 0) {
    a.partial[blockIdx.x] = sh[0];
    __threadfence();
    last = atomicAdd(a.count + l, 1u) == unsigned(nb) - 1u;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  acc = 0.0;
  for (int b = tid; b < nb; b += RT) acc += __ldcg(a.partial + first + b);
  sh[tid] = acc;
  __syncthreads();
  tree();
  if (tid != 0) return;
  const double total = sh[0];
  a.count[l] = 0u;   // for the next launch
  if (STAGE == START) {
    sc[0] = total;
    sc[4] = 0.0;
    sc[5] = 1.0;
  } else if (STAGE == PQ) {
    sc[1] = total;
    const bool ok = sc[5] > 0.5 && total > 0.0 && sc[0] > 0.0;
    sc[3] = ok ? sc[0] / total : 0.0;
    if (!ok) sc[5] = 0.0;
  } else {
    double* hist = a.hist + int64_t(a.hist_stride) * l;
    sc[2] = total;
    const bool ok = sc[5] > 0.5;
    const double beta = ok ? total / sc[0] : 0.0;
    sc[4] = beta;
    hist[2 * step + 0] = ok ? sc[3] : 0.0;
    hist[2 * step + 1] = beta;
    if (!(ok && total > 1e-300)) sc[5] = 0.0;
    sc[0] = total;
  }
}

// ---- CG: p = z + beta p_old, q = A p
template <int OP>
__global__ void __launch_bounds__(TPB) setup_apply_kernel(const __grid_constant__ SetupArgs a, int step) {
  using V = typename Comp<OP>::V;
  constexpr int NC = Comp<OP>::NC;
  struct Smem {
    union {
      float2 lin[NW * NW];
      V con[4][CW * CW];
    };
    V xs[NW * NW];
    float e[NW * NW];
    int32_t tile[20];
    uint8_t flag[NW * NW];
  };
  __shared__ Smem sm;
  const int tid = threadIdx.x;
  if (tid < 20) sm.tile[tid] = __ldg(reinterpret_cast<const int32_t*>(a.tiles + blockIdx.x) + tid);
  __syncthreads();
  const int l = sm.tile[19];
  const int32_t off = a.off[l], n = a.n[l];
  const int64_t v0 = NC * int64_t(off);
  const float* lin = a.lin32 + 4 * int64_t(off);
  int32_t slot[NPT];
  uint32_t cm[NPT];
  {
    uint8_t f[NPT];
    float2 li[NPT];
    float e[NPT];
#pragma unroll
    for (int k = 0; k < NPT; ++k) {
      const int w = tid + TPB * k;
      const int32_t s = w < NW * NW ? window_slot(sm.tile, w) : -1;
      slot[k] = s;
      const int32_t q = s < 0 ? 0 : s;
      f[k] = a.flags[off + q];
      cm[k] = a.cmask[off + q];
      li[k] = OP == OP_UU ? make_float2(lin[3 * int64_t(n) + q], 0.f) : make_float2(lin[q], lin[int64_t(n) + q]);
      e[k] = a.ecell32 != nullptr ? a.ecell32[off + q] : 1.f;
    }
#pragma unroll
    for (int k = 0; k < NPT; ++k) {
      const int w = tid + TPB * k;
      if (slot[k] < 0 || !(f[k] & 1)) {
        slot[k] = -1;
        f[k] = 0;
        cm[k] = 0;
        li[k] = make_float2(0.f, 0.f);
      }
      if (w < NW * NW) {
        sm.lin[w] = li[k];
        sm.e[w] = (f[k] & 32) ? e[k] : 1.f;
        sm.flag[w] = f[k];
      }
    }
  }
  __syncthreads();
  const int ci = tid % CW, cj = tid / CW, nA = ci + NW * cj, nB = nA + NW * HC;
  const bool actA = sm.flag[nA] & 32, actB = sm.flag[nB] & 32;
  P q[2][2], ec = pbc(1.f);
  if (actA || actB) {
    if (a.ecell32 != nullptr) ec = make_float2(sm.e[nA], sm.e[nB]);
    cell_coef<OP, NW>(sm.lin, nA, nB, a.mf, a.gf[l], ec, q);
  }
  // the tables and the linearisation were there before the first stage; from here on what
  // the preceding launch wrote
  pdl_wait();
  pdl_trigger();
  const double beta = a.sc[8 * l + 4];
  const double* zo = a.z + v0;
  const double* po = a.p[(step + 1) & 1] + v0;
  double* pn = a.p[step & 1] + v0;
  double pv[NPT][NC];
  {
    double zv[NPT][NC];
#pragma unroll
    for (int k = 0; k < NPT; ++k)
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        const int64_t at = c * int64_t(n) + (slot[k] < 0 ? 0 : slot[k]);
        zv[k][c] = zo[at];
        pv[k][c] = step == 0 ? 0.0 : po[at];
      }
#pragma unroll
    for (int k = 0; k < NPT; ++k) {
      const int w = tid + TPB * k;
      V x = V();
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        pv[k][c] = slot[k] < 0 ? 0.0 : step == 0 ? zv[k][c] : __fma_rn(beta, pv[k][c], zv[k][c]);
        comp(x, c) = float(pv[k][c]);
      }
      if (w < NW * NW) sm.xs[w] = x;
    }
  }
  __syncthreads();   // sm.lin is no longer read: sm.con takes its place
  {
    P r[NC][4];
    if (actA || actB) {
      cell_apply<OP, NW>(sm.xs, nA, nB, a.mf, a.gf[l], ec, q, r);
    } else {
#pragma unroll
      for (int c = 0; c < NC; ++c)
#pragma unroll
        for (int e = 0; e < 4; ++e) r[c][e] = pbc(0.f);
    }
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      V vA, vB;
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        comp(vA, c) = actA ? r[c][e].x : 0.f;
        comp(vB, c) = actB ? r[c][e].y : 0.f;
      }
      sm.con[e][ci + CW * cj] = vA;
      sm.con[e][ci + CW * (cj + HC)] = vB;
    }
  }
  __syncthreads();
#pragma unroll
  for (int k = 0; k < NPT; ++k) {
    const int w = tid + TPB * k, wx = w % NW, wy = w / NW;
    if (w < NW * NW && slot[k] >= 0 && wx >= 1 && wx <= TN && wy >= 1 && wy <= TN) {
      const int i = wx + CW * wy;   // the cell above right of the node
      const V c2 = sm.con[2][i - CW], c3 = sm.con[3][i - CW - 1], c1 = sm.con[1][i - 1], c0 = sm.con[0][i];
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        const int bit = OP == OP_UU ? 1 << c : 4;
        float y = ((comp(c2, c) + comp(c3, c)) + comp(c1, c)) + comp(c0, c);
        if (cm[k] & bit) y = 0.f;
        const int64_t at = c * int64_t(n) + slot[k];
        a.q[v0 + at] = y;
        pn[at] = pv[k][c];
      }
    }
  }
}

template <int OP>
cudaError_t launch_cg(const SetupArgs& a, int steps, cudaStream_t s) {
  const int ndot = a.dot0[kMaxLevels];
  if (ndot <= 0 || a.ntiles <= a.tile1) return cudaSuccess;
  SetupArgs b = a;
  b.tiles = a.tiles + a.tile1;   // level 0 takes no part
  b.ntiles = a.ntiles - a.tile1;
  cudaError_t e = launch_ex(true, &setup_dot_kernel<OP, START>, unsigned(ndot), unsigned(RT), 0, s, b, 0);
  for (int j = 0; j < steps && e == cudaSuccess; ++j) {
    e = launch_ex(true, &setup_apply_kernel<OP>, unsigned(b.ntiles), unsigned(TPB), 0, s, b, j);
    if (e == cudaSuccess) e = launch_ex(true, &setup_dot_kernel<OP, PQ>, unsigned(ndot), unsigned(RT), 0, s, b, j);
    if (e == cudaSuccess) e = launch_ex(true, &setup_dot_kernel<OP, RZ>, unsigned(ndot), unsigned(RT), 0, s, b, j);
  }
  return e;
}

}  // namespace

cudaError_t launch_setup_diag(const SetupArgs& a, int op, cudaStream_t s) {
  if (a.ntiles <= 0) return cudaSuccess;
  if (op == OP_UU) return launch_ex(false, &setup_diag_kernel<OP_UU>, unsigned(a.ntiles), unsigned(TPB), 0, s, a);
  if (op == OP_PP) return launch_ex(false, &setup_diag_kernel<OP_PP>, unsigned(a.ntiles), unsigned(TPB), 0, s, a);
  return cudaErrorInvalidValue;
}

cudaError_t launch_setup_cg(const SetupArgs& a, int op, int steps, cudaStream_t s) {
  if (op == OP_UU) return launch_cg<OP_UU>(a, steps, s);
  if (op == OP_PP) return launch_cg<OP_PP>(a, steps, s);
  return cudaErrorInvalidValue;
}

}  // namespace pff
