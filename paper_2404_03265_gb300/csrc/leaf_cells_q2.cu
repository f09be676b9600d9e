// Q2 leaf operators in FP64 as two passes over compact lists, as leaf_cells.cu for Q1:
// the leaf cells, then one thread per node slot.
//
// Pass 1 gathers a cell's nine nodes (the input, hanging nodes resolved from their
// parents, into a column of shared memory; the linearisation is read where a Gauss row
// needs it, from L1) and writes 27 nodal contributions; pass 2 adds those of the cells
// around a node in the order ((below + below-left) + left) + own, condenses hanging
// nodes' onto their parents and applies the constraint rows.
//
// Bound by the FP64 rate (a warp instruction occupies its quarter of an SM for 64
// cycles): what counts is the operations per cell (q2_jac.cuh) and that every quarter has
// work until the end.  The brick kernel gives a block of 256 cells to an SM at a time,
// fewer bricks than SMs on small meshes.  The contributions cost 216 bytes per cell
// written and read again.
#include "kernels.cuh"
#include "pdl.cuh"
#include "q2_jac.cuh"

namespace pff {

namespace {

constexpr int NODE_TPB = 256;
constexpr int NB = 30;   // node slots per brick side

// kernel arguments (small ones: they are copied per launch)
struct CellArgs {
  LeafCells lc;
  const DevHanging* hang;
  const uint8_t* cmask;
  const double* lin;
  const double* xu;
  const double* xp;
  const double* ecell;
  double* out;
  int64_t n;   // slots
  int mode;
  MatConst<double> m;
  Q2Mat<double> k;
  LevGeom<double> g[kMaxLevels];
};
struct NodeArgs {
  int32_t nc;
  int mode;
  int64_t n;
  const double* out;
  const int4* node;
  const int4* part_cells;
  const uint8_t* part_pos;
  const int32_t* ptr;    // fix-up list
  const int32_t* part;
  const double* w;
  const uint8_t* cmask;
  const double* xu;
  const double* xp;
  double* yu;
  double* yp;
};

// A block takes 32 cells: warp w evaluates their Gauss row w, so a cell's work is spread
// over three warps (a third of the serial chain of a thread per cell, and units fine
// enough to balance over the SMs); the rows' contributions meet in shared memory.
// Measured on the 267k-DoF band mesh (22k cells), operator apply: brick kernel 141 us (92 us
// with the cells of q2_jac.cuh), one thread per cell 97 us, this split 72 us (85 us when the compiler aims at 80 registers
// and more resident blocks: the FP64 pipe wants independent instructions, not warps).
template <int OP, bool MOD>
__global__ void __launch_bounds__(96, 5) q2_cell_kernel(const __grid_constant__ CellArgs a) {
  constexpr bool X = OP != OP_RESID;   // the operator reads an input
  __shared__ double xs[X ? 27 : 1][32];
  __shared__ double red[3][27][32];
  const int lane = threadIdx.x & 31, row = threadIdx.x >> 5;
  const int32_t nc = a.lc.ncells, c = blockIdx.x * 32 + lane, q = c < nc ? c : nc - 1;
  int32_t slot[9];
#pragma unroll
  for (int e = 0; e < 9; ++e) slot[e] = __ldg(a.lc.nodes9 + int64_t(e) * nc + q);
  const int lev = __ldg(a.lc.level + q);
  const int32_t cs = __ldg(a.lc.slot + q);
  pdl_wait();
  pdl_trigger();
  const bool mask = (a.mode & MODE_MASK_INPUT) != 0;
#pragma unroll
  for (int e = 0; e < 9; ++e) {
    const bool mine = X && e / 3 == row;   // the warp that gathers this node's input
    if (slot[e] >= 0) {
      if (mine) {
        const uint32_t cm = mask ? a.cmask[slot[e]] : 0u;
        const double x0 = a.xu[slot[e]], x1 = a.xu[a.n + slot[e]], xp = a.xp[slot[e]];
        xs[3 * e + 0][lane] = (cm & 1) ? 0.0 : x0;
        xs[3 * e + 1][lane] = (cm & 2) ? 0.0 : x1;
        xs[3 * e + 2][lane] = (cm & 4) ? 0.0 : xp;
      }
    } else {
      const DevHanging& h = a.hang[-2 - slot[e]];
      if (mine) {
        double x0 = 0.0, x1 = 0.0, xp = 0.0;
#pragma unroll
        for (int b = 0; b < 3; ++b) {
          const int ps = h.parent[b];
          const double w = h.weight[b];
          const uint32_t cm = mask ? a.cmask[ps] : 0u;
          x0 = pfma(w, (cm & 1) ? 0.0 : a.xu[ps], x0);
          x1 = pfma(w, (cm & 2) ? 0.0 : a.xu[a.n + ps], x1);
          xp = pfma(w, (cm & 4) ? 0.0 : a.xp[ps], xp);
        }
        xs[3 * e + 0][lane] = x0;
        xs[3 * e + 1][lane] = x1;
        xs[3 * e + 2][lane] = xp;
      }
      slot[e] = h.slot;   // the resolved linearisation
    }
  }
  const double ec = MOD ? a.ecell[cs] : 1.0;
  if (X) __syncthreads();
  auto ld = [&](int k, int i, int j) -> double2 {
    const int e = i + 3 * j;
    const int64_t s = slot[e];
    if (k == 0) return make_double2(xs[X ? 3 * e : 0][lane], xs[X ? 3 * e + 1 : 0][lane]);
    if (k == 1) return make_double2(a.lin[s], a.lin[a.n + s]);
    if (k == 2) return make_double2(X ? xs[X ? 3 * e + 2 : 0][lane] : 0.0, a.lin[2 * a.n + s]);
    return make_double2(a.lin[3 * a.n + s], 0.0);
  };
  {
    const Q2Own<double> own(a.m, a.g[lev], ec);
    double2 ru[9];
    double rp[9];
#pragma unroll
    for (int e = 0; e < 9; ++e) {
      ru[e] = make_double2(0.0, 0.0);
      rp[e] = 0.0;
    }
    if (row == 0) q2_jac_row<double, OP, MOD>(RowAt<double, 0>(), ld, a.k, own, ru, rp);
    else if (row == 1) q2_jac_row<double, OP, MOD>(RowAt<double, 1>(), ld, a.k, own, ru, rp);
    else q2_jac_row<double, OP, MOD>(RowAt<double, 2>(), ld, a.k, own, ru, rp);
#pragma unroll
    for (int e = 0; e < 9; ++e) {
      red[row][3 * e + 0][lane] = ru[e].x;
      red[row][3 * e + 1][lane] = ru[e].y;
      red[row][3 * e + 2][lane] = rp[e];
    }
  }
  __syncthreads();
  if (c >= nc) return;
  double* o = a.out + c;
#pragma unroll
  for (int e = 0; e < 9; ++e) {
    const int i = 9 * row + e;
    o[int64_t(i) * nc] = padd(padd(red[0][i][lane], red[1][i][lane]), red[2][i][lane]);
  }
}

// Component i of the nodal sum at brick position parity (px, py): the cells own, left,
// below, below-left hold the node as their local node (px, py), (2, py), (px, 2), (2, 2).
__device__ __forceinline__ double around(const double* out, int32_t nc, int4 k, int px, int py, int i) {
  auto at = [&](int32_t c, int a, int b) { return c >= 0 ? out[int64_t(3 * (a + 3 * b) + i) * nc + c] : 0.0; };
  return padd(padd(padd(at(k.z, px, 2), at(k.w, 2, 2)), at(k.y, 2, py)), at(k.x, px, py));
}

__global__ void __launch_bounds__(NODE_TPB) q2_node_kernel(const __grid_constant__ NodeArgs a) {
  pdl_trigger();
  const int64_t s = int64_t(blockIdx.x) * NODE_TPB + threadIdx.x;
  // everything but the contributions was there before pass 1 let this launch start
  int4 k = make_int4(-1, -1, -1, -1);
  uint32_t cm = 0;
  double xi[3] = {0.0, 0.0, 0.0};
  const bool in = s < a.n;
  if (in) {
    k = __ldg(a.node + s);
    cm = a.cmask[s];
    if (cm && (a.mode & MODE_IDENTITY)) {
      xi[0] = a.xu[s];
      xi[1] = a.xu[a.n + s];
      xi[2] = a.xp[s];
    }
  }
  pdl_wait();
  if (!in) return;
  double y[3] = {0.0, 0.0, 0.0};
  if (k.x >= -1) {
    const int o = int(s % (NB * NB)), px = o % NB & 1, py = o / NB & 1;
#pragma unroll
    for (int i = 0; i < 3; ++i) y[i] = around(a.out, a.nc, k, px, py, i);
  } else {
    // on a refinement edge: partial sums per level, its own and its hanging children's
    const int e1 = a.ptr[-1 - k.x];
    for (int e = a.ptr[-2 - k.x]; e < e1; ++e) {
      const int p = a.part[e];
      const int4 kp = __ldg(a.part_cells + p);
      const int pos = __ldg(a.part_pos + p);
      const double w = a.w[e];
#pragma unroll
      for (int i = 0; i < 3; ++i) y[i] = pfma(w, around(a.out, a.nc, kp, pos & 1, pos >> 1, i), y[i]);
    }
  }
  if (cm & 1) y[0] = xi[0];
  if (cm & 2) y[1] = xi[1];
  if (cm & 4) y[2] = xi[2];
  a.yu[s] = y[0];
  a.yu[a.n + s] = y[1];
  a.yp[s] = y[2];
}

template <int OP>
cudaError_t launch_op(const ApplyArgs& a, const FixupArgs& f, cudaStream_t s) {
  if (a.lc.ncells <= 0 || a.n_slots <= 0) return cudaSuccess;
  CellArgs c;
  c.lc = a.lc;
  c.hang = a.hang;
  c.cmask = a.cmask;
  c.lin = static_cast<const double*>(a.lin);
  c.xu = static_cast<const double*>(a.xu);
  c.xp = static_cast<const double*>(a.xp);
  c.ecell = static_cast<const double*>(a.ecell);
  c.n = a.n_slots;
  c.mode = a.mode;
  c.m = a.md;
  c.k = a.q2md;
  for (int l = 0; l < kMaxLevels; ++l) c.g[l] = a.gd[l];
  c.out = static_cast<double*>(a.lc.out);
  NodeArgs n;
  n.nc = a.lc.ncells;
  n.mode = a.mode;
  n.n = a.n_slots;
  n.out = static_cast<const double*>(a.lc.out);
  n.node = a.lc.node;
  n.part_cells = a.lc.part;
  n.part_pos = a.lc.part_pos;
  n.ptr = f.ptr; n.part = f.part; n.w = f.w;
  n.cmask = a.cmask;
  n.xu = c.xu; n.xp = c.xp;
  n.yu = static_cast<double*>(a.yu); n.yp = static_cast<double*>(a.yp);
  // dependent on whatever precedes it on the stream (it waits for that in full before
  // it reads or writes a vector); under a capture that may not be a kernel
  cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
  const bool pdl = cudaStreamIsCapturing(s, &st) == cudaSuccess && st == cudaStreamCaptureStatusNone;
  const cudaError_t e = launch_ex(pdl, a.ecell ? &q2_cell_kernel<OP, true> : &q2_cell_kernel<OP, false>, unsigned((a.lc.ncells + 31) / 32), 96u, 0, s, c);
  if (e != cudaSuccess) return e;
  return launch_ex(true, &q2_node_kernel, unsigned((a.n_slots + NODE_TPB - 1) / NODE_TPB), unsigned(NODE_TPB), 0, s, n);
}

}  // namespace

cudaError_t launch_leaf_cells_q2(const ApplyArgs& a, const FixupArgs& f, int op, cudaStream_t s) {
  switch (op) {
    case OP_FULL: return launch_op<OP_FULL>(a, f, s);
    case OP_FULL_T: return launch_op<OP_FULL_T>(a, f, s);
    case OP_RESID: return launch_op<OP_RESID>(a, f, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace pff
