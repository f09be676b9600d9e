// Q1 leaf operators as two passes over compact lists: the cells of the leaf mesh, then
// its node slots.
//
// Pass 1: one thread per leaf cell (no lane is spent on a cell that does not exist)
// gathers the cell's four nodes, resolving hanging ones from their parents, evaluates
// the operator (q1_cell.cuh) and writes the 12 nodal contributions.  Pass 2: one thread
// per node slot adds the contributions of the cells around it, condenses the hanging
// nodes' onto their parents (C^T) and applies the constraint rows.  Cells, nodal sums
// and condensation are evaluated with the expressions and in the order of the column
// sweep and its fix-up kernel, so the results are the same bits.
//
// What bounds it: in FP64 the arithmetic rate of GB300 (1/64 of FP32; a cell of the
// Jacobian is about 280 FP64 instructions), so the work that counts is the number of
// cells evaluated.  The sweep evaluates every position of its bricks in lock step: on a
// crack mesh (1.04M DoFs, 348k nodes in 743k slots) 2.4 times the cells that exist, in
// 826 one-warp strips for 152 SMs.  The contributions cost 96 bytes per cell written and
// read again, from L2 at these sizes.  Jacobian 647 -> 200 us there, 971 -> 724 us on 4.1M
// DoFs.
#include "cheb.cuh"
#include "kernels.cuh"
#include "pdl.cuh"
#include "q1_cell.cuh"

#include <type_traits>

namespace pff {

namespace {

constexpr int CELL_TPB = 128;
constexpr int NODE_TPB = 256;

// Kernel arguments, in the precision T of the pass (small ones: they are copied per launch).
template <typename T>
struct CellArgs {
  LeafCells lc;
  const DevHanging* hang;
  const uint8_t* cmask;
  const T* lin;
  const T* xu;
  const T* xp;
  const T* ecell;
  int64_t n;   // slots
  int mode;
  MatConst<T> m;
  LevGeom<T> g[kMaxLevels];
};
template <typename T>
struct NodeArgs {
  int32_t nc;
  int mode;
  int64_t n;
  const T* out;
  const int4* node;
  const int4* part_cells;
  const int32_t* ptr;    // fix-up list
  const int32_t* part;
  const double* w;
  const uint8_t* cmask;
  const T* xu;
  const T* xp;
  T* yu;
  T* yp;
};

template <typename T> void constants(CellArgs<T>& c, const ApplyArgs& a);
template <> void constants<float>(CellArgs<float>& c, const ApplyArgs& a) {
  c.m = a.mf;
  for (int l = 0; l < kMaxLevels; ++l) c.g[l] = a.gf[l];
}
template <> void constants<double>(CellArgs<double>& c, const ApplyArgs& a) {
  c.m = a.md;
  for (int l = 0; l < kMaxLevels; ++l) c.g[l] = a.gd[l];
}

// Node of a cell: fields read from its slot (code >= 0), or for hanging entry -2 - code
// the resolved linearisation from its slot and the input from its parents.
template <typename T, int OP>
__device__ __forceinline__ NodePair<T> cell_node(const CellArgs<T>& a, int32_t code, bool mask) {
  using N = Needs<OP>;
  NodePair<T> v{};
  const T *xu = a.xu, *xp = a.xp, *lin = a.lin;
  const int64_t n = a.n;
  int32_t slot = code;
  if (code >= 0) {
    const uint32_t cm = mask && (N::xu || N::xp) ? a.cmask[slot] : 0u;
    if (N::xu) { v.x0 = xu[slot]; v.x1 = xu[n + slot]; }
    if (N::xp) v.xp = xp[slot];
    if (N::xu) {
      if (cm & 1) v.x0 = T(0);
      if (cm & 2) v.x1 = T(0);
    }
    if (N::xp && (cm & 4)) v.xp = T(0);
  } else {
    const DevHanging& e = a.hang[-2 - code];
    slot = e.slot;
    if (N::xu || N::xp) {
#pragma unroll
      for (int b = 0; b < 2; ++b) {
        const int ps = e.parent[b];
        const T w = T(e.weight[b]);
        const uint32_t cm = mask ? a.cmask[ps] : 0u;
        if (N::xu) {
          v.x0 = pfma(w, (cm & 1) ? T(0) : xu[ps], v.x0);
          v.x1 = pfma(w, (cm & 2) ? T(0) : xu[n + ps], v.x1);
        }
        if (N::xp) v.xp = pfma(w, (cm & 4) ? T(0) : xp[ps], v.xp);
      }
    }
  }
  if (N::linU) { v.lx = lin[slot]; v.ly = lin[n + slot]; }
  if (N::phi) v.lz = lin[2 * n + slot];
  if (N::phit) v.lw = lin[3 * n + slot];
  return v;
}

template <typename P>
__device__ __forceinline__ NodePair<P> diff(const NodePair<P>& r, const NodePair<P>& l) {
  NodePair<P> h;
  h.x0 = psub(r.x0, l.x0); h.x1 = psub(r.x1, l.x1); h.xp = psub(r.xp, l.xp);
  h.lx = psub(r.lx, l.lx); h.ly = psub(r.ly, l.ly); h.lz = psub(r.lz, l.lz); h.lw = psub(r.lw, l.lw);
  return h;
}

// Components an operator writes.
template <int OP> struct Out {
  static constexpr bool u = (OP != OP_TCV && OP != OP_PHIT_VJP);
  static constexpr int c0 = u ? 0 : 2;
};

__device__ __forceinline__ NodePair<float2> zip(const NodePair<float>& a, const NodePair<float>& b) {
  return {make_float2(a.x0, b.x0), make_float2(a.x1, b.x1), make_float2(a.xp, b.xp), make_float2(a.lx, b.lx),
          make_float2(a.ly, b.ly), make_float2(a.lz, b.lz), make_float2(a.lw, b.lw)};
}

// FP32: a thread takes two neighbouring cells of one level as the pairs of the packed
// operations (the list is even within each level); FP64 one.
template <typename T, int OP>
__global__ void __launch_bounds__(CELL_TPB) leaf_cell_kernel(const __grid_constant__ CellArgs<T> a) {
  constexpr int M = sizeof(T) == 4 ? 2 : 1;
  using P = typename std::conditional<M == 2, float2, T>::type;
  const int32_t nc = a.lc.ncells;
  const int32_t c = M * (blockIdx.x * CELL_TPB + threadIdx.x);
  int4 k[M];
  int lev, cs[M];
#pragma unroll
  for (int h = 0; h < M; ++h) {   // mesh tables
    const int32_t q = c < nc ? c + h : 0;
    k[h] = __ldg(a.lc.corner + q);
    cs[h] = __ldg(a.lc.slot + q);
  }
  lev = __ldg(a.lc.level + (c < nc ? c : 0));
  pdl_wait();
  pdl_trigger();
  if (c >= nc) return;
  const bool mask = (a.mode & MODE_MASK_INPUT) != 0;
  NodePair<T> n[M][4];
  T e[M];
#pragma unroll
  for (int h = 0; h < M; ++h) {
    n[h][0] = cell_node<T, OP>(a, k[h].x, mask);
    n[h][1] = cell_node<T, OP>(a, k[h].y, mask);
    n[h][2] = cell_node<T, OP>(a, k[h].z, mask);
    n[h][3] = cell_node<T, OP>(a, k[h].w, mask);
    e[h] = a.ecell != nullptr ? a.ecell[cs[h]] : T(1);
  }
  const LevGeom<T> g = a.g[lev];
  P out[12];
  if constexpr (M == 2) {
    const NodePair<P> b = zip(n[0][0], n[1][0]), t = zip(n[0][2], n[1][2]);
    q1_cell<P, OP>(b, diff(zip(n[0][1], n[1][1]), b), t, diff(zip(n[0][3], n[1][3]), t), a.m, g,
                   make_float2(e[0], e[1]), out);
  } else {
    q1_cell<P, OP>(n[0][0], diff(n[0][1], n[0][0]), n[0][2], diff(n[0][3], n[0][2]), a.m, g, e[0], out);
  }
  T* o = reinterpret_cast<T*>(a.lc.out) + c;
#pragma unroll
  for (int q = 0; q < 4; ++q)
#pragma unroll
    for (int i = Out<OP>::c0; i < 3; ++i) *reinterpret_cast<P*>(o + int64_t(3 * q + i) * nc) = out[3 * q + i];
}

// Sum of component q of the contributions to the node with own, left, below and
// below-left cells k.x, k.y, k.z, k.w (-1 none).
template <typename T>
__device__ __forceinline__ T around(const T* out, int32_t nc, int4 k, int q) {
  const T c2 = k.z >= 0 ? out[int64_t(6 + q) * nc + k.z] : T(0);
  const T c3 = k.w >= 0 ? out[int64_t(9 + q) * nc + k.w] : T(0);
  const T c1 = k.y >= 0 ? out[int64_t(3 + q) * nc + k.y] : T(0);
  const T c0 = k.x >= 0 ? out[int64_t(q) * nc + k.x] : T(0);
  return padd(padd(padd(c2, c3), c1), c0);
}

template <typename T, int OP>
__global__ void __launch_bounds__(NODE_TPB) leaf_node_kernel(const __grid_constant__ NodeArgs<T> a) {
  constexpr int C0 = Out<OP>::c0;
  pdl_trigger();
  const int64_t s = int64_t(blockIdx.x) * NODE_TPB + threadIdx.x;
  // everything but the contributions was there before pass 1 let this launch start
  int4 k = make_int4(-1, -1, -1, -1);
  uint32_t cm = 0;
  T xi[3] = {T(0), T(0), T(0)};
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
  T y[3] = {T(0), T(0), T(0)};
  if (k.x >= -1) {
#pragma unroll
    for (int q = C0; q < 3; ++q) y[q] = around(a.out, a.nc, k, q);
  } else {
    // on a refinement edge: partial sums per level, its own and its hanging children's
    const int e1 = a.ptr[-1 - k.x];
    for (int e = a.ptr[-2 - k.x]; e < e1; ++e) {
      const int4 kp = __ldg(a.part_cells + a.part[e]);
      const T w = T(a.w[e]);
#pragma unroll
      for (int q = C0; q < 3; ++q) y[q] = pfma(w, around(a.out, a.nc, kp, q), y[q]);
    }
  }
  if (cm & 1) y[0] = xi[0];
  if (cm & 2) y[1] = xi[1];
  if (cm & 4) y[2] = xi[2];
  if (Out<OP>::u) {
    a.yu[s] = y[0];
    a.yu[a.n + s] = y[1];
  }
  a.yp[s] = y[2];
}

template <typename T, int OP>
cudaError_t launch_op(const ApplyArgs& a, const FixupArgs& f, cudaStream_t s) {
  if (a.lc.ncells <= 0 || a.n_slots <= 0) return cudaSuccess;
  CellArgs<T> c;
  c.lc = a.lc;
  c.hang = a.hang;
  c.cmask = a.cmask;
  c.lin = static_cast<const T*>(a.lin);
  c.xu = static_cast<const T*>(a.xu);
  c.xp = static_cast<const T*>(a.xp);
  c.ecell = static_cast<const T*>(a.ecell);
  c.n = a.n_slots;
  c.mode = a.mode;
  constants<T>(c, a);
  NodeArgs<T> n;
  n.nc = a.lc.ncells;
  n.mode = a.mode;
  n.n = a.n_slots;
  n.out = static_cast<const T*>(a.lc.out);
  n.node = a.lc.node;
  n.part_cells = a.lc.part;
  n.ptr = f.ptr; n.part = f.part; n.w = f.w;
  n.cmask = a.cmask;
  n.xu = c.xu; n.xp = c.xp;
  n.yu = static_cast<T*>(a.yu); n.yp = static_cast<T*>(a.yp);
  const int32_t nt = sizeof(T) == 4 ? a.lc.ncells / 2 : a.lc.ncells;   // threads of pass 1
  // dependent on whatever precedes it on the stream (it waits for that in full before
  // it reads or writes a vector); under a capture that may not be a kernel
  cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
  const bool pdl = cudaStreamIsCapturing(s, &st) == cudaSuccess && st == cudaStreamCaptureStatusNone;
  const cudaError_t e = launch_ex(pdl, &leaf_cell_kernel<T, OP>, unsigned((nt + CELL_TPB - 1) / CELL_TPB),
                                  unsigned(CELL_TPB), 0, s, c);
  if (e != cudaSuccess) return e;
  return launch_ex(true, &leaf_node_kernel<T, OP>, unsigned((a.n_slots + NODE_TPB - 1) / NODE_TPB), unsigned(NODE_TPB),
                   0, s, n);
}

}  // namespace

template <>
cudaError_t launch_leaf_cells<double>(const ApplyArgs& a, const FixupArgs& f, int op, cudaStream_t s) {
  switch (op) {
    case OP_FULL: return launch_op<double, OP_FULL>(a, f, s);
    case OP_FULL_T: return launch_op<double, OP_FULL_T>(a, f, s);
    case OP_RESID: return launch_op<double, OP_RESID>(a, f, s);
    case OP_TCV: return launch_op<double, OP_TCV>(a, f, s);
    case OP_TCV_GRAD: return launch_op<double, OP_TCV_GRAD>(a, f, s);
    case OP_PHIT_VJP: return launch_op<double, OP_PHIT_VJP>(a, f, s);
    default: return cudaErrorInvalidValue;
  }
}

template <>
cudaError_t launch_leaf_cells<float>(const ApplyArgs& a, const FixupArgs& f, int op, cudaStream_t s) {
  switch (op) {
    case OP_FULL: return launch_op<float, OP_FULL>(a, f, s);
    case OP_FULL_T: return launch_op<float, OP_FULL_T>(a, f, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace pff
