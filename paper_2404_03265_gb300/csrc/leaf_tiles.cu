// FP32 Q1 leaf Jacobian on the regular bricks of a large mesh, a 15 x 15 node tile (16 x 16
// cells) per block.
//
// Thread (i, j) takes the cells (i, 2 j) and (i, 2 j + 1) of the tile's window as the pairs of
// the packed operations and owns their lower-left nodes.  The left cells' contributions come
// by shuffle and the row below through shared memory.  Cells and nodal sums are evaluated with
// the expressions and in the order of the column sweep: the same bits.
//
// Why not the sweep: a strip of the sweep is a chain of 16 dependent row steps, and with 16
// warps per SM that latency, not the issue rate, set its time; the irregular bricks' strips
// took 2.6 times as long per step and ended last.  A tile has one round of loads, and blocks
// at different stages overlap; the irregular bricks go in two passes around this launch.
// Measured on 4.1M DoFs (1395 regular bricks of 1681): the whole operator 38.9 us as a sweep,
// 36.2 us so (repeated on few vectors 34.1 us, and 37.0 us with the irregular bricks swept
// beside the tiles).  What bounds it now:
// this launch, 27 us alone, with issue slots 58% busy (its operations take 9 us, its bytes 8).
#include "kernels.cuh"
#include "pdl.cuh"
#include "q1_cell.cuh"

namespace pff {

namespace {

constexpr int NB = 30, TN = 15, CW = TN + 1, NW = TN + 2, TPB = CW * CW / 2;
constexpr int NPT = (NW * NW + TPB - 1) / TPB;

constexpr int MIN_BLOCKS = 5;   // 20 warps per SM at 96 registers (4: 37.9 us, 6 spills, 7: 36.6 us)

__device__ __forceinline__ NodePair<float2> stacked(const float4* sx, const float4* sl, int lo, int hi) {
  const float4 p = sx[lo], q = sx[hi], s = sl[lo], t = sl[hi];
  return {make_float2(p.x, q.x), make_float2(p.y, q.y), make_float2(p.z, q.z), make_float2(s.x, t.x),
          make_float2(s.y, t.y), make_float2(s.z, t.z), make_float2(s.w, t.w)};
}
__device__ __forceinline__ NodePair<float2> minus(const NodePair<float2>& r, const NodePair<float2>& l) {
  NodePair<float2> h;
  h.x0 = psub(r.x0, l.x0); h.x1 = psub(r.x1, l.x1); h.xp = psub(r.xp, l.xp);
  h.lx = psub(r.lx, l.lx); h.ly = psub(r.ly, l.ly); h.lz = psub(r.lz, l.lz); h.lw = psub(r.lw, l.lw);
  return h;
}

// Blocks 4 b .. 4 b + 3 take the tiles of regular brick b.  after: pass 1 of the other bricks runs
// before this grid on the stream and may still be running; the first block waits for it, so that
// pass 2, which waits for this grid, finds both done.
template <int OP>
__global__ void __launch_bounds__(TPB, MIN_BLOCKS) leaf_tile_kernel(const __grid_constant__ ApplyArgs a, int after) {
  using P = float2;
  __shared__ float4 sx[NW * NW], sl[NW * NW];   // x (fixed components 0) and the cell's modulus; linearisation
  __shared__ float up[3][TPB];
  __shared__ uint8_t sc[NW * NW];
  pdl_trigger();
  const int tid = threadIdx.x, q = blockIdx.x & 3;
  const BrickDesc* bd = a.lc.reg + (blockIdx.x >> 2);
  const int tx = TN * (q & 1), ty = TN * (q >> 1);
  const bool mask = (a.mode & MODE_MASK_INPUT) != 0;
  const int64_t n = a.n_slots;
  const float* xu = static_cast<const float*>(a.xu);
  const float* xp = static_cast<const float*>(a.xp);
  const float* lin = static_cast<const float*>(a.lin);
  const float* ec = static_cast<const float*>(a.ecell);
  int32_t at[NPT];
#pragma unroll
  for (int e = 0; e < NPT; ++e) {
    const int w = tid + e * TPB < NW * NW ? tid + e * TPB : 0;
    const int i = tx - 1 + w % NW, r = ty - 1 + w / NW;
    const int dx = i < 0 ? 0 : (i >= NB ? 2 : 1), dy = r < 0 ? 0 : (r >= NB ? 2 : 1);
    at[e] = __ldg(bd->nbr_base + 3 * dy + dx) + (i - NB * (dx - 1)) + NB * (r - NB * (dy - 1));
  }
  const LevGeom<float> g = a.gf[__ldg(&bd->level)];
  float4 x[NPT], l[NPT];
  uint8_t c[NPT];
#pragma unroll
  for (int e = 0; e < NPT; ++e) {
    const int32_t s = at[e];
    x[e] = make_float4(__ldg(xu + s), __ldg(xu + n + s), __ldg(xp + s), ec != nullptr ? __ldg(ec + s) : 1.f);
    l[e] = make_float4(__ldg(lin + s), __ldg(lin + n + s), __ldg(lin + 2 * n + s), __ldg(lin + 3 * n + s));
    c[e] = a.cmask[s];
  }
#pragma unroll
  for (int e = 0; e < NPT; ++e) {
    const int w = tid + e * TPB;
    if (w < NW * NW) {
      if (mask) {
        if (c[e] & 1) x[e].x = 0.f;
        if (c[e] & 2) x[e].y = 0.f;
        if (c[e] & 4) x[e].z = 0.f;
      }
      sx[w] = x[e];
      sl[w] = l[e];
      sc[w] = c[e];
    }
  }
  __syncthreads();
  const int ci = tid % CW, cj = tid / CW, w0 = ci + NW * 2 * cj;
  P out[12];
  {
    const NodePair<P> b = stacked(sx, sl, w0, w0 + NW), t = stacked(sx, sl, w0 + NW, w0 + 2 * NW);
    const NodePair<P> hb = minus(stacked(sx, sl, w0 + 1, w0 + NW + 1), b);
    const NodePair<P> ht = minus(stacked(sx, sl, w0 + NW + 1, w0 + 2 * NW + 1), t);
    q1_cell<P, OP>(b, hb, t, ht, a.mf, g, make_float2(sx[w0].w, sx[w0 + NW].w), out);
  }
  // node sums ((own upper-left + left upper-right of the row below) + left lower-right) + own
  // lower-left; a left neighbour in the other half of the warp belongs to a node not owned
  P carry[3], br[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    br[k].x = __shfl_up_sync(0xffffffffu, out[3 + k].x, 1);
    br[k].y = __shfl_up_sync(0xffffffffu, out[3 + k].y, 1);
    const P tr = make_float2(__shfl_up_sync(0xffffffffu, out[9 + k].x, 1), __shfl_up_sync(0xffffffffu, out[9 + k].y, 1));
    carry[k] = padd(out[6 + k], tr);
    up[k][tid] = carry[k].y;
  }
  __syncthreads();
  if (ci >= 1) {
    P y[3];
#pragma unroll
    for (int k = 0; k < 3; ++k)
      y[k] = padd(padd(make_float2(cj > 0 ? up[k][tid - CW] : 0.f, carry[k].x), br[k]), out[k]);
    float* yu = static_cast<float*>(a.yu);
    float* yp = static_cast<float*>(a.yp);
    const bool ident = (a.mode & MODE_IDENTITY) != 0;
    const int s1 = __ldg(bd->nbr_base + 4) + tx + ci - 1 + NB * (ty + 2 * cj);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      if (h == 0 && cj == 0) continue;
      const int s = h ? s1 : s1 - NB;
      const uint8_t cm = sc[w0 + h * NW];
      float v0 = h ? y[0].y : y[0].x, v1 = h ? y[1].y : y[1].x, v2 = h ? y[2].y : y[2].x;
      if (cm) {
        if (cm & 1) v0 = ident ? __ldg(xu + s) : 0.f;
        if (cm & 2) v1 = ident ? __ldg(xu + n + s) : 0.f;
        if (cm & 4) v2 = ident ? __ldg(xp + s) : 0.f;
      }
      yu[s] = v0;
      yu[n + s] = v1;
      yp[s] = v2;
    }
  }
  if (after && blockIdx.x == 0) pdl_wait();
}

}  // namespace

cudaError_t launch_leaf_tiles(const ApplyArgs& a, int op, bool after, cudaStream_t s) {
  if (a.lc.nreg <= 0) return cudaSuccess;
  const unsigned grid = 4u * unsigned(a.lc.nreg), tpb = TPB;
  if (op == OP_FULL) return launch_ex(after, &leaf_tile_kernel<OP_FULL>, grid, tpb, 0, s, a, int(after));
  if (op == OP_FULL_T) return launch_ex(after, &leaf_tile_kernel<OP_FULL_T>, grid, tpb, 0, s, a, int(after));
  return cudaErrorInvalidValue;
}

}  // namespace pff
