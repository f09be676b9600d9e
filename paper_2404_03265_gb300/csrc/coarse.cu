// Dense level-0 blocks of the direct coarse solve (Sec. 3.2 of Kolditz & Wick,
// arXiv 2404.03265): assembly from element matrices and inversion, on the device, FP64.
//
// Inversion in place by blocked Gauss-Jordan elimination without pivoting.  With P a panel
// of 32 pivots, R the others and X = A_PP^-1,
//   A_PP <- X, A_PR <- X A_PR, A_RP <- -A_RP X, A_RR <- A_RR - A_RP (X A_PR)
// (old A_RP, A_PR on the right).  The pivots of an SPD matrix are Schur complements; a
// non-positive one is reported.
//
// What bounds it: FP64 (450 entries: 91M multiply-adds, 150 us at the chip's rate) and,
// in a first form, the serial pivot block: one block inverted it (35 us a panel) before 60
// blocks of 128 x 32 tiles, each with its own X A_PR, updated the rest (52 us).  Now a
// panel is two launches: X A_PR and A_RP X once, spread by 8 rows; then 16 x 32 tiles for
// the rest, beside one block that already forms and inverts the next panel's pivot block
// from copies the previous panel's launches made.  Sums keep their order.  Both blocks of
// the preconditioner run in the same launches.
#include "coarse.cuh"

#include <algorithm>

#include "pdl.cuh"

namespace pff {

namespace {

constexpr int SB = 32;    // pivots per panel
constexpr int TR = 16;    // rows of an update tile (its columns: SB)
constexpr int TPB = 256;

__host__ __device__ inline int32_t padded(int32_t n) { return (n + SB - 1) / SB * SB; }

// scratch: X[2], D[2] (SB x SB: a pivot block's inverse; the pivot block of the panel after
// next), C[2] (padded(n) x SB: a panel's old columns), R[2] (SB x padded(n): its old rows),
// Q (SB x padded(n): X A_PR)
struct Scr {
  double *X, *D, *C, *R, *Q;
  int32_t np;
  __device__ Scr(const CoarseBlock& b) : np(padded(b.n)) {
    X = b.scr;
    D = X + 2 * SB * SB;
    C = D + 2 * SB * SB;
    R = C + 2 * int64_t(np) * SB;
    Q = R + 2 * int64_t(np) * SB;
  }
  __device__ double* x(int p) const { return X + (p & 1) * SB * SB; }
  __device__ double* d(int p) const { return D + (p & 1) * SB * SB; }
  __device__ double* c(int p) const { return C + (p & 1) * int64_t(np) * SB; }
  __device__ double* r(int p) const { return R + (p & 1) * int64_t(np) * SB; }
};

// In-place inverse of the SB x SB pivot block M (padded with the identity) by scalar
// Gauss-Jordan steps, one reciprocal each: the thread that forms the next pivot inverts it.
// Written to x with zeros past b.
__device__ void invert_pivot(double (*M)[SB + 1], double* ip, int b, double* x, int32_t* bad) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  if (threadIdx.x == 0) {
    if (!(M[0][0] > 0.0)) *bad = 1;
    ip[0] = 1.0 / M[0][0];
  }
  __syncthreads();
  for (int k = 0; k < SB; ++k) {
    const double r = ip[k & 1];
    const double sk = M[k][lane] * r;   // row k scaled by the pivot's reciprocal
    double v[SB / 8];
#pragma unroll
    for (int q = 0; q < SB / 8; ++q) {
      const int i = w + 8 * q;
      const double pc = M[i][k];
      if (i == k) v[q] = lane == k ? r : sk;
      else if (lane == k) v[q] = -pc * r;
      else v[q] = fma(-pc, sk, M[i][lane]);
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < SB / 8; ++q) {
      const int i = w + 8 * q;
      M[i][lane] = v[q];
      if (i == k + 1 && lane == k + 1) {
        if (!(v[q] > 0.0)) *bad = 1;
        ip[(k + 1) & 1] = 1.0 / v[q];
      }
    }
    __syncthreads();
  }
#pragma unroll
  for (int q = 0; q < SB / 8; ++q) {
    const int i = w + 8 * q;
    x[i * SB + lane] = i < b && lane < b ? M[i][lane] : 0.0;
  }
}

// Panel 0: its inverse, copies of its columns and rows, and panel 1's pivot block
__global__ void __launch_bounds__(TPB) k_gj_first(const __grid_constant__ CoarseArgs a) {
  __shared__ double M[SB][SB + 1], ip[2];
  pdl_wait();
  pdl_trigger();
  const CoarseBlock& b = a.b[blockIdx.y];
  const int n = b.n;
  if (n <= 0) return;
  const Scr s(b);
  if (blockIdx.x == 0) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    for (int i = w; i < SB; i += TPB / 32) {
      M[i][lane] = i < n && lane < n ? b.A[int64_t(i) * n + lane] : (i == lane ? 1.0 : 0.0);
      const int r = SB + i, c = SB + lane;
      s.d(1)[i * SB + lane] = r < n && c < n ? b.A[int64_t(r) * n + c] : (i == lane ? 1.0 : 0.0);
    }
    __syncthreads();
    invert_pivot(M, ip, min(n, SB), s.x(0), a.bad + blockIdx.y);
    return;
  }
  const int64_t e = int64_t(blockIdx.x - 1) * TPB + threadIdx.x;
  if (e >= int64_t(s.np) * SB) return;
  const int r = int(e / SB), c = int(e % SB), rr = int(e / s.np), cc = int(e % s.np);
  s.c(0)[e] = r < n && c < n ? b.A[int64_t(r) * n + c] : 0.0;
  s.r(0)[e] = rr < n && cc < n ? b.A[int64_t(rr) * n + cc] : 0.0;
}

// Panel p, its rows and columns: 8 rows of one SB-wide tile per block.  blockIdx.x: tile
// T = x / 4 % nt, group x % 4; x / (4 nt): 0 the rows A_PR <- X A_PR (columns of T, rows
// 8 g ..), 1 the columns A_RP <- -A_RP X (rows 8 g .. of T).
__global__ void __launch_bounds__(TPB) k_gj_panel(const __grid_constant__ CoarseArgs a, int p) {
  __shared__ double U[8][SB], V[SB][SB];
  pdl_wait();
  pdl_trigger();
  const CoarseBlock& b = a.b[blockIdx.y];
  const int n = b.n, k0 = p * SB;
  if (k0 >= n) return;
  const Scr s(b);
  const int nt = s.np / SB, x = blockIdx.x, T = x / 4 % nt, g = x % 4;
  if (x >= 8 * nt) return;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const double* X = s.x(p);
  if (x < 4 * nt) {
    const int k = 8 * g + w, j = T * SB + lane;
    if (T == p) {   // A_PP <- X
      if (k0 + k < n && j < n) b.A[int64_t(k0 + k) * n + j] = X[k * SB + lane];
      return;
    }
    U[w][lane] = X[k * SB + lane];
    for (int m = w; m < SB; m += 8) V[m][lane] = s.r(p)[int64_t(m) * s.np + j];
    __syncthreads();
    double acc = 0.0;
#pragma unroll
    for (int m = 0; m < SB; ++m) acc = fma(U[w][m], V[m][lane], acc);
    s.Q[int64_t(k) * s.np + j] = acc;
    const bool in = k0 + k < n && j < n;
    if (in) b.A[int64_t(k0 + k) * n + j] = acc;
    if (T == p + 1) s.c(p + 1)[int64_t(k0 + k) * SB + lane] = in ? acc : 0.0;
    return;
  }
  if (T == p) return;
  const int i = T * SB + 8 * g + w;
  U[w][lane] = s.c(p)[int64_t(i) * SB + lane];
  for (int m = w; m < SB; m += 8) V[m][lane] = X[m * SB + lane];
  __syncthreads();
  double acc = 0.0;
#pragma unroll
  for (int k = 0; k < SB; ++k) acc = fma(U[w][k], V[k][lane], acc);
  const bool in = i < n && k0 + lane < n;
  if (in) b.A[int64_t(i) * n + k0 + lane] = -acc;
  if (T == p + 1) s.r(p + 1)[int64_t(i - (k0 + SB)) * s.np + k0 + lane] = in ? -acc : 0.0;
}

// Panel p, the rest: tiles of TR x SB (copying the next panel's columns and rows and the
// pivot block after it); block 0: the next panel's pivot block and its inverse.
__global__ void __launch_bounds__(TPB) k_gj_rest(const __grid_constant__ CoarseArgs a, int p) {
  __shared__ double Cs[SB][SB], Qs[SB][SB], M[SB][SB + 1], ip[2];
  pdl_wait();
  pdl_trigger();
  const CoarseBlock& b = a.b[blockIdx.y];
  const int n = b.n, k0 = p * SB, k1 = k0 + SB, k2 = k1 + SB;
  if (k0 >= n || (blockIdx.x == 0 && k1 >= n)) return;
  const Scr s(b);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nt = s.np / SB;
  const bool ahead = blockIdx.x == 0;
  const int t = int(blockIdx.x) - 1, J = ahead ? p + 1 : t % nt, i0 = ahead ? k1 : t / nt * TR;
  if (!ahead && (i0 >= s.np || J == p || i0 / SB == p)) return;
  for (int r = w; r < (ahead ? SB : TR); r += 8) Cs[r][lane] = s.c(p)[int64_t(i0 + r) * SB + lane];
  for (int k = w; k < SB; k += 8) Qs[k][lane] = s.Q[int64_t(k) * s.np + J * SB + lane];
  __syncthreads();
  if (ahead) {
    for (int r = w; r < SB; r += 8) {
      double acc = 0.0;
#pragma unroll
      for (int k = 0; k < SB; ++k) acc = fma(Cs[r][k], Qs[k][lane], acc);
      const bool in = k1 + r < n && k1 + lane < n;
      M[r][lane] = in ? s.d(p + 1)[r * SB + lane] - acc : (r == lane ? 1.0 : 0.0);
    }
    __syncthreads();
    invert_pivot(M, ip, min(n - k1, SB), s.x(p + 1), a.bad + blockIdx.y);
    return;
  }
  const int j = J * SB + lane;
  double q[SB];
#pragma unroll
  for (int k = 0; k < SB; ++k) q[k] = Qs[k][lane];
#pragma unroll
  for (int r0 = 0; r0 < TR; r0 += 8) {
    const int r = r0 + w, i = i0 + r;
    double acc = 0.0;
#pragma unroll
    for (int k = 0; k < SB; ++k) acc = fma(Cs[r][k], q[k], acc);
    const bool in = i < n && j < n;
    double v = 0.0;
    if (in) {
      double* at = b.A + int64_t(i) * n + j;
      v = *at - acc;
      *at = v;
    }
    if (J == p + 1) s.c(p + 1)[int64_t(i) * SB + lane] = v;
    if (i >= k1 && i < k2) s.r(p + 1)[int64_t(i - k1) * s.np + j] = v;
    if (i >= k2 && i < k2 + SB && J == p + 2) s.d(p + 2)[(i - k2) * SB + lane] = in ? v : (i - k2 == lane ? 1.0 : 0.0);
  }
}

// Free entries in the order of the list, then fixed ones; one block per matrix
__global__ void __launch_bounds__(1024) k_coarse_order(const __grid_constant__ CoarseArgs a) {
  __shared__ int warps[32], base[2];
  const CoarseBlock& b = a.b[blockIdx.x];
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  if (tid == 0) a.bad[blockIdx.x] = 0;
  auto fixed = [&](int e) { return (a.cmask[b.all[e] % a.n0] & (b.fix0 << (b.all[e] / a.n0))) != 0; };
  int nfree = 0;
  for (int e0 = 0; e0 < b.n; e0 += 1024) nfree += __syncthreads_count(e0 + tid < b.n && !fixed(e0 + tid));
  if (tid == 0) { base[0] = 0; base[1] = nfree; }
  __syncthreads();
  for (int e0 = 0; e0 < b.n; e0 += 1024) {
    const int e = e0 + tid;
    const bool in = e < b.n, fr = in && !fixed(e);
    const unsigned m = __ballot_sync(0xffffffffu, fr);
    if (lane == 0) warps[w] = __popc(m);
    __syncthreads();
    int before = 0, total = 0;
    for (int q = 0; q < 32; ++q) {
      if (q < w) before += warps[q];
      total += warps[q];
    }
    before += __popc(m & ((1u << lane) - 1u));
    if (in) {
      const int at = fr ? base[0] + before : base[1] + (tid - before);
      b.idx[at] = b.all[e];
      b.ent[b.all[e]] = at;
    }
    __syncthreads();
    if (tid == 0) {
      base[0] += total;
      base[1] += min(1024, b.n - e0) - total;
    }
    __syncthreads();
  }
}

// One warp per matrix row: the element matrices of the cells around its node, cells in
// row order, one lane per column entry
__global__ void __launch_bounds__(TPB) k_coarse_fill(const __grid_constant__ CoarseArgs a) {
  pdl_wait();
  pdl_trigger();
  const CoarseBlock& b = a.b[blockIdx.y];
  const int row = (blockIdx.x * TPB + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (row >= b.n) return;
  double* A = b.A + int64_t(row) * b.n;
  const int e = b.idx[row], comp = e / a.n0, slot = e % a.n0;
  const bool fixed = a.cmask[slot] & (b.fix0 << comp);
  for (int c = lane; c < b.n; c += 32) A[c] = fixed && c == row ? 1.0 : 0.0;
  if (fixed) return;
  __syncwarp();
  const int k = a.k, X = a.gx[slot], Y = a.gy[slot], nd = (k + 1) * (k + 1) * b.nc, nx = a.ncx * k + 1;
  const int ci0 = max(X % k ? X / k : X / k - 1, 0), ci1 = min(X / k, a.ncx - 1);
  const int cj0 = max(Y % k ? Y / k : Y / k - 1, 0), cj1 = min(Y / k, a.ncy - 1);
  for (int cj = cj0; cj <= cj1; ++cj)
    for (int ci = ci0; ci <= ci1; ++ci) {
      const int rd = ((X - ci * k) + (k + 1) * (Y - cj * k)) * b.nc + comp;
      const double* K = b.Ke + (int64_t(ci + a.ncx * cj) * nd + rd) * nd;
      for (int col = lane; col < nd; col += 32) {
        const int N = col / b.nc, cc = col % b.nc;
        const int cs = a.node_slot[ci * k + N % (k + 1) + nx * (cj * k + N / (k + 1))];
        const int ce = b.ent[cc * a.n0 + cs];
        if (ce >= 0 && !(a.cmask[cs] & (b.fix0 << cc))) A[ce] += K[col];
      }
      __syncwarp();
    }
}

}  // namespace

int64_t coarse_scratch(int32_t n) { return 4 * SB * SB + 5 * int64_t(padded(n)) * SB; }

cudaError_t coarse_fill(const CoarseArgs& a, cudaStream_t s) {
  const int32_t n = std::max(a.b[0].n, a.b[1].n);
  if (n <= 0) return cudaSuccess;
  k_coarse_order<<<2, 1024, 0, s>>>(a);
  k_coarse_fill<<<dim3(unsigned((n + TPB / 32 - 1) / (TPB / 32)), 2), TPB, 0, s>>>(a);
  return cudaGetLastError();
}

cudaError_t coarse_invert(const CoarseArgs& a, cudaStream_t s) {
  const int32_t n = std::max(a.b[0].n, a.b[1].n);
  if (n <= 0) return cudaSuccess;
  const int64_t np = padded(n), nt = np / SB;
  cudaError_t e = launch_ex2(true, &k_gj_first, dim3(unsigned(1 + (np * SB + TPB - 1) / TPB), 2), TPB, s, a);
  for (int p = 0; p < int(nt) && e == cudaSuccess; ++p) {
    e = launch_ex2(true, &k_gj_panel, dim3(unsigned(8 * nt), 2), TPB, s, a, p);
    if (e == cudaSuccess && nt > 1)
      e = launch_ex2(true, &k_gj_rest, dim3(unsigned(1 + np / TR * nt), 2), TPB, s, a, p);
  }
  return e;
}

}  // namespace pff
