// Multigrid kernels of libpff (see mg.cuh).  Level vectors of a block are
// stored per level as ncomp consecutive blocks of the level's slot count.
// Fixed rows (Dirichlet u for the u-block, active phi for the phi-block) and
// holes carry zeros; the inverse diagonal is zero off the interior, so the
// Chebyshev updates leave edge and fixed entries untouched.
#include "mg.cuh"

#include <algorithm>

#include "cheb.cuh"
#include "pdl.cuh"

namespace pff {

namespace {

constexpr int TPB = 256;

inline unsigned blocks_for(int64_t n) {
  int64_t b = (n + TPB - 1) / TPB;
  if (b > 65535 * 8) b = 65535 * 8;
  return unsigned(b < 1 ? 1 : b);
}

#define GRID_STRIDE(i, n) for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < (n); i += int64_t(gridDim.x) * blockDim.x)

constexpr int TB = 8;   // transfer-row entries whose loads are issued together

template <typename T>
__global__ void k_cheb_first(int64_t n, T* x, T* xprev, const T* dinv, const T* d, T c0) {
  pdl_trigger();
  pdl_wait();
  GRID_STRIDE(i, n) {
    x[i] = cheb_first_of(c0, dinv[i], d[i]);
    xprev[i] = T(0);
  }
}

template <typename T>
__global__ void k_cheb_step(int64_t n, T* xnew, const T* x, const T* xprev, const T* dinv, const T* d, const T* ax,
                            T a, T b) {
  pdl_trigger();
  pdl_wait();
  GRID_STRIDE(i, n) {
    xnew[i] = cheb_next(x[i], xprev[i], dinv[i], d[i], ax[i], a, b);
  }
}

template <typename T>
__global__ void k_restrict(int32_t nc, int ncomp, int64_t ncs, int64_t nfs, const int32_t* __restrict__ ptr,
                           const int32_t* __restrict__ col, const float* __restrict__ val, const T* __restrict__ df,
                           const T* __restrict__ axf, T* dc, const uint8_t* __restrict__ cmask_c, int fixbits,
                           const T* __restrict__ dinv_c, T* cur_c, T* prev_c, T c0) {
  pdl_trigger();
  pdl_wait();
  GRID_STRIDE(y, nc) {
    const uint8_t cm = cmask_c[y];
    const int e0 = ptr[y], e1 = ptr[y + 1];
    // ncomp is 1 or 2: the second sum is acc1
    T acc0 = dc[y], acc1 = ncomp > 1 ? dc[ncs + y] : T(0);
    // the row in batches of TB entries: indices and weights, then values, then the
    // sums in entry order (as one entry at a time)
    for (int eb = e0; eb < e1; eb += TB) {
      int z[TB];
      T w[TB];
#pragma unroll
      for (int q = 0; q < TB; ++q) {
        z[q] = eb + q < e1 ? col[eb + q] : 0;
        w[q] = eb + q < e1 ? T(val[eb + q]) : T(0);
      }
      for (int c = 0; c < ncomp; ++c) {
        T d[TB];
#pragma unroll
        for (int q = 0; q < TB; ++q) d[q] = eb + q < e1 ? df[c * nfs + z[q]] - axf[c * nfs + z[q]] : T(0);
        T a = c == 0 ? acc0 : acc1;
#pragma unroll
        for (int q = 0; q < TB; ++q)
          if (eb + q < e1) a += w[q] * d[q];
        if (c == 0) acc0 = a; else acc1 = a;
      }
    }
    for (int c = 0; c < ncomp; ++c) {
      const int bit = (fixbits == 4) ? 4 : (1 << c);
      const T v = (cm & bit) ? T(0) : (c == 0 ? acc0 : acc1);
      dc[c * ncs + y] = v;
      if (cur_c != nullptr) {
        cur_c[c * ncs + y] = cheb_first_of(c0, dinv_c[c * ncs + y], v);
        prev_c[c * ncs + y] = T(0);
      }
    }
  }
}

template <typename T>
__global__ void k_prolong(int32_t nf, int ncomp, int64_t nfs, int64_t ncs, const int32_t* __restrict__ ptr,
                          const int32_t* __restrict__ col, const float* __restrict__ val, const T* __restrict__ xc,
                          T* xf, const uint8_t* __restrict__ cmask_f, int fixbits) {
  pdl_trigger();
  pdl_wait();
  GRID_STRIDE(z, nf) {
    const uint8_t cm = cmask_f[z];
    const int e0 = ptr[z], e1 = ptr[z + 1];
    T acc0 = xf[z], acc1 = ncomp > 1 ? xf[nfs + z] : T(0);
    for (int eb = e0; eb < e1; eb += TB) {
      int yy[TB];
      T w[TB];
#pragma unroll
      for (int q = 0; q < TB; ++q) {
        yy[q] = eb + q < e1 ? col[eb + q] : 0;
        w[q] = eb + q < e1 ? T(val[eb + q]) : T(0);
      }
      for (int c = 0; c < ncomp; ++c) {
        T v[TB];
#pragma unroll
        for (int q = 0; q < TB; ++q) v[q] = eb + q < e1 ? xc[c * ncs + yy[q]] : T(0);
        T a = c == 0 ? acc0 : acc1;
#pragma unroll
        for (int q = 0; q < TB; ++q)
          if (eb + q < e1) a += w[q] * v[q];
        if (c == 0) acc0 = a; else acc1 = a;
      }
    }
    for (int c = 0; c < ncomp; ++c) {
      const int bit = (fixbits == 4) ? 4 : (1 << c);
      xf[c * nfs + z] = (cm & bit) ? T(0) : (c == 0 ? acc0 : acc1);
    }
  }
}

template <typename T>
__global__ void k_copy_in(int64_t nsl, int ncomp, DevHome home, const double* __restrict__ r, T* d,
                          const uint8_t* __restrict__ lcm, int fixbits) {
  GRID_STRIDE(s, nsl) {
    const int32_t b = home.slot[s];
    if (b < 0) continue;
    const int64_t base = int64_t(ncomp) * home.off[s] + b, nl = home.nsl[s];
    const uint8_t cm = lcm[s];
    for (int c = 0; c < ncomp; ++c) {
      const int bit = (fixbits == 4) ? 4 : (1 << c);
      if (!(cm & bit)) d[base + c * nl] = T(r[c * nsl + s]);
    }
  }
}

// One block per level brick: every level slot is written, so the level defects
// need no separate clearing.  The loads of a thread's slots are issued together.
constexpr int LD_SLOTS = 900;                            // slots per brick
constexpr int LD_N = (LD_SLOTS + TPB - 1) / TPB;
template <typename T>
__global__ void __launch_bounds__(TPB) k_level_defects(const LevBrick* __restrict__ bricks,
                                                       const int32_t* __restrict__ home_leaf, int ncomp, int64_t nsl,
                                                       const double* __restrict__ r, T* d, T* x0,
                                                       const uint8_t* __restrict__ lcm, int fixbits) {
  pdl_trigger();
  const LevBrick b = bricks[blockIdx.x];
  int32_t leaf[LD_N];
#pragma unroll
  for (int k = 0; k < LD_N; ++k) {
    const int i = threadIdx.x + TPB * k;
    leaf[k] = i < LD_SLOTS ? home_leaf[b.off + b.base + i] : -1;
  }
  double v[LD_N][2];
  uint8_t cm[LD_N];
#pragma unroll
  for (int k = 0; k < LD_N; ++k) {
    cm[k] = leaf[k] >= 0 ? lcm[leaf[k]] : uint8_t(0);
    v[k][0] = leaf[k] >= 0 ? r[leaf[k]] : 0.0;
    v[k][1] = leaf[k] >= 0 && ncomp > 1 ? r[nsl + leaf[k]] : 0.0;
  }
#pragma unroll
  for (int k = 0; k < LD_N; ++k) {
    const int i = threadIdx.x + TPB * k;
    if (i >= LD_SLOTS) break;
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      if (c >= ncomp) break;
      const int bit = (fixbits == 4) ? 4 : (1 << c);
      const int64_t o = int64_t(ncomp) * b.off + c * int64_t(b.n) + b.base + i;
      d[o] = (cm[k] & bit) ? T(0) : T(v[k][c]);
      if (b.off == 0) x0[o] = T(0);
    }
  }
}

template <typename T>
__global__ void k_copy_out(int64_t nsl, int ncomp, DevHome home, const T* __restrict__ x,
                           const double* __restrict__ r, double* z, const uint8_t* __restrict__ lcm,
                           const uint8_t* __restrict__ lflags, int fixbits) {
  pdl_trigger();
  bool waited = false;   // the tables of the first slot are read before the wait
  GRID_STRIDE(s, nsl) {
    const uint8_t cm = lcm[s], lf = lflags[s];
    const int32_t b = home.slot[s];
    const int64_t off = home.off[s], nl = home.nsl[s];
    const bool node = (lf & 1) && !(lf & 4);
    const int64_t base = b >= 0 ? int64_t(ncomp) * off + b : 0;
    if (!waited) { pdl_wait(); waited = true; }
    for (int c = 0; c < ncomp; ++c) {
      const int bit = (fixbits == 4) ? 4 : (1 << c);
      double v = 0.0;
      if (cm & bit) v = node ? r[c * nsl + s] : 0.0;
      else if (b >= 0) v = double(x[base + c * nl]);
      z[c * nsl + s] = v;
    }
  }
  if (!waited) pdl_wait();
}

template <typename T>
__global__ void k_cheb_first_res(int64_t n, T* x, T* xprev, T* r, const T* __restrict__ dinv,
                                 const T* __restrict__ d, const T* __restrict__ ax, T c0, T* xadd) {
  pdl_trigger();
  pdl_wait();
  GRID_STRIDE(i, n) {
    const T ri = d[i] - ax[i];
    const T v = cheb_first_of(c0, dinv[i], ri);
    if (xadd != nullptr) {
      xadd[i] += v;
    } else {
      r[i] = ri;
      x[i] = v;
      xprev[i] = T(0);
    }
  }
}

template <typename T>
__global__ void k_cheb_step_add(int64_t n, T* xadd, const T* __restrict__ x, const T* __restrict__ xprev,
                                const T* __restrict__ dinv, const T* __restrict__ d, const T* __restrict__ ax, T a,
                                T b) {
  pdl_trigger();
  pdl_wait();
  GRID_STRIDE(i, n) {
    xadd[i] += cheb_next(x[i], xprev[i], dinv[i], d[i], ax[i], a, b);
  }
}

// Dense FP64 coarse solve x[idx] = Ainv d[idx], d taken to FP64: one warp per row,
// lanes stride the columns, fixed-order warp reduction.  The first CP columns of a
// lane (all of them on a 16 x 16 coarse mesh) and their indices are read before the wait.
// The next launch may start after the wait (the FP32 tiles count on that, see
// launch_smooth_up); in FP64, whose sweeps do not, at once: with both blocks' V-cycles side
// by side the warps that already wait spread over the SMs, and their FP64 work with them.
// Both V-cycles of a GMRES step, 65k DoFs: 1411 -> 1290 us, one alone 934 -> 992 us.
template <typename T>
__global__ void k_coarse_matvec(int32_t n, const int32_t* __restrict__ idx, const double* __restrict__ A, const T* d,
                                T* x) {
  constexpr int CP = 16;
  const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  const int row = warp < n ? warp : n - 1;
  if (sizeof(T) == 8) pdl_trigger();
  double a[CP];
  int32_t ix[CP];
#pragma unroll
  for (int q = 0; q < CP; ++q) {
    const int j = lane + 32 * q;
    a[q] = j < n ? A[int64_t(row) * n + j] : 0.0;
    ix[q] = j < n ? idx[j] : 0;
  }
  const int32_t out = idx[row];
  pdl_wait();
  if (sizeof(T) == 4) pdl_trigger();
  if (warp >= n) return;
  T t[CP];
#pragma unroll
  for (int q = 0; q < CP; ++q) t[q] = d[ix[q]];
  double acc = 0.0;
#pragma unroll
  for (int q = 0; q < CP; ++q)
    if (lane + 32 * q < n) acc += a[q] * double(t[q]);
  for (int j = lane + 32 * CP; j < n; j += 32) acc += A[int64_t(row) * n + j] * double(d[idx[j]]);
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
  if (lane == 0) x[out] = T(acc);
}

// level linearisations from the leaf's, one block per level brick of all levels
__global__ void __launch_bounds__(TPB) k_inject_lin(const LevBrick* __restrict__ bricks,
                                                    const int32_t* __restrict__ lev_leaf,
                                                    const double* __restrict__ lin, int64_t nsleaf, double* l64,
                                                    float* l32) {
  const LevBrick b = bricks[blockIdx.x];
  for (int i = threadIdx.x; i < LD_SLOTS; i += TPB) {
    const int ls = lev_leaf[b.off + b.base + i];
#pragma unroll
    for (int f = 0; f < 4; ++f) {
      const double v = ls >= 0 ? lin[f * nsleaf + ls] : 0.0;
      const int64_t o = 4 * int64_t(b.off) + f * int64_t(b.n) + b.base + i;
      l64[o] = v;
      l32[o] = float(v);
    }
  }
}

__global__ void k_level_cmask(int32_t nsl, const uint8_t* __restrict__ flags, const int32_t* __restrict__ sl,
                              const uint8_t* __restrict__ lcm, const int32_t* __restrict__ Rp,
                              const int32_t* __restrict__ Rc, const uint8_t* __restrict__ cmf, uint8_t* cm) {
  GRID_STRIDE(s, nsl) {
    const uint8_t f = flags[s];
    uint8_t c = 0;
    if ((f & 1) && (f & 2)) c |= 3;
    if (f & 1) {
      const int ls = sl[s];
      bool act = ls >= 0 && (lcm[ls] & 4);
      if (!act && Rp != nullptr && !(f & 16)) {
        for (int e = Rp[s]; e < Rp[s + 1]; ++e)
          if (cmf[Rc[e]] & 4) { act = true; break; }
      }
      if (act) c |= 4;
    }
    cm[s] = c;
  }
}

__global__ void k_invert_diag(int32_t nsl, int ncomp, const double* __restrict__ diag,
                              const uint8_t* __restrict__ flags, const uint8_t* __restrict__ cm, int fixbits,
                              double* d64, float* d32) {
  GRID_STRIDE(s, nsl) {
    const uint8_t f = flags[s];
    for (int c = 0; c < ncomp; ++c) {
      const int bit = (fixbits == 4) ? 4 : (1 << c);
      const int64_t i = c * int64_t(nsl) + s;
      const double dg = diag[i];
      const bool interior = (f & 1) && !(f & 8) && !(cm[s] & bit) && dg != 0.0;
      const double v = interior ? 1.0 / dg : 0.0;
      d64[i] = v;
      d32[i] = float(v);
    }
  }
}

__device__ __forceinline__ uint64_t splitmix64(uint64_t x) {
  uint64_t z = x + 0x9E3779B97F4A7C15ull;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

constexpr int DOT_BLOCKS = 512;

__global__ void k_dot_partial(int64_t n, const double* __restrict__ a, const double* __restrict__ b, double* part) {
  __shared__ double sh[TPB];
  double acc = 0.0;
  GRID_STRIDE(i, n) acc += a[i] * b[i];
  sh[threadIdx.x] = acc;
  __syncthreads();
  for (int o = TPB / 2; o > 0; o >>= 1) {
    if (threadIdx.x < o) sh[threadIdx.x] += sh[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) part[blockIdx.x] = sh[0];
}

__global__ void k_dot_final(int nb, const double* __restrict__ part, double* out) {
  __shared__ double sh[TPB];
  double acc = 0.0;
  for (int i = threadIdx.x; i < nb; i += TPB) acc += part[i];
  sh[threadIdx.x] = acc;
  __syncthreads();
  for (int o = TPB / 2; o > 0; o >>= 1) {
    if (threadIdx.x < o) sh[threadIdx.x] += sh[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) out[0] = sh[0];
}

// Jacobi-preconditioned CG of a set-up chain: three launches a step beside the operator
// apply (dot p.q; r, z and dot r.z; p).  A dot's last block to finish adds the blocks'
// partial sums in a fixed order and forms the scalars
//   sc: 0 rz, 1 pq, 2 rz_new, 3 alpha, 4 beta, 5 ok (1 while the iteration is healthy).
// Each step's coefficients go to hist (alpha_j, beta_j; alpha_j = 0 marks a stop).
// Q: precision of q = A p.
enum CgStage : int { CG_START = 0, CG_PQ = 1, CG_RZ = 2 };
template <int STAGE, typename Q>
__global__ void __launch_bounds__(TPB) k_cg(int64_t n, int32_t nsl, const int32_t* __restrict__ gx,
                                            const int32_t* __restrict__ gy, const double* __restrict__ dinv, double* r,
                                            double* z, double* p, Q* pq, const Q* q, double* sc, double* hist, int step,
                                            double* partial, unsigned* count) {
  __shared__ double sh[TPB];
  __shared__ bool last;
  pdl_wait();
  pdl_trigger();
  const int tid = threadIdx.x;
  const double alpha = STAGE == CG_RZ ? sc[3] : 0.0;
  double acc = 0.0;
  GRID_STRIDE(i, n) {
    if (STAGE == CG_START) {
      // r: 1 + 0.01 (splitmix64((gx << 32) | gy) mod 1000) / 1000 on interior entries; p = z = D^-1 r
      const int32_t s = int32_t(i % nsl);
      double v = 0.0;
      const double di = dinv[i];
      if (gx[s] >= 0 && di != 0.0) {
        const uint64_t h = splitmix64((uint64_t(uint32_t(gx[s])) << 32) | uint64_t(uint32_t(gy[s])));
        v = 1.0 + 0.01 * double(h % 1000ull) / 1000.0;
      }
      const double zi = di * v;
      r[i] = v;
      z[i] = zi;
      p[i] = zi;
      if (sizeof(Q) == 4) pq[i] = Q(zi);
      acc += v * zi;
    } else if (STAGE == CG_PQ) {
      acc += p[i] * double(q[i]);
    } else {
      const double ri = r[i] - alpha * double(q[i]);
      const double zi = dinv[i] * ri;
      r[i] = ri;
      z[i] = zi;
      acc += ri * zi;
    }
  }
  sh[tid] = acc;
  __syncthreads();
  for (int o = TPB / 2; o > 0; o >>= 1) {
    if (tid < o) sh[tid] += sh[tid + o];
    __syncthreads();
  }
  if (tid == 0) {
    partial[blockIdx.x] = sh[0];
    __threadfence();
    last = atomicAdd(count, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  acc = 0.0;
  for (unsigned b = tid; b < gridDim.x; b += TPB) acc += __ldcg(partial + b);
  sh[tid] = acc;
  __syncthreads();
  for (int o = TPB / 2; o > 0; o >>= 1) {
    if (tid < o) sh[tid] += sh[tid + o];
    __syncthreads();
  }
  if (tid != 0) return;
  *count = 0u;   // for the next launch
  if (STAGE == CG_START) {
    sc[0] = sh[0];
    sc[5] = 1.0;
  } else if (STAGE == CG_PQ) {
    sc[1] = sh[0];
    const bool ok = sc[5] > 0.5 && sh[0] > 0.0 && sc[0] > 0.0;
    sc[3] = ok ? sc[0] / sh[0] : 0.0;
    if (!ok) sc[5] = 0.0;
  } else {
    sc[2] = sh[0];
    const bool ok = sc[5] > 0.5;
    const double beta = ok ? sh[0] / sc[0] : 0.0;
    sc[4] = beta;
    hist[2 * step + 0] = ok ? sc[3] : 0.0;
    hist[2 * step + 1] = beta;
    if (!(ok && sh[0] > 1e-300)) sc[5] = 0.0;
    sc[0] = sh[0];
  }
}

template <typename Q>
__global__ void k_cg_p(int64_t n, double* p, Q* pq, const double* __restrict__ z, const double* __restrict__ sc) {
  pdl_wait();
  pdl_trigger();
  const double beta = sc[4];
  GRID_STRIDE(i, n) {
    const double v = z[i] + beta * p[i];
    p[i] = v;
    if (sizeof(Q) == 4) pq[i] = Q(v);
  }
}

}  // namespace

template <typename T>
cudaError_t mg_chebyshev_first(int64_t n, T* x, T* xprev, const T* dinv, const T* d, T c0, cudaStream_t s, bool pdl) {
  if (n > 0) return launch_ex(pdl, &k_cheb_first<T>, blocks_for(n), TPB, 0, s, n, x, xprev, dinv, d, c0);
  return cudaGetLastError();
}
template <typename T>
cudaError_t mg_chebyshev_step(int64_t n, T* xnew, const T* x, const T* xprev, const T* dinv, const T* d,
                              const T* ax, T a, T b, cudaStream_t s, bool pdl) {
  if (n > 0) return launch_ex(pdl, &k_cheb_step<T>, blocks_for(n), TPB, 0, s, n, xnew, x, xprev, dinv, d, ax, a, b);
  return cudaGetLastError();
}
template <typename T>
cudaError_t mg_restrict(int32_t nc, int ncomp, int64_t ncs, int64_t nfs, const int32_t* ptr, const int32_t* col,
                        const float* val, const T* d_f, const T* ax_f, T* d_c, const uint8_t* cmask_c, int fixbits,
                        cudaStream_t s, bool pdl, const T* dinv_c, T* cur_c, T* prev_c, T c0) {
  if (nc > 0)
    return launch_ex(pdl, &k_restrict<T>, blocks_for(nc), TPB, 0, s, nc, ncomp, ncs, nfs, ptr, col, val, d_f, ax_f,
                     d_c, cmask_c, fixbits, dinv_c, cur_c, prev_c, c0);
  return cudaGetLastError();
}
template <typename T>
cudaError_t mg_prolong(int32_t nf, int ncomp, int64_t nfs, int64_t ncs, const int32_t* ptr, const int32_t* col,
                       const float* val, const T* x_c, T* x_f, const uint8_t* cmask_f, int fixbits, cudaStream_t s,
                       bool pdl) {
  if (nf > 0)
    return launch_ex(pdl, &k_prolong<T>, blocks_for(nf), TPB, 0, s, nf, ncomp, nfs, ncs, ptr, col, val, x_c, x_f,
                     cmask_f, fixbits);
  return cudaGetLastError();
}
template <typename T>
cudaError_t mg_copy_in(int64_t ns_leaf, int ncomp, DevHome home, const double* r, T* d, const uint8_t* leaf_cmask,
                       int fixbits, cudaStream_t s) {
  if (ns_leaf > 0) k_copy_in<T><<<blocks_for(ns_leaf), TPB, 0, s>>>(ns_leaf, ncomp, home, r, d, leaf_cmask, fixbits);
  return cudaGetLastError();
}
template <typename T>
cudaError_t mg_level_defects(int32_t nbricks, const LevBrick* bricks, const int32_t* home_leaf, int ncomp,
                             int64_t ns_leaf, const double* r, T* d, T* x0, const uint8_t* leaf_cmask, int fixbits,
                             cudaStream_t s) {
  if (nbricks > 0)
    k_level_defects<T><<<unsigned(nbricks), TPB, 0, s>>>(bricks, home_leaf, ncomp, ns_leaf, r, d, x0, leaf_cmask,
                                                         fixbits);
  return cudaGetLastError();
}
template <typename T>
cudaError_t mg_copy_out(int64_t ns_leaf, int ncomp, DevHome home, const T* x, const double* r, double* z,
                        const uint8_t* leaf_cmask, const uint8_t* leaf_flags, int fixbits, cudaStream_t s, bool pdl) {
  if (ns_leaf > 0)
    return launch_ex(pdl, &k_copy_out<T>, blocks_for(ns_leaf), TPB, 0, s, ns_leaf, ncomp, home, x, r, z, leaf_cmask,
                     leaf_flags, fixbits);
  return cudaGetLastError();
}
template <typename T>
cudaError_t mg_chebyshev_first_res(int64_t n, T* x, T* xprev, T* r, const T* dinv, const T* d, const T* ax, T c0,
                                   T* xadd, cudaStream_t s, bool pdl) {
  if (n > 0)
    return launch_ex(pdl, &k_cheb_first_res<T>, blocks_for(n), TPB, 0, s, n, x, xprev, r, dinv, d, ax, c0, xadd);
  return cudaGetLastError();
}
template <typename T>
cudaError_t mg_chebyshev_step_add(int64_t n, T* xadd, const T* x, const T* xprev, const T* dinv, const T* d,
                                  const T* ax, T a, T b, cudaStream_t s, bool pdl) {
  if (n > 0)
    return launch_ex(pdl, &k_cheb_step_add<T>, blocks_for(n), TPB, 0, s, n, xadd, x, xprev, dinv, d, ax, a, b);
  return cudaGetLastError();
}
template <typename T>
cudaError_t mg_coarse(int32_t n, const int32_t* idx, const double* Ainv, const T* d, T* x, cudaStream_t s, bool pdl) {
  if (n <= 0) return cudaSuccess;
  const int warps_per_block = TPB / 32;
  return launch_ex(pdl, &k_coarse_matvec<T>, unsigned((n + warps_per_block - 1) / warps_per_block), TPB, 0, s, n, idx,
                   Ainv, d, x);
}

cudaError_t mg_inject_lin(int32_t nbricks, const LevBrick* bricks, const int32_t* lev_leaf, const double* lin64,
                          int64_t ns_leaf, double* lev64, float* lev32, cudaStream_t s) {
  if (nbricks > 0) k_inject_lin<<<unsigned(nbricks), TPB, 0, s>>>(bricks, lev_leaf, lin64, ns_leaf, lev64, lev32);
  return cudaGetLastError();
}
cudaError_t mg_level_cmask(int32_t ns_l, const uint8_t* flags, const int32_t* slot_leaf, const uint8_t* leaf_cmask,
                           const int32_t* R_ptr, const int32_t* R_col, const uint8_t* cmask_fine, uint8_t* cmask,
                           cudaStream_t s) {
  if (ns_l > 0) k_level_cmask<<<blocks_for(ns_l), TPB, 0, s>>>(ns_l, flags, slot_leaf, leaf_cmask, R_ptr, R_col,
                                                                cmask_fine, cmask);
  return cudaGetLastError();
}
cudaError_t mg_invert_diag(int32_t ns_l, int ncomp, const double* diag, const uint8_t* flags, const uint8_t* cmask,
                           int fixbits, double* dinv64, float* dinv32, cudaStream_t s) {
  if (ns_l > 0) k_invert_diag<<<blocks_for(ns_l), TPB, 0, s>>>(ns_l, ncomp, diag, flags, cmask, fixbits, dinv64,
                                                                dinv32);
  return cudaGetLastError();
}
cudaError_t dot64(int64_t n, const double* a, const double* b, double* partial, double* out, cudaStream_t s) {
  k_dot_partial<<<DOT_BLOCKS, TPB, 0, s>>>(n, a, b, partial);
  k_dot_final<<<1, TPB, 0, s>>>(DOT_BLOCKS, partial, out);
  return cudaGetLastError();
}
template <typename Q>
cudaError_t cg_start(int64_t n, int32_t ns_l, const int32_t* gx, const int32_t* gy, const CgChain<Q>& c, cudaStream_t s) {
  const unsigned grid = unsigned(std::min<int64_t>(DOT_BLOCKS, std::max<int64_t>(1, (n + TPB - 1) / TPB)));
  return launch_ex(true, &k_cg<CG_START, Q>, grid, unsigned(TPB), 0, s, n, ns_l, gx, gy, c.dinv, c.r, c.z, c.p, c.pq,
                   static_cast<const Q*>(c.q), c.sc, c.hist, 0, c.partial, c.count);
}
template <typename Q>
cudaError_t cg_step(int64_t n, const CgChain<Q>& c, int step, cudaStream_t s) {
  const unsigned grid = unsigned(std::min<int64_t>(DOT_BLOCKS, std::max<int64_t>(1, (n + TPB - 1) / TPB)));
  const int32_t* none = nullptr;
  cudaError_t e = launch_ex(true, &k_cg<CG_PQ, Q>, grid, unsigned(TPB), 0, s, n, 1, none, none, c.dinv, c.r, c.z, c.p,
                            c.pq, static_cast<const Q*>(c.q), c.sc, c.hist, step, c.partial, c.count);
  if (e == cudaSuccess)
    e = launch_ex(true, &k_cg<CG_RZ, Q>, grid, unsigned(TPB), 0, s, n, 1, none, none, c.dinv, c.r, c.z, c.p, c.pq,
                  static_cast<const Q*>(c.q), c.sc, c.hist, step, c.partial, c.count);
  if (e == cudaSuccess)
    e = launch_ex(true, &k_cg_p<Q>, blocks_for(n), unsigned(TPB), 0, s, n, c.p, c.pq,
                  static_cast<const double*>(c.z), static_cast<const double*>(c.sc));
  return e;
}
template cudaError_t cg_start<float>(int64_t, int32_t, const int32_t*, const int32_t*, const CgChain<float>&, cudaStream_t);
template cudaError_t cg_start<double>(int64_t, int32_t, const int32_t*, const int32_t*, const CgChain<double>&, cudaStream_t);
template cudaError_t cg_step<float>(int64_t, const CgChain<float>&, int, cudaStream_t);
template cudaError_t cg_step<double>(int64_t, const CgChain<double>&, int, cudaStream_t);
int mg_dot_partials() { return DOT_BLOCKS; }
#define INST(T)                                                                                                \
  template cudaError_t mg_chebyshev_first<T>(int64_t, T*, T*, const T*, const T*, T, cudaStream_t, bool);     \
  template cudaError_t mg_chebyshev_step<T>(int64_t, T*, const T*, const T*, const T*, const T*, const T*, T,  \
                                            T, cudaStream_t, bool);                                            \
  template cudaError_t mg_restrict<T>(int32_t, int, int64_t, int64_t, const int32_t*, const int32_t*,          \
                                      const float*, const T*, const T*, T*, const uint8_t*, int, cudaStream_t, \
                                      bool, const T*, T*, T*, T);                                              \
  template cudaError_t mg_prolong<T>(int32_t, int, int64_t, int64_t, const int32_t*, const int32_t*,           \
                                     const float*, const T*, T*, const uint8_t*, int, cudaStream_t, bool);     \
  template cudaError_t mg_copy_in<T>(int64_t, int, DevHome, const double*, T*, const uint8_t*, int, cudaStream_t); \
  template cudaError_t mg_level_defects<T>(int32_t, const LevBrick*, const int32_t*, int, int64_t, const double*, T*, \
                                           T*, const uint8_t*, int, cudaStream_t);                              \
  template cudaError_t mg_copy_out<T>(int64_t, int, DevHome, const T*, const double*, double*, const uint8_t*,     \
                                      const uint8_t*, int, cudaStream_t, bool);                                    \
  template cudaError_t mg_chebyshev_first_res<T>(int64_t, T*, T*, T*, const T*, const T*, const T*, T, T*,        \
                                                 cudaStream_t, bool);                                              \
  template cudaError_t mg_chebyshev_step_add<T>(int64_t, T*, const T*, const T*, const T*, const T*, const T*, T, \
                                                T, cudaStream_t, bool);                                            \
  template cudaError_t mg_coarse<T>(int32_t, const int32_t*, const double*, const T*, T*, cudaStream_t, bool);
INST(float)
INST(double)
#undef INST

}  // namespace pff
