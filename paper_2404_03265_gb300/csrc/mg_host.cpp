// Host driver of the block-diagonal geometric multigrid preconditioner.
//
// Kolditz & Wick (arXiv 2404.03265), Sec. 3.2: one V-cycle per diagonal block
// (u-u, phi-phi) of the Jacobian; Chebyshev-accelerated Jacobi smoothing with
// the inverse diagonal from cell-local assembly and a CG-based estimate of the
// largest eigenvalue, smoothing range [0.08, 1.2] * lambda_max; local
// smoothing on the level meshes; coarse level solved directly (FP64).
//
// V-cycle of one block (levels L..1, coarse 0):
//   copy the leaf defect to the coarsest level on which each DoF is interior;
//   down: Chebyshev from zero, defect d - A x on interior and edge rows,
//         restriction P^T into the next coarser level;
//   coarse: x_0 = A_0^{-1} d_0 on the interior;
//   up: x += P x_coarse on all level nodes, Chebyshev on d - A x;
//   copy the level solutions back to the leaf DoFs (fixed leaf rows: z = r).
#include <algorithm>
#include <cmath>
#include <cstring>

#include "solve.cuh"
#include "state.h"

namespace pff {

namespace {

constexpr int kMaxLanczos = 64;   // CG coefficient pairs stored per set-up chain

inline int block_op(int b) { return b == 0 ? OP_UU : OP_PP; }
inline int block_diag_op(int b) { return b == 0 ? OP_UU_DIAG : OP_PP_DIAG; }

// Largest eigenvalue of the symmetric tridiagonal matrix (d, e) by bisection on Sturm counts.
double tridiag_max_eig(const std::vector<double>& d, const std::vector<double>& e) {
  const int m = int(d.size());
  if (m == 0) return 0.0;
  double lo = d[0], hi = d[0];
  for (int i = 0; i < m; ++i) {
    const double r = (i > 0 ? std::fabs(e[i - 1]) : 0.0) + (i < m - 1 ? std::fabs(e[i]) : 0.0);
    lo = std::min(lo, d[i] - r);
    hi = std::max(hi, d[i] + r);
  }
  auto count_below = [&](double x) {  // eigenvalues < x
    int c = 0;
    double q = d[0] - x;
    if (q < 0) ++c;
    for (int i = 1; i < m; ++i) {
      const double qq = (q == 0.0) ? 1e-300 : q;
      q = d[i] - x - e[i - 1] * e[i - 1] / qq;
      if (q < 0) ++c;
    }
    return c;
  };
  for (int it = 0; it < 200 && hi - lo > 1e-15 * std::max(std::fabs(hi), 1e-300); ++it) {
    const double mid = 0.5 * (lo + hi);
    if (count_below(mid) == m) hi = mid; else lo = mid;
  }
  return 0.5 * (lo + hi);
}

// Smallest eigenvalue of the same symmetric tridiagonal matrix (bisection on the Sturm count).
double tridiag_min_eig(const std::vector<double>& d, const std::vector<double>& e) {
  const int m = int(d.size());
  if (m == 0) return 0.0;
  double lo = d[0], hi = d[0];
  for (int i = 0; i < m; ++i) {
    const double r = (i > 0 ? std::fabs(e[i - 1]) : 0.0) + (i < m - 1 ? std::fabs(e[i]) : 0.0);
    lo = std::min(lo, d[i] - r);
    hi = std::max(hi, d[i] + r);
  }
  auto count_below = [&](double x) {
    int c = 0;
    double q = d[0] - x;
    if (q < 0) ++c;
    for (int i = 1; i < m; ++i) {
      const double qq = (q == 0.0) ? 1e-300 : q;
      q = d[i] - x - e[i - 1] * e[i - 1] / qq;
      if (q < 0) ++c;
    }
    return c;
  };
  for (int it = 0; it < 200 && hi - lo > 1e-15 * std::max(std::fabs(hi), 1e-300); ++it) {
    const double mid = 0.5 * (lo + hi);
    if (count_below(mid) >= 1) hi = mid; else lo = mid;
  }
  return 0.5 * (lo + hi);
}

// Smallest degree m with 1 / T_m((b + a) / (b - a)) <= tol (Chebyshev error bound on [a, b]).
int chebyshev_degree(double a, double b, double tol = 1e-3, int cap = 64) {
  const double sigma = (b + a) / (b - a);
  for (int m = 1; m <= cap; ++m)
    if (1.0 / std::cosh(m * std::acosh(sigma)) <= tol) return m;
  return cap;
}

#define CK(call)                                              \
  do {                                                        \
    cudaError_t e_ = (call);                                  \
    if (e_ != cudaSuccess) return std::string(#call) + ": " + cudaGetErrorString(e_); \
  } while (0)

}  // namespace

// arguments of a level operator in precision T, but for its vectors
template <typename T>
static ApplyArgs level_args(pff_mg& mg, int level) {
  pff_problem& pb = *mg.pb;
  const Mesh& M = pb.mesh->m;
  const DevMesh::Level& L = pb.mesh->dev.levels[level];
  ApplyArgs a;
  std::memset(&a, 0, sizeof(a));
  a.lay = L.lay;
  a.hang = nullptr;
  a.cmask = mg.cmask + L.lv.off;
  const int64_t n = L.lv.n_slots;
  if (sizeof(T) == 8) a.lin = mg.lin64 + 4 * L.lv.off; else a.lin = mg.lin32 + 4 * L.lv.off;
  a.n_slots = n;
  for (int l = 0; l <= M.Lf && l < kMaxLevels; ++l) { a.hx[l] = M.tree.hx(l); a.hy[l] = M.tree.hy(l); }
  fill_material(pb.prm, a, pb.has_ecell);
  if (pb.has_ecell) {
    if (sizeof(T) == 8) a.ecell = pb.lev_ecell64 + L.lv.off; else a.ecell = pb.lev_ecell32 + L.lv.off;
  }
  fill_cell_constants(a, M.Lf + 1);
  a.fe_degree = M.k;
  a.sweep_sh = pb.sweep_sh;
  a.mode = MODE_MASK_INPUT;
  return a;
}

// pdl: launched dependent on the preceding kernel of the stream (the V-cycle chain)
template <typename T>
cudaError_t level_apply(pff_mg& mg, int level, int op, const T* x, T* y, cudaStream_t s, bool pdl,
                        const ChebEpi* ch) {
  ApplyArgs a = level_args<T>(mg, level);
  a.xu = x; a.xp = x; a.yu = y; a.yp = y;
  a.pdl_in = pdl ? 1 : 0;
  if (ch) a.ch = *ch;
  return launch_apply<T>(a, op, s);
}

std::string mg_alloc(pff_mg& mg) {
  const DevMesh& D = mg.pb->mesh->dev;
  const int64_t N = D.lev_total;
  const int64_t ns = mg.pb->mesh->m.lay.n_slots;
  const int nchain = 2 * int(D.levels.size());
  // Cleared: slots without a node keep a zero inverse diagonal and zero CG vectors, and the
  // counters are 0 between launches.
  for (int b = 0; b < 2; ++b) {
    MGBlock& B = mg.blk[b];
    B.ncomp = b == 0 ? 2 : 1;
    B.fixbits = b == 0 ? 3 : 4;
    mg.mem.reserve(B.dinv64, B.ncomp * N);
    mg.mem.reserve(B.dinv32, B.ncomp * N);
    mg.mem.reserve(mg.su_vec[b], 5 * B.ncomp * N);
    B.lam.assign(D.levels.size(), 0.0);
  }
  mg.mem.reserve(mg.su_count, nchain);
  mg.mem.reserve(mg.spd_bad, 2);
  mg.mem.commit(true);
  mg.mem.reserve(mg.vc_in, 3 * ns);
  mg.mem.reserve(mg.vc_out, 3 * ns);
  mg.mem.reserve(mg.lin64, 4 * N);
  mg.mem.reserve(mg.lin32, 4 * N);
  mg.mem.reserve(mg.cmask, N);
  for (MGBlock& B : mg.blk)
    for (void** p : {&B.d, &B.x, &B.r, &B.y, &B.yp, &B.t})
      mg.mem.reserve(reinterpret_cast<unsigned char*&>(*p),
                     size_t(B.ncomp) * N * (mg.precision == PFF_F64 ? sizeof(double) : sizeof(float)));
  mg.mem.reserve(mg.su_partial, int64_t(nchain) * mg_dot_partials());
  mg.mem.reserve(mg.su_sc, 8 * nchain);
  mg.mem.reserve(mg.su_hist, 2 * kMaxLanczos * nchain);
  for (int b = 0; b < 2; ++b) mg.mem.reserve(mg.su_part[b], 512 * D.levels.size());
  mg.mem.commit();
  if (!mg.mem.err.empty()) return mg.mem.err;
  mg.host_len = size_t(2) * kMaxLanczos * nchain;
  if (cudaMallocHost(reinterpret_cast<void**>(&mg.host), mg.host_len * sizeof(double) + 2 * sizeof(int32_t)) != cudaSuccess) {
    mg.host = nullptr;
    return "cudaMallocHost failed";
  }
  return "";
}

// Tables and buffers of the direct coarse solve, made by the first set-up that needs them:
// the entries of each block (every component of every level-0 node but Dirichlet ones),
// the grid's node slots, element matrices, the dense blocks and the inversion's scratch.
static std::string coarse_alloc(pff_mg& mg) {
  const Mesh& M = mg.pb->mesh->m;
  DevAllocs& mem = mg.coarse_mem;
  mem.release();   // (what an attempt cut short by an exception left)
  const DevMesh& D = mg.pb->mesh->dev;
  const LevelMesh& lm = M.levels[0];
  const int32_t n0 = D.levels[0].lv.n_slots;
  const int k = M.k, ncx = M.tree.ncx, ncy = M.tree.ncy, nx = k * ncx + 1;
  std::vector<int32_t> node_slot(size_t(nx) * (k * ncy + 1), 0);
  for (int32_t s = 0; s < n0; ++s)
    if (lm.slot_X[s] >= 0) node_slot[size_t(lm.slot_X[s] >> M.Lf) + size_t(nx) * (lm.slot_Y[s] >> M.Lf)] = s;
  CoarseArgs& a = mg.coarse;
  std::memset(&a, 0, sizeof(a));
  for (int b = 0; b < 2; ++b) {
    MGBlock& B = mg.blk[b];
    std::vector<int32_t> idx, ent(size_t(B.ncomp) * n0, -1);
    for (int32_t s = 0; s < n0; ++s)
      for (int c = 0; c < B.ncomp; ++c)
        if (lm.slot_X[s] >= 0 && !(b == 0 && (lm.slot_flags[s] & 2))) {
          ent[size_t(c) * n0 + s] = int32_t(idx.size());
          idx.push_back(c * n0 + s);
        }
    const int nd = (k + 1) * (k + 1) * B.ncomp;
    CoarseBlock& q = a.b[b];
    q.n = int32_t(idx.size());
    q.nc = B.ncomp;
    q.fix0 = b == 0 ? 1 : 4;
    B.coarse_idx = mem.alloc<int32_t>(idx.size());
    q.all = mem.upload(idx);
    q.idx = B.coarse_idx;
    q.ent = mem.upload(ent);
    q.Ke = mem.alloc<double>(size_t(ncx) * ncy * nd * nd);
    B.coarse_inv = mem.alloc<double>(size_t(q.n) * q.n);
    q.A = B.coarse_inv;
    q.scr = mem.alloc<double>(size_t(coarse_scratch(q.n)));
    B.n_coarse = q.n;
  }
  a.k = k; a.ncx = ncx; a.ncy = ncy;
  a.n0 = n0;
  a.node_slot = mem.upload(node_slot);
  a.gx = D.levels[0].gx;
  a.gy = D.levels[0].gy;
  a.cmask = mg.cmask;   // level 0 comes first
  a.bad = mg.spd_bad;
  std::string err = mem.err;
  if (!err.empty()) {   // give everything back: a later set-up starts afresh
    mem.release();
    std::memset(&a, 0, sizeof(a));
    for (MGBlock& B : mg.blk) {
      B.coarse_idx = nullptr;
      B.coarse_inv = nullptr;
      B.n_coarse = 0;
    }
  }
  mg.coarse_ready = err.empty();
  return err;
}

// The direct coarse solve's blocks on stream t: element matrices, assembly, inversion
static cudaError_t launch_coarse_setup(pff_mg& mg, cudaStream_t t) {
  const CoarseArgs& a = mg.coarse;
  const ApplyArgs k = level_args<double>(mg, 0);
  cudaError_t e = cudaSuccess;
  for (int b = 0; b < 2 && e == cudaSuccess; ++b)
    if (a.b[b].n > 0) e = launch_coarse_elements(k, block_op(b), a.ncx, a.ncx * a.ncy, a.node_slot, a.b[b].Ke, t);
  if (e == cudaSuccess) e = coarse_fill(a, t);
  if (e == cudaSuccess) e = coarse_invert(a, t);
  return e;
}

// Per Newton step: level linearisation, level constraint masks, inverse
// diagonals, eigenvalue estimates and the coarse inverse of both blocks.
void mg_release_graphs(pff_mg& mg) {
  for (int g = 0; g < 3; ++g) {
    if (mg.vc_exec[g]) { cudaGraphExecDestroy(mg.vc_exec[g]); mg.vc_exec[g] = nullptr; }
    if (mg.vc_graph[g]) { cudaGraphDestroy(mg.vc_graph[g]); mg.vc_graph[g] = nullptr; }
  }
}

void mg_release_setup_graph(pff_mg& mg) {
  if (mg.su_exec) { cudaGraphExecDestroy(mg.su_exec); mg.su_exec = nullptr; }
  mg.su_key.clear();
}

// The CG run of one (block, level) chain on stream t.  Its vectors, dot products
// and coefficients are FP64; the level apply q = A p runs in precision Q.  In FP32, p is
// rounded into and q read from two FP32 vectors that take the chain's diagonal slot (free
// once the inverse diagonal is formed): the apply's rounding is relative to its operands,
// so the small residuals of a converging run keep their accuracy.
template <typename Q>
static cudaError_t setup_cg(pff_mg& mg, int b, int l, cudaStream_t t) {
  const DevMesh& D = mg.pb->mesh->dev;
  const int nl = int(D.levels.size());
  const int64_t N = D.lev_total;
  MGBlock& B = mg.blk[b];
  const DevLevel& lv = D.levels[l].lv;
  const int64_t nn = B.ncomp * int64_t(lv.n_slots), o = B.ncomp * lv.off, vs = B.ncomp * N;
  const int c = b * nl + l;
  CgChain<Q> g;
  g.dinv = B.dinv64 + o;
  g.r = mg.su_vec[b] + vs + o;
  g.z = mg.su_vec[b] + 2 * vs + o;
  g.p = mg.su_vec[b] + 3 * vs + o;
  if constexpr (sizeof(Q) == 4) {
    g.pq = reinterpret_cast<Q*>(mg.su_vec[b] + o);
    g.q = g.pq + nn;
  } else {
    g.pq = g.p;
    g.q = mg.su_vec[b] + 4 * vs + o;
  }
  g.sc = mg.su_sc + 8 * c;
  g.hist = mg.su_hist + 2 * kMaxLanczos * c;
  g.partial = mg.su_partial + int64_t(c) * mg_dot_partials();
  g.count = mg.su_count + c;
  cudaError_t e = cg_start<Q>(nn, lv.n_slots, D.levels[l].gx, D.levels[l].gy, g, t);
  const bool q1 = mg.pb->mesh->m.k == 1;   // (the Q2 kernel does not wait for its predecessor)
  for (int j = 0; j < mg.lanczos_steps && e == cudaSuccess; ++j) {
    e = level_apply<Q>(mg, l, block_op(b), g.pq, g.q, t, q1);
    if (e == cudaSuccess) e = cg_step<Q>(nn, g, j, t);
  }
  return e;
}

// Arguments of the tiled set-up of block b (setup.cu)
static SetupArgs setup_args(pff_mg& mg, int b) {
  pff_problem& pb = *mg.pb;
  const Mesh& M = pb.mesh->m;
  const DevMesh& D = pb.mesh->dev;
  const int nl = int(D.levels.size());
  const MGBlock& B = mg.blk[b];
  const int64_t vs = B.ncomp * D.lev_total;
  ApplyArgs k;
  std::memset(&k, 0, sizeof(k));
  for (int l = 0; l <= M.Lf && l < kMaxLevels; ++l) { k.hx[l] = M.tree.hx(l); k.hy[l] = M.tree.hy(l); }
  fill_material(pb.prm, k, pb.has_ecell);
  fill_cell_constants(k, M.Lf + 1);
  SetupArgs a;
  std::memset(&a, 0, sizeof(a));
  a.tiles = D.setup_tiles; a.ntiles = D.n_setup_tiles;
  a.flags = D.lev_flags; a.cmask = mg.cmask;
  a.lin64 = mg.lin64; a.lin32 = mg.lin32;
  a.ecell64 = pb.has_ecell ? pb.lev_ecell64 : nullptr;
  a.ecell32 = pb.has_ecell ? pb.lev_ecell32 : nullptr;
  a.gx = D.lev_gx; a.gy = D.lev_gy;
  a.dinv64 = B.dinv64; a.dinv32 = B.dinv32;
  a.q = reinterpret_cast<float*>(mg.su_vec[b]);
  a.r = mg.su_vec[b] + vs;
  a.z = mg.su_vec[b] + 2 * vs;
  a.p[0] = mg.su_vec[b] + 3 * vs;
  a.p[1] = mg.su_vec[b] + 4 * vs;
  a.sc = mg.su_sc + 8 * b * nl;
  a.hist = mg.su_hist + 2 * kMaxLanczos * b * nl;
  a.hist_stride = 2 * kMaxLanczos;
  a.partial = mg.su_part[b];
  a.count = mg.su_count + b * nl;
  a.tile1 = nl > 1 ? D.levels[1].tile0 : a.ntiles;
  for (int l = 0; l < nl; ++l) {
    a.off[l] = int32_t(D.levels[l].lv.off);
    a.n[l] = D.levels[l].lv.n_slots;
    a.dot0[l + 1] = a.dot0[l] + (l == 0 ? 0 : setup_dot_blocks(B.ncomp * int64_t(a.n[l])));
  }
  for (int l = nl; l < kMaxLevels; ++l) a.dot0[l + 1] = a.dot0[nl];
  a.mf = k.mf; a.md = k.md;
  for (int l = 0; l < kMaxLevels; ++l) { a.gf[l] = k.gf[l]; a.gd[l] = k.gd[l]; }
  return a;
}

// Launches of the set-up chains on the pool streams: inverse diagonals (FP64, cast to both
// precisions) and CG runs (applies in the V-cycle's precision; level 0, for the Chebyshev
// coarse solver: FP64); on the extra stream K the direct coarse solve's blocks.
//  - FP32, Q1, default cell loop: all levels of a block in shared launches (setup.cu).
//  - else one chain per (block, level), finest levels first, spread over the pool.
static cudaError_t launch_setup_chains(pff_mg& mg) {
  pff_problem& pb = *mg.pb;
  const DevMesh& D = pb.mesh->dev;
  const int nl = int(D.levels.size());
  constexpr int K = pff_mg::kSetupStreams;
  cudaError_t e = cudaSuccess;
  if (mg.precision == PFF_F32 && pb.mesh->m.k == 1 && pb.sweep_sh == 0) {
    for (int b = 0; b < 2 && e == cudaSuccess; ++b) {
      const SetupArgs a = setup_args(mg, b);
      e = launch_setup_diag(a, block_op(b), mg.su_stream[b]);
      if (e == cudaSuccess) e = launch_setup_cg(a, block_op(b), mg.lanczos_steps, mg.su_stream[b]);
      if (e == cudaSuccess && mg.coarse_mode != 0) e = setup_cg<double>(mg, b, 0, mg.su_stream[b]);
    }
  } else {
    int chain = 0;
    for (int l = nl - 1; l >= 0; --l)
      for (int b = 0; b < 2; ++b, ++chain) {
        cudaStream_t t = mg.su_stream[chain % K];
        MGBlock& B = mg.blk[b];
        const DevLevel& lv = D.levels[l].lv;
        const int64_t o = B.ncomp * lv.off;
        double* diag = mg.su_vec[b] + o;
        e = level_apply<double>(mg, l, block_diag_op(b), diag, diag, t);
        if (e == cudaSuccess)
          e = mg_invert_diag(lv.n_slots, B.ncomp, diag, lv.flags, mg.cmask + lv.off, B.fixbits, B.dinv64 + o,
                             B.dinv32 + o, t);
        if (e != cudaSuccess) return e;
        if (l == 0 && mg.coarse_mode == 0) continue;
        e = mg.precision == PFF_F32 && l > 0 ? setup_cg<float>(mg, b, l, t) : setup_cg<double>(mg, b, l, t);
        if (e != cudaSuccess) return e;
      }
  }
  if (e == cudaSuccess && mg.coarse_mode == 0) e = launch_coarse_setup(mg, mg.su_stream[K]);
  return e;
}

// What the chains' captured launches depend on besides fixed buffers
static std::vector<unsigned char> setup_key(const pff_mg& mg) {
  const pff_problem& pb = *mg.pb;
  std::vector<unsigned char> k;
  auto put = [&](const void* v, size_t n) {
    const unsigned char* c = static_cast<const unsigned char*>(v);
    k.insert(k.end(), c, c + n);
  };
  put(&pb.prm, sizeof(pb.prm));
  put(&pb.has_ecell, sizeof(pb.has_ecell));
  put(&pb.lev_ecell64, sizeof(pb.lev_ecell64));
  put(&pb.lev_ecell32, sizeof(pb.lev_ecell32));
  put(&pb.sweep_sh, sizeof(pb.sweep_sh));
  put(&mg.coarse_mode, sizeof(mg.coarse_mode));
  put(&mg.lanczos_steps, sizeof(mg.lanczos_steps));
  put(&mg.precision, sizeof(mg.precision));
  return k;
}

// Capture the chains: a fork from the capture stream to the pool, the chains, a
// join back; false (no graph) if any step fails
static bool capture_setup_chains(pff_mg& mg) {
  constexpr int K = pff_mg::kSetupStreams;
  if (!mg.cap_stream && cudaStreamCreateWithFlags(&mg.cap_stream, cudaStreamNonBlocking) != cudaSuccess) return false;
  if (cudaStreamBeginCapture(mg.cap_stream, cudaStreamCaptureModeThreadLocal) != cudaSuccess) return false;
  cudaError_t e = cudaEventRecord(mg.su_start, mg.cap_stream);
  for (int i = 0; i <= K && e == cudaSuccess; ++i) e = cudaStreamWaitEvent(mg.su_stream[i], mg.su_start, 0);
  if (e == cudaSuccess) e = launch_setup_chains(mg);
  for (int i = 0; i <= K && e == cudaSuccess; ++i) {
    e = cudaEventRecord(mg.su_done[i], mg.su_stream[i]);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(mg.cap_stream, mg.su_done[i], 0);
  }
  cudaGraph_t g = nullptr;
  const cudaError_t e2 = cudaStreamEndCapture(mg.cap_stream, &g);
  bool ok = e == cudaSuccess && e2 == cudaSuccess && g != nullptr;
  if (ok) ok = cudaGraphInstantiate(&mg.su_exec, g, 0) == cudaSuccess;
  if (g) cudaGraphDestroy(g);
  if (!ok) {
    mg.su_exec = nullptr;
    cudaGetLastError();   // clear a capture error; the chains are launched directly
  }
  return ok;
}

// Lambda_max (and on level 0 the Chebyshev interval) of one (block, level) from
// the CG coefficients alpha_j, beta_j of its chain: the Lanczos tridiagonal
// d_j = 1/alpha_j + beta_{j-1}/alpha_{j-1}, e_j = sqrt(beta_j)/alpha_j.
static void eigen_from_cg(pff_mg& mg, MGBlock& B, int l, const double* hist) {
  std::vector<double> al, be;
  for (int j = 0; j < mg.lanczos_steps; ++j) {
    if (!(hist[2 * j] > 0)) break;
    al.push_back(hist[2 * j]);
    be.push_back(hist[2 * j + 1]);
  }
  const int m = int(al.size());
  std::vector<double> dd(m), ee(m > 0 ? m - 1 : 0);
  for (int j = 0; j < m; ++j) dd[j] = 1.0 / al[j] + (j > 0 ? be[j - 1] / al[j - 1] : 0.0);
  for (int j = 0; j + 1 < m; ++j) ee[j] = std::sqrt(std::max(be[j], 0.0)) / al[j];
  B.lam[l] = tridiag_max_eig(dd, ee);
  if (l == 0 && B.lam[0] > 0.0) {
    // Chebyshev coarse solver: both Ritz extremes of the same CG run
    B.c0_a = 0.9 * tridiag_min_eig(dd, ee);
    B.c0_b = 1.2 * B.lam[0];
    B.c0_deg = B.c0_a > 0.0 ? chebyshev_degree(B.c0_a, B.c0_b) : 0;
  }
}

std::string mg_setup(pff_mg& mg, cudaStream_t s) {
  mg_release_graphs(mg);   // the V-cycle graphs hold this set-up's coefficients
  pff_problem& pb = *mg.pb;
  const Mesh& M = pb.mesh->m;
  const DevMesh& D = pb.mesh->dev;
  const int nl = int(D.levels.size());
  const int64_t nsleaf = M.lay.n_slots;
  const int64_t N = D.lev_total;
  if (mg.lanczos_steps > kMaxLanczos) return "too many Lanczos steps";
  CK(mg_inject_lin(D.n_lev_bricks, D.lev_bricks, D.lev_leaf, pb.lin64, nsleaf, mg.lin64, mg.lin32, s));
  for (int l = nl - 1; l >= 0; --l) {
    const DevLevel& lv = D.levels[l].lv;
    const DevLevel* fine = (l + 1 < nl) ? &D.levels[l + 1].lv : nullptr;
    CK(mg_level_cmask(lv.n_slots, lv.flags, lv.slot_leaf, pb.cmask, fine ? fine->R_ptr : nullptr,
                      fine ? fine->R_col : nullptr, fine ? mg.cmask + fine->off : nullptr, mg.cmask + lv.off, s));
  }
  // Inverse diagonals, then the Jacobi-preconditioned CG runs whose coefficients give
  // lambda_max of D^-1 A on the interior (level 0: only for the Chebyshev coarse solver);
  // on the extra pool stream K the direct coarse solve's blocks.  The chains share no
  // buffer.  From the second set-up on they replay as one graph on su_side (re-captured
  // when their arguments change).
  constexpr int K = pff_mg::kSetupStreams;
  if (!mg.su_start) CK(cudaEventCreateWithFlags(&mg.su_start, cudaEventDisableTiming));
  if (!mg.su_chains) CK(cudaEventCreateWithFlags(&mg.su_chains, cudaEventDisableTiming));
  if (!mg.su_side) CK(cudaStreamCreateWithFlags(&mg.su_side, cudaStreamNonBlocking));
  for (int i = 0; i <= K; ++i) {
    if (!mg.su_stream[i]) CK(cudaStreamCreateWithFlags(&mg.su_stream[i], cudaStreamNonBlocking));
    if (!mg.su_done[i]) CK(cudaEventCreateWithFlags(&mg.su_done[i], cudaEventDisableTiming));
  }
  for (int b = 0; b < 2; ++b) {
    MGBlock& B = mg.blk[b];
    for (int l = 0; l < nl; ++l) B.lam[l] = 0.0;
    B.c0_a = B.c0_b = 0.0;
    B.c0_deg = 0;
  }
  if (mg.coarse_mode == 0 && !mg.coarse_ready) {
    mg.settled = false;
    const std::string e = coarse_alloc(mg);
    if (!e.empty()) return e;
  }
  if (!mg.settled) CK(after_clears(s));
  bool replay = false;
  if (mg.su_graph_ok && mg.su_setups > 0) {
    std::vector<unsigned char> key = setup_key(mg);
    if (mg.su_exec && key != mg.su_key) mg_release_setup_graph(mg);
    if (!mg.su_exec) {
      if (capture_setup_chains(mg)) mg.su_key = key;
      else mg.su_graph_ok = false;
    }
    replay = mg.su_exec != nullptr;
  }
  ++mg.su_setups;
  CK(cudaEventRecord(mg.su_start, s));
  if (replay) {
    CK(cudaStreamWaitEvent(mg.su_side, mg.su_start, 0));
    CK(cudaGraphLaunch(mg.su_exec, mg.su_side));
    CK(cudaEventRecord(mg.su_chains, mg.su_side));
    CK(cudaStreamWaitEvent(s, mg.su_chains, 0));
  } else {
    for (int i = 0; i <= K; ++i) CK(cudaStreamWaitEvent(mg.su_stream[i], mg.su_start, 0));
    CK(launch_setup_chains(mg));
    for (int i = 0; i <= K; ++i) {
      CK(cudaEventRecord(mg.su_done[i], mg.su_stream[i]));
      CK(cudaStreamWaitEvent(s, mg.su_done[i], 0));
    }
  }
  // the CG coefficients and the coarse status in one host read (pinned)
  double* hist = mg.host;
  int32_t* bad = reinterpret_cast<int32_t*>(mg.host + mg.host_len);
  bad[0] = bad[1] = 0;
  CK(cudaMemcpyAsync(hist, mg.su_hist, mg.host_len * sizeof(double), cudaMemcpyDeviceToHost, s));
  if (mg.coarse_mode == 0) CK(cudaMemcpyAsync(bad, mg.spd_bad, 2 * sizeof(int32_t), cudaMemcpyDeviceToHost, s));
  CK(cudaStreamSynchronize(s));
  mg.settled = true;
  if (bad[0] || bad[1]) return "coarse level block is not positive definite";
  for (int b = 0; b < 2; ++b)
    for (int l = 0; l < nl; ++l) {
      if (l == 0 && mg.coarse_mode == 0) continue;
      eigen_from_cg(mg, mg.blk[b], l, hist + size_t(b * nl + l) * 2 * kMaxLanczos);
    }
  mg.ready = true;
  return "";
}

namespace {

// While a V-cycle graph is captured: the node of the kernel just launched on s, which
// takes nargs arguments, r at position r_arg and z at z_arg (-1: not)
cudaError_t note_node(pff_mg& mg, int b, int which, int nargs, int r_arg, int z_arg, cudaStream_t s) {
  if (!mg.vc_note[b]) return cudaSuccess;
  cudaStreamCaptureStatus st;
  const cudaGraphNode_t* dep = nullptr;
  size_t n = 0;
  const cudaError_t e = cudaStreamGetCaptureInfo(s, &st, nullptr, nullptr, &dep, nullptr, &n);
  if (e != cudaSuccess) return e;
  if (st != cudaStreamCaptureStatusActive || n != 1) return cudaErrorUnknown;
  pff_mg::VcIo& io = *mg.vc_note[b];
  io.node[which] = dep[0];
  io.arg[which].resize(size_t(nargs));
  io.r_arg[which] = r_arg;
  if (which == 1) io.z_arg = z_arg;
  return cudaSuccess;
}

template <typename T>
cudaError_t vcycle_t(pff_mg& mg, int b, const double* r, double* z, cudaStream_t s) {
  pff_problem& pb = *mg.pb;
  const Mesh& M = pb.mesh->m;
  const DevMesh& D = pb.mesh->dev;
  MGBlock& B = mg.blk[b];
  const int nc = B.ncomp, nl = int(D.levels.size());
  const int64_t N = D.lev_total;
  const int64_t nsleaf = M.lay.n_slots;
  T* d = static_cast<T*>(B.d);
  T* x = static_cast<T*>(B.x);
  T* rr = static_cast<T*>(B.r);
  T* y = static_cast<T*>(B.y);
  T* yp = static_cast<T*>(B.yp);
  T* t = static_cast<T*>(B.t);
  const T* dinv = sizeof(T) == 8 ? reinterpret_cast<const T*>(B.dinv64) : reinterpret_cast<const T*>(B.dinv32);
  cudaError_t e;
#define VC(call) do { e = (call); if (e != cudaSuccess) return e; } while (0)
  // each Chebyshev step is the store of the level apply that applies A
  const bool fuse = mg.fused != 0;
  auto epi = [&](int mode, const T* prev, const T* dinv_l, const T* rhs, T* out, T* r_out, T* xprev_out, double ca,
                 double cb) {
    ChebEpi c;
    std::memset(&c, 0, sizeof(c));
    c.mode = mode; c.prev = prev; c.dinv = dinv_l; c.rhs = rhs; c.out = out; c.r = r_out; c.xprev = xprev_out;
    c.af = float(T(ca)); c.bf = float(T(cb)); c.ad = double(T(ca)); c.bd = double(T(cb));
    return c;
  };
  // One launch per level and direction (smooth.cu): FP32, Q1, the default cell loop.
  // FP64 stays on the sweeps (its time is the FP64 rate, and the tiles' halo cells
  // would add to it); a forced strip height asks for the sweeps.
  const bool tiles = sizeof(T) == 4 && M.k == 1 && fuse && pb.sweep_sh == 0 && mg.degree == 3;
  if (tiles) {
    VC(mg_level_defects<T>(D.n_lev_bricks, D.lev_bricks, D.home_leaf, nc, nsleaf, r, d, rr, pb.cmask, B.fixbits, s));
    VC(note_node(mg, b, 0, 9, 4, -1, s));
  } else {
    VC(cudaMemsetAsync(d, 0, nc * N * sizeof(T), s));
    VC(cudaMemsetAsync(x, 0, nc * N * sizeof(T), s));
    VC(mg_copy_in<T>(nsleaf, nc, D.home, r, d, pb.cmask, B.fixbits, s));
    VC(note_node(mg, b, 0, 7, 3, -1, s));
  }
  // Chebyshev on level l over [a, bb], `degree` applications of D^-1: solve A v = rhs
  // from v = 0 into out (buffers yp, y, t).  The three iterates (current,
  // previous, next) rotate roles each step; the start is chosen so that the last
  // step writes `out`.
  auto cheb_bufs = [&](int64_t o, T* out, int degree, T*& cur, T*& prev, T*& nxt) {
    T* w0 = out;
    T* w1 = yp + o;
    T* w2 = y + o;
    switch ((degree - 1) % 3) {   // each step maps (cur, prev, nxt) to (nxt, cur, prev)
      case 0: cur = w0; prev = w1; nxt = w2; break;
      case 1: cur = w1; prev = w2; nxt = w0; break;
      default: cur = w1; prev = w0; nxt = w2; break;
    }
  };
  // first_done: the first iterate was formed with the level's defect (mg_restrict)
  auto cheb_ab = [&](int l, const T* rhs, T* out, double a, double bb, int degree, bool first_done) -> cudaError_t {
    const DevLevel& lv = D.levels[l].lv;
    const int64_t n = nc * int64_t(lv.n_slots), o = nc * lv.off;
    if (!(bb > 0) || degree < 1) return cudaMemsetAsync(out, 0, n * sizeof(T), s);
    const double theta = 0.5 * (bb + a), delta = 0.5 * (bb - a), sigma = theta / delta;
    T *cur, *prev, *nxt;
    cheb_bufs(o, out, degree, cur, prev, nxt);
    cudaError_t ee = first_done ? cudaSuccess
                                : mg_chebyshev_first<T>(n, cur, prev, dinv + o, rhs, T(1.0 / theta), s, true);
    if (ee != cudaSuccess) return ee;
    double rho = 1.0 / sigma;
    for (int j = 1; j < degree; ++j) {
      const double rho_n = 1.0 / (2.0 * sigma - rho);
      // next = cur + rho_n rho (cur - prev) + 2 rho_n / delta D^-1 (rhs - A cur)
      if (fuse) {
        const ChebEpi c = epi(CHEB_STEP, prev, dinv + o, rhs, nxt, nullptr, nullptr, rho_n * rho, 2.0 * rho_n / delta);
        ee = level_apply<T>(mg, l, block_op(b), cur, t + o, s, true, &c);
      } else {
        ee = level_apply<T>(mg, l, block_op(b), cur, t + o, s, true);
        if (ee == cudaSuccess)
          ee = mg_chebyshev_step<T>(n, nxt, cur, prev, dinv + o, rhs, t + o, T(rho_n * rho), T(2.0 * rho_n / delta),
                                    s, true);
      }
      if (ee != cudaSuccess) return ee;
      T* old_prev = prev;
      prev = cur;
      cur = nxt;
      nxt = old_prev;
      rho = rho_n;
    }
    return cudaSuccess;
  };
  if constexpr (sizeof(T) == 4) {
    if (tiles) {
      auto args = [&](int l) {
        const DevLevel& lv = D.levels[l].lv;
        const DevLevel& lc = D.levels[l - 1].lv;
        const int64_t o = nc * lv.off, oc = nc * lc.off;
        ApplyArgs k;
        std::memset(&k, 0, sizeof(k));
        for (int q = 0; q <= M.Lf && q < kMaxLevels; ++q) { k.hx[q] = M.tree.hx(q); k.hy[q] = M.tree.hy(q); }
        fill_material(pb.prm, k, pb.has_ecell);
        fill_cell_constants(k, M.Lf + 1);
        SmoothArgs a;
        std::memset(&a, 0, sizeof(a));
        a.tiles = lv.tiles; a.ntiles = lv.ntiles; a.tile = lv.tile;
        a.n = lv.n_slots; a.nc = lc.n_slots;
        a.flags = lv.flags; a.cmask = mg.cmask + lv.off; a.cmask_c = mg.cmask + lc.off;
        a.lin = mg.lin32 + 4 * lv.off;
        a.ecell = pb.has_ecell ? pb.lev_ecell32 + lv.off : nullptr;
        a.dinv = dinv + o; a.d = d + o; a.dc = d + oc;
        a.m = k.mf; a.g = k.gf[l];
        const double lam = B.lam[l];
        if (lam > 0) {
          const double lo = mg.lo * lam, hi = mg.hi * lam;
          const double theta = 0.5 * (hi + lo), delta = 0.5 * (hi - lo), sigma = theta / delta;
          const double r0 = 1.0 / sigma, r1 = 1.0 / (2.0 * sigma - r0), r2 = 1.0 / (2.0 * sigma - r1);
          a.c0 = float(1.0 / theta);
          a.a1 = float(r1 * r0); a.b1 = float(2.0 * r1 / delta);
          a.a2 = float(r2 * r1); a.b2 = float(2.0 * r2 / delta);
        }
        return a;
      };
      for (int l = nl - 1; l >= 1; --l) {
        SmoothArgs a = args(l);
        a.xout = x + nc * D.levels[l].lv.off;
        VC(launch_smooth_down(a, block_op(b), s));
      }
      if (mg.coarse_mode == 1) VC(cheb_ab(0, d, rr, B.c0_a, B.c0_b, B.c0_deg, false));
      else VC(mg_coarse<T>(B.n_coarse, B.coarse_idx, B.coarse_inv, d, rr, s, true));
      for (int l = 1; l < nl; ++l) {
        SmoothArgs a = args(l);
        a.x = x + nc * D.levels[l].lv.off;
        a.xc = rr + nc * D.levels[l - 1].lv.off;
        a.xout = rr + nc * D.levels[l].lv.off;
        // the first one is dependent in this way only behind k_coarse_matvec: without a
        // coarse launch down(1) itself precedes it, and the Chebyshev coarse solver's
        // kernels let it start before they wait
        VC(launch_smooth_up(a, block_op(b), s, l > 1 || (mg.coarse_mode == 0 && B.n_coarse > 0)));
      }
      VC(mg_copy_out<T>(nsleaf, nc, D.home, rr, r, z, pb.cmask, pb.mesh->dev.slot_flags, B.fixbits, s, true));
      return note_node(mg, b, 1, 9, 4, 5, s);
    }
  }
  // smoothing on level l >= 1: degree mg.degree on [lo, hi] * lambda_max
  auto smooths = [&](int l) { return l >= 1 && B.lam[l] > 0 && mg.degree >= 1; };
  auto cheb = [&](int l, const T* rhs, T* out, bool first_done) -> cudaError_t {
    const double lam = B.lam[l];
    return cheb_ab(l, rhs, out, mg.lo * lam, mg.hi * lam, lam > 0 ? mg.degree : 0, first_done);
  };
  // down sweep; with the fused smoother the restriction also forms the coarser
  // level's first Chebyshev iterate
  bool first_done = false;
  for (int l = nl - 1; l >= 1; --l) {
    const DevLevel& lv = D.levels[l].lv;
    const DevLevel& lc = D.levels[l - 1].lv;
    const int64_t o = nc * lv.off, oc = nc * lc.off;
    VC(cheb(l, d + o, x + o, first_done));
    VC(level_apply<T>(mg, l, block_op(b), x + o, t + o, s, true));
    first_done = fuse && smooths(l - 1);
    if (first_done) {
      const double lam = B.lam[l - 1], theta = 0.5 * (mg.lo * lam + mg.hi * lam);
      T *cur, *prev, *nxt;
      cheb_bufs(oc, x + oc, mg.degree, cur, prev, nxt);
      VC(mg_restrict<T>(lc.n_slots, nc, lc.n_slots, lv.n_slots, lv.R_ptr, lv.R_col, lv.R_val, d + o, t + o, d + oc,
                        mg.cmask + lc.off, B.fixbits, s, true, dinv + oc, cur, prev, T(1.0 / theta)));
    } else {
      VC(mg_restrict<T>(lc.n_slots, nc, lc.n_slots, lv.n_slots, lv.R_ptr, lv.R_col, lv.R_val, d + o, t + o, d + oc,
                        mg.cmask + lc.off, B.fixbits, s, true));
    }
  }
  // coarse
  if (mg.coarse_mode == 1) VC(cheb_ab(0, d, x, B.c0_a, B.c0_b, B.c0_deg, false));
  else VC(mg_coarse<T>(B.n_coarse, B.coarse_idx, B.coarse_inv, d, x, s, true));
  // Post-smoothing on level l of the defect d - A x, from zero, added to x: the
  // first step applies A to x and forms the defect, the last adds instead of
  // storing.  The level defect d is free once the first step has read it.
  auto cheb_post = [&](int l) -> cudaError_t {
    const DevLevel& lv = D.levels[l].lv;
    const int64_t n = nc * int64_t(lv.n_slots), o = nc * lv.off;
    const double lam = B.lam[l];
    const int degree = mg.degree;
    if (!(lam > 0) || degree < 1) return cudaSuccess;   // a zero correction
    const double a = mg.lo * lam, bb = mg.hi * lam;
    const double theta = 0.5 * (bb + a), delta = 0.5 * (bb - a), sigma = theta / delta;
    cudaError_t ee;
    if (degree == 1) {
      // x += c0 D^-1 (d - A x) reads and writes x: never fused
      ee = level_apply<T>(mg, l, block_op(b), x + o, t + o, s, true);
      if (ee != cudaSuccess) return ee;
      return mg_chebyshev_first_res<T>(n, nullptr, nullptr, nullptr, dinv + o, d + o, t + o, T(1.0 / theta), x + o, s,
                                       true);
    }
    T* cur = yp + o;
    T* prev = y + o;
    T* nxt = d + o;
    if (fuse) {
      const ChebEpi c = epi(CHEB_FIRST_RES, nullptr, dinv + o, d + o, cur, rr + o, prev, 1.0 / theta, 0.0);
      ee = level_apply<T>(mg, l, block_op(b), x + o, t + o, s, true, &c);
    } else {
      ee = level_apply<T>(mg, l, block_op(b), x + o, t + o, s, true);
      if (ee == cudaSuccess)
        ee = mg_chebyshev_first_res<T>(n, cur, prev, rr + o, dinv + o, d + o, t + o, T(1.0 / theta), nullptr, s,
                                       true);
    }
    if (ee != cudaSuccess) return ee;
    double rho = 1.0 / sigma;
    for (int j = 1; j < degree; ++j) {
      const double rho_n = 1.0 / (2.0 * sigma - rho);
      const bool last = j == degree - 1;
      if (fuse) {
        const ChebEpi c = epi(last ? CHEB_STEP_ADD : CHEB_STEP, prev, dinv + o, rr + o, last ? x + o : nxt, nullptr,
                              nullptr, rho_n * rho, 2.0 * rho_n / delta);
        ee = level_apply<T>(mg, l, block_op(b), cur, t + o, s, true, &c);
        if (ee != cudaSuccess || last) return ee;
      } else {
        ee = level_apply<T>(mg, l, block_op(b), cur, t + o, s, true);
        if (ee != cudaSuccess) return ee;
        if (last)
          return mg_chebyshev_step_add<T>(n, x + o, cur, prev, dinv + o, rr + o, t + o, T(rho_n * rho),
                                          T(2.0 * rho_n / delta), s, true);
        ee = mg_chebyshev_step<T>(n, nxt, cur, prev, dinv + o, rr + o, t + o, T(rho_n * rho), T(2.0 * rho_n / delta),
                                  s, true);
        if (ee != cudaSuccess) return ee;
      }
      T* old_prev = prev;
      prev = cur;
      cur = nxt;
      nxt = old_prev;
      rho = rho_n;
    }
    return cudaSuccess;
  };
  // up sweep
  for (int l = 1; l < nl; ++l) {
    const DevLevel& lv = D.levels[l].lv;
    const DevLevel& lc = D.levels[l - 1].lv;
    const int64_t o = nc * lv.off;
    VC(mg_prolong<T>(lv.n_slots, nc, lv.n_slots, lc.n_slots, lv.P_ptr, lv.P_col, lv.P_val, x + nc * lc.off, x + o,
                     mg.cmask + lv.off, B.fixbits, s, true));
    VC(cheb_post(l));
  }
  VC(mg_copy_out<T>(nsleaf, nc, D.home, x, r, z, pb.cmask, pb.mesh->dev.slot_flags, B.fixbits, s, true));
  VC(note_node(mg, b, 1, 9, 4, 5, s));
#undef VC
  return cudaSuccess;
}

}  // namespace

static cudaError_t vcycle_direct(pff_mg& mg, int block, const double* r, double* z, cudaStream_t s) {
  if (mg.precision == PFF_F64) return vcycle_t<double>(mg, block, r, z, s);
  return vcycle_t<float>(mg, block, r, z, s);
}

// Capture graph g: block g, or both for g = 2.  The blocks share no buffer (each has
// its own level vectors, inverse diagonals and coarse data; the staging vectors are
// split at 2 n_slots), so the phi block runs on a second branch forked from and joined
// back into the capture stream.  False if the graph could not be made (the direct path
// is used).
static bool vcycle_capture(pff_mg& mg, int g) {
  const int64_t n = mg.pb->mesh->m.lay.n_slots;
  if (!mg.cap_stream && cudaStreamCreateWithFlags(&mg.cap_stream, cudaStreamNonBlocking) != cudaSuccess) return false;
  if (!mg.cap_stream2 && cudaStreamCreateWithFlags(&mg.cap_stream2, cudaStreamNonBlocking) != cudaSuccess) return false;
  if (!mg.ev_fork && cudaEventCreateWithFlags(&mg.ev_fork, cudaEventDisableTiming) != cudaSuccess) return false;
  if (!mg.ev_join && cudaEventCreateWithFlags(&mg.ev_join, cudaEventDisableTiming) != cudaSuccess) return false;
  if (cudaStreamBeginCapture(mg.cap_stream, cudaStreamCaptureModeThreadLocal) != cudaSuccess) return false;
  for (int b = 0; b < 2; ++b) {
    mg.vc_io[g][b] = pff_mg::VcIo();
    mg.vc_note[b] = &mg.vc_io[g][b];
  }
  cudaError_t e = cudaSuccess;
  if (g < 2) {
    const int64_t off = g == 0 ? 0 : 2 * n;
    e = vcycle_direct(mg, g, mg.vc_in + off, mg.vc_out + off, mg.cap_stream);
  } else {
    e = cudaEventRecord(mg.ev_fork, mg.cap_stream);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(mg.cap_stream2, mg.ev_fork, 0);
    if (e == cudaSuccess) e = vcycle_direct(mg, 1, mg.vc_in + 2 * n, mg.vc_out + 2 * n, mg.cap_stream2);
    if (e == cudaSuccess) e = vcycle_direct(mg, 0, mg.vc_in, mg.vc_out, mg.cap_stream);
    if (e == cudaSuccess) e = cudaEventRecord(mg.ev_join, mg.cap_stream2);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(mg.cap_stream, mg.ev_join, 0);
  }
  mg.vc_note[0] = mg.vc_note[1] = nullptr;
  cudaGraph_t gr = nullptr;
  const cudaError_t e2 = cudaStreamEndCapture(mg.cap_stream, &gr);
  bool ok = e == cudaSuccess && e2 == cudaSuccess && gr != nullptr;
  for (int b = 0; b < 2 && ok; ++b) {
    if (g < 2 && b != g) continue;
    pff_mg::VcIo& io = mg.vc_io[g][b];
    for (int w = 0; w < 2 && ok; ++w) {
      ok = io.node[w] && cudaGraphKernelNodeGetParams(io.node[w], &io.prm[w]) == cudaSuccess;
      if (ok) std::copy_n(io.prm[w].kernelParams, io.arg[w].size(), io.arg[w].begin());
    }
  }
  if (ok) ok = cudaGraphInstantiate(&mg.vc_exec[g], gr, 0) == cudaSuccess;
  if (!ok) {
    if (gr) cudaGraphDestroy(gr);
    mg.vc_exec[g] = nullptr;
    cudaGetLastError();   // clear a capture error; the direct path follows
    return false;
  }
  mg.vc_graph[g] = gr;
  return true;
}

// r and z of block b in graph g's next launch
static cudaError_t vcycle_bind(pff_mg& mg, int g, int b, const double* r, double* z) {
  pff_mg::VcIo& io = mg.vc_io[g][b];
  for (int w = 0; w < 2; ++w) {
    io.arg[w][io.r_arg[w]] = &r;
    if (w == 1) io.arg[w][io.z_arg] = &z;
    io.prm[w].kernelParams = io.arg[w].data();
    const cudaError_t e = cudaGraphExecKernelNodeSetParams(mg.vc_exec[g], io.node[w], &io.prm[w]);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

// One replay of graph g; blocks of the call: b0 .. b1
static cudaError_t vcycle_replay(pff_mg& mg, int g, const double* r, double* z, cudaStream_t s) {
  const int64_t n = mg.pb->mesh->m.lay.n_slots;
  const int b0 = g == 2 ? 0 : g, b1 = g == 2 ? 1 : g;
  const int64_t off = b0 == 0 ? 0 : 2 * n, len = (b0 == 0 ? 2 * n : 0) + (b1 == 1 ? n : 0);
  // the last kernel reads r on fixed rows while it writes z: vectors that share memory go
  // through the staging vectors
  const uintptr_t ra = reinterpret_cast<uintptr_t>(r), za = reinterpret_cast<uintptr_t>(z);
  const uintptr_t span = uintptr_t(len) * sizeof(double);
  cudaError_t e = cudaSuccess;
  if (ra < za + span && za < ra + span) {
    const size_t bytes = size_t(len) * sizeof(double);
    for (int b = b0; b <= b1 && e == cudaSuccess; ++b)
      e = vcycle_bind(mg, g, b, mg.vc_in + (b == 0 ? 0 : 2 * n), mg.vc_out + (b == 0 ? 0 : 2 * n));
    if (e == cudaSuccess) e = cudaMemcpyAsync(mg.vc_in + off, r, bytes, cudaMemcpyDeviceToDevice, s);
    if (e == cudaSuccess) e = cudaGraphLaunch(mg.vc_exec[g], s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(z, mg.vc_out + off, bytes, cudaMemcpyDeviceToDevice, s);
    return e;
  }
  for (int b = b0; b <= b1 && e == cudaSuccess; ++b)
    e = vcycle_bind(mg, g, b, r + (b == b0 ? 0 : 2 * n), z + (b == b0 ? 0 : 2 * n));
  return e == cudaSuccess ? cudaGraphLaunch(mg.vc_exec[g], s) : e;
}

cudaError_t mg_vcycle(pff_mg& mg, int block, const double* r, double* z, cudaStream_t s) {
  if (mg.graphs_ok && mg.vc_in && mg.vc_out) {
    if (!mg.vc_exec[block] && !vcycle_capture(mg, block)) mg.graphs_ok = false;
    if (mg.vc_exec[block]) return vcycle_replay(mg, block, r, z, s);
  }
  return vcycle_direct(mg, block, r, z, s);
}

cudaError_t mg_precond(pff_mg& mg, const double* v, double* z, cudaStream_t s) {
  const int64_t n = mg.pb->mesh->m.lay.n_slots;
  if (mg.graphs_ok && mg.vc_in && mg.vc_out) {
    if (!mg.vc_exec[2] && !vcycle_capture(mg, 2)) mg.graphs_ok = false;
    if (mg.vc_exec[2]) return vcycle_replay(mg, 2, v, z, s);
  }
  cudaError_t e = vcycle_direct(mg, 0, v, z, s);
  if (e == cudaSuccess) e = vcycle_direct(mg, 1, v + 2 * n, z + 2 * n, s);
  return e;
}

template cudaError_t level_apply<float>(pff_mg&, int, int, const float*, float*, cudaStream_t, bool, const ChebEpi*);
template cudaError_t level_apply<double>(pff_mg&, int, int, const double*, double*, cudaStream_t, bool,
                                         const ChebEpi*);

}  // namespace pff
