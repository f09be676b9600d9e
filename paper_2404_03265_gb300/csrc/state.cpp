// Device uploads and operator dispatch behind the C-ABI.
#include "state.h"

#include <algorithm>
#include <cstring>
#include <unordered_map>

namespace pff {

static DevLayout upload_layout(DevAllocs& mem, const Layout& L) {
  DevLayout d;
  d.bricks = mem.upload(L.bricks);
  d.nbricks = int32_t(L.bricks.size());
  d.win = mem.upload(L.win);
  d.own_part = mem.upload(L.own_part);
  d.own_act = mem.upload(L.own_act);
  std::vector<int32_t> own(L.own_part.size());
  for (size_t i = 0; i < own.size(); ++i)
    own[i] = int32_t(uint32_t(L.own_part[i] + 1) | (uint32_t(L.own_act[i]) << 30));
  d.own = mem.upload(own);
  const std::vector<int32_t> units = sweep_units(L.bricks, d.unit_off);
  d.units = mem.upload(units);
  d.cellmask = mem.upload(L.cellmask);
  return d;
}

cudaError_t after_clears(cudaStream_t s) {
  if (s == nullptr || s == cudaStreamLegacy) return cudaSuccess;
  cudaEvent_t ev = nullptr;
  cudaError_t e = cudaEventCreateWithFlags(&ev, cudaEventDisableTiming);
  if (e == cudaSuccess) e = cudaEventRecord(ev, cudaStreamLegacy);
  if (e == cudaSuccess) e = cudaStreamWaitEvent(s, ev, 0);
  if (ev) cudaEventDestroy(ev);   // released when it has completed
  return e;
}

// Tiles of the fused smoothers: every tn x tn part of a brick of level mesh lm that
// holds a node, with the storage bases around the brick and around its parent brick (bx / 2,
// by / 2) of the next coarser level.
static std::vector<SmoothTile> smooth_tiles(const LevelMesh& lm, const LevelMesh& coarse, int tn) {
  const int NB = lm.lay.NB;
  std::unordered_map<uint64_t, int32_t> parent;
  for (size_t b = 0; b < coarse.lay.bricks.size(); ++b)
    parent[cell_key(coarse.lay.bricks[b].bx, coarse.lay.bricks[b].by)] = int32_t(b);
  std::vector<SmoothTile> out;
  for (size_t b = 0; b < lm.lay.bricks.size(); ++b) {
    const BrickDesc& d = lm.lay.bricks[b];
    const auto it = parent.find(cell_key(d.bx >> 1, d.by >> 1));
    const int side = NB / tn;
    for (int q = 0; q < side * side; ++q) {
      const int x0 = tn * (q % side), y0 = tn * (q / side);
      bool any = false;
      for (int j = y0; j < y0 + tn && !any; ++j)
        for (int i = x0; i < x0 + tn && !any; ++i)
          any = lm.slot_X[b * size_t(NB) * NB + i + size_t(NB) * j] >= 0;
      if (!any) continue;
      SmoothTile t;
      for (int e = 0; e < 9; ++e) {
        t.fb[e] = d.nbr_base[e];
        t.cb[e] = it == parent.end() ? -1 : coarse.lay.bricks[it->second].nbr_base[e];
      }
      t.pos = q % side | (q / side) << 3 | (d.bx & 1) << 6 | (d.by & 1) << 7;
      t.pad = 0;
      out.push_back(t);
    }
  }
  return out;
}

// Tables of the two-pass leaf operators
static LeafCells upload_leaf_cells(DevAllocs& mem, const Mesh& M) {
  constexpr int NB = 30;
  constexpr size_t SLOTS = size_t(NB) * NB;
  const size_t ns = size_t(M.lay.n_slots), nb = M.lay.bricks.size();
  const int k = M.k, W = M.lay.W;
  // cells in the order of their slots (brick by brick, and so level by level), each
  // level filled up to an even number with a repeated cell that no node refers to
  std::vector<int32_t> at(ns, -1), in_brick(nb, 0);
  for (int32_t s : M.cell_slot) {
    at[s] = 0;
    ++in_brick[size_t(s) / SLOTS];
  }
  size_t nc = 0;
  for (size_t b = 0; b < nb; ++b) {
    nc += size_t(in_brick[b]);
    if (b + 1 == nb || M.lay.bricks[b + 1].level != M.lay.bricks[b].level) nc += nc % 2;
  }
  std::vector<int4> corner(k == 1 ? nc : 0), node(ns, make_int4(-1, -1, -1, -1)), part(size_t(M.n_partials));
  std::vector<int32_t> nodes9(k == 2 ? 9 * nc : 0), slot(nc);
  std::vector<uint8_t> level(nc), part_pos(size_t(M.n_partials), 0);
  size_t q = 0;
  for (size_t b = 0; b < nb; ++b) {
    const BrickDesc& d = M.lay.bricks[b];
    const int32_t* win = d.irr >= 0 ? M.lay.win.data() + size_t(d.irr) * W * W : nullptr;
    // node at brick position (i, j), 0..NB
    auto code = [&](int i, int j) -> int32_t {
      if (win) return win[(i + k) + size_t(W) * (j + k)];
      return d.nbr_base[(j < NB ? 3 : 6) + (i < NB ? 1 : 2)] + (i < NB ? i : i - NB) + NB * (j < NB ? j : j - NB);
    };
    for (int r = 0; in_brick[b] && r < NB; ++r)
      for (int n = 0; n < NB; ++n) {
        const size_t s = b * SLOTS + size_t(n + NB * r);
        if (at[s] < 0) continue;
        at[s] = int32_t(q);
        slot[q] = int32_t(s);
        level[q] = uint8_t(d.level);
        if (k == 1) corner[q] = make_int4(code(n, r), code(n + 1, r), code(n, r + 1), code(n + 1, r + 1));
        else
          for (int e = 0; e < 9; ++e) nodes9[size_t(e) * nc + q] = code(n + e % 3, r + e / 3);
        ++q;
      }
    if (q % 2 && (b + 1 == nb || M.lay.bricks[b + 1].level != d.level)) {
      slot[q] = slot[q - 1];
      level[q] = level[q - 1];
      if (k == 1) corner[q] = corner[q - 1];
      else
        for (int e = 0; e < 9; ++e) nodes9[size_t(e) * nc + q] = nodes9[size_t(e) * nc + q - 1];
      ++q;
    }
  }
  for (size_t b = 0; b < nb; ++b) {
    const BrickDesc& d = M.lay.bricks[b];
    auto cell_at = [&](int n, int r) -> int32_t {   // the leaf cell of this level with lower-left node (n, r) >= -k
      const int32_t base = d.nbr_base[(r < 0 ? 0 : 3) + (n < 0 ? 0 : 1)];
      return base < 0 ? -1 : at[size_t(base) + size_t((n < 0 ? n + NB : n) + NB * (r < 0 ? r + NB : r))];
    };
    for (int r = 0; r < NB; ++r)
      for (int n = 0; n < NB; ++n) {
        const size_t o = size_t(n + NB * r), s = b * SLOTS + o;
        const int px = n & (k - 1), py = r & (k - 1), n0 = n - px, r0 = r - py;   // inside a Q2 cell: no left (lower) neighbour
        const int4 q = make_int4(cell_at(n0, r0), px ? -1 : cell_at(n0 - k, r0), py ? -1 : cell_at(n0, r0 - k),
                                 px || py ? -1 : cell_at(n0 - k, r0 - k));
        const int32_t p = d.irr >= 0 ? M.lay.own_part[size_t(d.irr) * SLOTS + o] : -1;
        if (p >= 0) {
          part[p] = q;
          part_pos[p] = uint8_t(px | py << 1);
        }
        if (M.slot_node[s] >= 0) node[s] = q;
      }
  }
  for (size_t i = 0; i < M.fix_slot.size(); ++i) node[M.fix_slot[i]] = make_int4(-2 - int32_t(i), -1, -1, -1);
  LeafCells L;
  L.ncells = int32_t(nc);
  if (k == 1) {
    L.corner = mem.upload(corner);
  } else {
    L.nodes9 = mem.upload(nodes9);
    L.part_pos = mem.upload(part_pos);
  }
  L.level = mem.upload(level);
  L.slot = mem.upload(slot);
  L.node = mem.upload(node);
  L.part = mem.upload(part);
  return L;
}

// A leaf operator and its fix-up: Q1 in two passes over the cell and node lists where
// that is the faster path (leaf_cells.cu), else the cell loop and the fix-up kernel.
//  - FP64: two passes (bound by the FP64 rate, and they evaluate only cells that exist):
//    Jacobian 971 -> 724 us on 4.1M DoFs, 647 -> 200 us on the 1.04M-DoF crack mesh, 44 ->
//    20 us on 4.3k DoFs.  A forced strip height asks for the sweep's Jacobian.
//    The mass, which reads nothing and does next to no arithmetic, stays with the sweep:
//    28 against 56 us on 4.1M DoFs, 22.6 against 20.6 on the crack mesh, 9.4 against 9.1 on
//    4.3k.
//  - FP32: two passes while the contributions (48 bytes per cell, written and read again)
//    cost less than the sweep's cells that do not exist and its few long units.  Both loops
//    (us; input vectors in L2, and rotating through more than L2), sweep against passes:
//      86k cells, 0.76 of the slots   12.1 / 12.3 against 12.3 / 13.9
//      340k, 0.46 (crack mesh)        28.5 / 29.3 against 19.6 / 24.6
//      401k, 0.77                     22.5 / 23.2 against 18.9 / 23.6
//      433k, 0.85                     21.2 / 22.5 against 18.8 / 24.6
//      507k, 0.54                     37.0 / 38.9 against 26.8 / 31.0
//      534k, 0.89                     22.1 / 22.5 against 23.0 / 27.5
//      619k, 0.82                     27.6 / 28.9 against 31.9 / 36.1
//      648k, 0.72                     29.9 / 30.7 against 35.6 / 38.0
//    So up to 450k cells, and up to 550k where bricks are less than 0.6 full.
// Without a buffer of contributions (see below) the Jacobian takes the cell loop.
static bool two_passes_f32(int64_t cells, int64_t slots) {
  return cells <= 450000 || (cells <= 550000 && 10 * cells < 6 * slots);
}

// Who may use the contributions.  On a mesh without refinement edges the cell loop writes
// nothing but the result, and applies of one problem (pff_apply) may run at the same time
// on several streams and from several threads.  The two passes keep that: FP64 applies take
// a buffer of their stream, both passes launched under one lock; the cell loop serves a
// stream beyond the fourth, a capture (its graph may run beside any stream) and memory
// that is out.  FP32 stays with the cell loop there, which is the faster one: 8.6 against
// 12.2 us on 198k DoFs.  FP64: 217 -> 143 us on 0.79M DoFs, 884 -> 550 us on 3.2M.
// On other meshes applies of one precision share partial sums and hanging inputs anyway,
// and the contributions have a buffer per precision as those have.  The operators inside a
// solver call share the solver's workspace and always use the FP64 buffer of the problem.
static bool refinement_edges(const DevMesh& D) { return D.nhang > 0 || D.nfix > 0; }

// Contributions of the FP64 operators: with the problem while they are small, larger ones
// (FP32 applies never read them: 131 MB on 4.1M Q1 DoFs) on first use.
constexpr size_t kCellsWithProblem = size_t(64) << 20;
static size_t cell_values(const pff_problem& pb) {
  return (pb.mesh->m.k == 1 ? 12 : 27) * size_t(pb.mesh->dev.cells.ncells);
}

// nullptr when memory is out (the Jacobian then takes the cell loop)
static double* alloc_cells64(const pff_problem& pb) {
  // a stream of the caller may be capturing, and this memory is no part of its graph
  cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
  cudaThreadExchangeStreamCaptureMode(&mode);
  void* p = nullptr;
  const cudaError_t e = cudaMalloc(&p, std::max<size_t>(cell_values(pb), 1) * sizeof(double));
  cudaThreadExchangeStreamCaptureMode(&mode);
  if (e == cudaSuccess) return static_cast<double*>(p);
  cudaGetLastError();
  return nullptr;
}

double* leaf_contributions64(pff_problem& pb) {
  std::lock_guard<std::mutex> lk(pb.cells_mu);
  if (!pb.cells64) pb.cells64 = pb.cells64_late = alloc_cells64(pb);
  return pb.cells64;
}

// The buffer of stream s; the caller holds cells_mu until both passes are launched
static double* stream_contributions(pff_problem& pb, cudaStream_t s) {
  cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
  unsigned long long id = 0;
  if (cudaStreamIsCapturing(s, &st) != cudaSuccess || st != cudaStreamCaptureStatusNone ||
      cudaStreamGetId(s, &id) != cudaSuccess) {
    cudaGetLastError();
    return nullptr;
  }
  for (auto& c : pb.stream_cells) {
    if (!c.values) {
      c.values = alloc_cells64(pb);
      c.stream = id;
    }
    if (c.stream == id) return c.values;
  }
  return nullptr;
}

static bool use_two_passes(const ApplyArgs& a, int op, bool f64) {
  if (op == OP_VJP || op == OP_MASS || a.lc.out == nullptr) return false;
  const bool jacobian = op == OP_FULL || op == OP_FULL_T;
  if (a.fe_degree == 2) return f64 && (jacobian || op == OP_RESID);
  if (a.sweep_sh != 0 && jacobian) return false;
  return f64 || (jacobian && two_passes_f32(a.lc.ncells, a.n_slots));
}

template <typename T>
cudaError_t launch_leaf(const ApplyArgs& a, const FixupArgs& f, int op, cudaStream_t s) {
  if (use_two_passes(a, op, sizeof(T) == 8))
    return a.fe_degree == 1 ? launch_leaf_cells<T>(a, f, op, s) : launch_leaf_cells_q2(a, f, op, s);
  const cudaError_t e = launch_apply<T>(a, op, s);
  if (e != cudaSuccess || op == OP_VJP) return e;   // OP_VJP: per-cell outputs only
  return launch_fixup<T>(f, s);
}
template cudaError_t launch_leaf<float>(const ApplyArgs&, const FixupArgs&, int, cudaStream_t);
template cudaError_t launch_leaf<double>(const ApplyArgs&, const FixupArgs&, int, cudaStream_t);

std::string upload_mesh(pff_mesh& pm) {
  DevMesh& D = pm.dev;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return std::string("cudaGetDevice: ") + cudaGetErrorString(e);
  if (D.uploaded) {
    if (D.device != dev) return "mesh tables live on another device";
    return "";
  }
  const Mesh& M = pm.m;
  D.leaf = upload_layout(D.mem, M.lay);
  D.cells = upload_leaf_cells(D.mem, M);
  std::vector<DevHanging> hh(M.hang.size());
  for (size_t h = 0; h < M.hang.size(); ++h) {
    hh[h].slot = M.hang[h].slot;
    for (int b = 0; b < 3; ++b) {
      hh[h].parent[b] = M.hang[h].parent[b];
      hh[h].weight[b] = M.hang[h].weight[b];
    }
  }
  D.hang = D.mem.upload(hh);
  D.nhang = int32_t(hh.size());
  D.nfix = int32_t(M.fix_slot.size());
  D.fix_slot = D.mem.upload(M.fix_slot);
  D.fix_ptr = D.mem.upload(M.fix_ptr);
  D.fix_part = D.mem.upload(M.fix_part);
  D.fix_w = D.mem.upload(M.fix_w);
  D.slot_flags = D.mem.upload(M.slot_flags);
  D.n_leaf_cells = int32_t(M.cell_slot.size());
  D.cell_slot = D.mem.upload(M.cell_slot);
  D.levels.resize(M.levels.size());
  int64_t off = 0;
  for (size_t l = 0; l < M.levels.size(); ++l) {
    const LevelMesh& lm = M.levels[l];
    DevMesh::Level& L = D.levels[l];
    L.lay = upload_layout(D.mem, lm.lay);
    L.lv.n_slots = int32_t(lm.lay.n_slots);
    L.lv.off = off;
    off += lm.lay.n_slots;
    if (M.k == 1 && l > 0) {
      std::vector<SmoothTile> tiles;
      // Small levels take small tiles (a shorter chain per block) as long as the tiles are
      // few per SM: up to 2 of side 6, 4 of side 10; large ones side 15, which repeats the
      // least work.  u-block V-cycles (us) on 4.3k, 65k, 0.26M-DoF box and 1.04M-DoF crack
      // meshes: 32.8, 46.5, 69.6, 129.0; with 1 and 2 per SM 32.8, 46.7, 67.7, 128.1; with 4
      // and 8 32.8, 45.1, 69.6, 129.6 (a 1M-DoF box 94.3, 94.3, 98.2); side 15 alone 36.9,
      // 51.2, 69.9, 130.7.
      for (int tn : {6, 10, 15}) {
        const int64_t most = int64_t(tn == 6 ? 2 : 4) * sm_count();
        if (tn < 15 && lm.n_nodes > most * tn * tn) continue;   // more tiles than that
        tiles = smooth_tiles(lm, M.levels[l - 1], tn);
        L.lv.tile = tn;
        if (int64_t(tiles.size()) <= most) break;
      }
      L.lv.tiles = D.mem.upload(tiles);
      L.lv.ntiles = int32_t(tiles.size());
    }
    std::vector<float> pv(lm.P_val.begin(), lm.P_val.end()), rv(lm.R_val.begin(), lm.R_val.end());
    if (l > 0) {
      L.lv.P_ptr = D.mem.upload(lm.P_ptr);
      L.lv.P_col = D.mem.upload(lm.P_col);
      L.lv.P_val = D.mem.upload(pv);
      L.lv.R_ptr = D.mem.upload(lm.R_ptr);
      L.lv.R_col = D.mem.upload(lm.R_col);
      L.lv.R_val = D.mem.upload(rv);
    }
    L.n_cells = int32_t(lm.cell_dst.size());
    L.cell_dst = D.mem.upload(lm.cell_dst);
    L.cell_src = D.mem.upload(lm.cell_src);
    L.cell_child = D.mem.upload(lm.cell_child);
  }
  D.lev_total = off;
  {
    std::vector<LevBrick> lb;
    std::vector<int32_t> home(size_t(off), -1), leaf(static_cast<size_t>(off)), gx(static_cast<size_t>(off)),
        gy(static_cast<size_t>(off));
    std::vector<uint8_t> flags(static_cast<size_t>(off));
    std::vector<SmoothTile> tiles;
    for (size_t l = 0; l < M.levels.size(); ++l) {
      const LevelMesh& lm = M.levels[l];
      const DevLevel& lv = D.levels[l].lv;
      for (size_t b = 0; b < lm.lay.bricks.size(); ++b)
        lb.push_back({int32_t(lv.off), lv.n_slots, int32_t(b) * lm.lay.NB * lm.lay.NB});
      std::copy(lm.slot_leaf.begin(), lm.slot_leaf.end(), leaf.begin() + lv.off);
      std::copy(lm.slot_flags.begin(), lm.slot_flags.end(), flags.begin() + lv.off);
      const int shift = M.Lf - int(l);
      for (size_t q = 0; q < lm.slot_X.size(); ++q) {   // (a hole's -1 stays -1)
        gx[size_t(lv.off) + q] = lm.slot_X[q] >> shift;
        gy[size_t(lv.off) + q] = lm.slot_Y[q] >> shift;
      }
      if (M.k == 1) {
        D.levels[l].tile0 = int32_t(tiles.size());
        for (SmoothTile t : smooth_tiles(lm, lm, kSetupTile)) {
          t.pad = int32_t(l);
          tiles.push_back(t);
        }
      }
      for (size_t i = 0; i < lm.copy_leaf.size(); ++i) home[size_t(lv.off) + lm.copy_level[i]] = lm.copy_leaf[i];
    }
    D.lev_bricks = D.mem.upload(lb);
    D.n_lev_bricks = int32_t(lb.size());
    D.home_leaf = D.mem.upload(home);
    D.lev_leaf = D.mem.upload(leaf);
    D.lev_flags = D.mem.upload(flags);
    D.lev_gx = D.mem.upload(gx);
    D.lev_gy = D.mem.upload(gy);
    if (M.k == 1) D.setup_tiles = D.mem.upload(tiles);
    D.n_setup_tiles = int32_t(tiles.size());
    if (D.mem.err.empty())
      for (auto& L : D.levels) {
        L.lv.slot_leaf = D.lev_leaf + L.lv.off;
        L.lv.flags = D.lev_flags + L.lv.off;
        L.gx = D.lev_gx + L.lv.off;
        L.gy = D.lev_gy + L.lv.off;
      }
  }
  {
    // each free leaf node is on the copy list of exactly one level (its home)
    std::vector<int32_t> hoff(size_t(M.lay.n_slots), 0), hslot(size_t(M.lay.n_slots), -1),
        hnsl(size_t(M.lay.n_slots), 0);
    for (size_t l = 0; l < M.levels.size(); ++l) {
      const LevelMesh& lm = M.levels[l];
      for (size_t i = 0; i < lm.copy_leaf.size(); ++i) {
        const int32_t s = lm.copy_leaf[i];
        if (hslot[s] >= 0) {
          D.release();
          return "leaf slot on two copy lists";
        }
        hoff[s] = int32_t(D.levels[l].lv.off);
        hslot[s] = lm.copy_level[i];
        hnsl[s] = D.levels[l].lv.n_slots;
      }
    }
    D.home.off = D.mem.upload(hoff);
    D.home.slot = D.mem.upload(hslot);
    D.home.nsl = D.mem.upload(hnsl);
  }
  if (!D.mem.err.empty()) {
    std::string err = D.mem.err;
    D.release();
    return err;
  }
  D.uploaded = true;
  D.device = dev;
  return "";
}

std::string alloc_problem(pff_problem& pb) {
  const Mesh& M = pb.mesh->m;
  const int64_t ns = M.lay.n_slots;
  const int64_t nh = int64_t(M.hang.size());
  const DevMesh& D = pb.mesh->dev;
  const size_t nv = cell_values(pb);
  if (M.k == 1 && refinement_edges(D) && two_passes_f32(D.cells.ncells, ns)) pb.bufs.reserve(pb.cells32, nv);
  if (refinement_edges(D) && nv * sizeof(double) <= kCellsWithProblem) pb.bufs.reserve(pb.cells64, nv);
  pb.bufs.reserve(pb.lin64, 4 * ns);
  pb.bufs.reserve(pb.lin32, 4 * ns);
  pb.bufs.reserve(pb.cmask, ns);
  pb.bufs.reserve(pb.cmask_dir, ns);
  pb.bufs.reserve(pb.ibuf64, 3 * M.n_partials);
  pb.bufs.reserve(pb.ibuf32, 3 * M.n_partials);
  pb.bufs.reserve(pb.hlin64, 4 * nh);
  pb.bufs.reserve(pb.hlin32, 4 * nh);
  pb.bufs.reserve(pb.hx64, 3 * nh);
  pb.bufs.reserve(pb.hx32, 3 * nh);
  pb.bufs.commit();
  if (!pb.bufs.err.empty()) {
    std::string err = pb.bufs.err;
    pb.bufs.release();
    return err;
  }
  cudaMemset(pb.lin64, 0, 4 * ns * sizeof(double));
  cudaMemset(pb.lin32, 0, 4 * ns * sizeof(float));
  cudaError_t e = launch_leaf_cmask(ns, pb.mesh->dev.slot_flags, nullptr, pb.cmask, 0);
  if (e == cudaSuccess) e = launch_leaf_cmask(ns, pb.mesh->dev.slot_flags, nullptr, pb.cmask_dir, 0);
  if (e != cudaSuccess) return std::string("cmask: ") + cudaGetErrorString(e);
  cudaError_t e2 = cudaDeviceSynchronize();
  if (e2 != cudaSuccess) return std::string("sync: ") + cudaGetErrorString(e2);
  return "";
}

void fill_material(const pff_params& prm, ApplyArgs& a, bool unit_E) {
  const double E = unit_E ? 1.0 : prm.E;
  a.mu = E / (2.0 * (1.0 + prm.nu));
  a.lam = E * prm.nu / ((1.0 + prm.nu) * (1.0 - 2.0 * prm.nu));
  a.ell = prm.eps;
  a.kappa = prm.kappa;
  a.p = prm.p;
  a.gc_over_l = prm.Gc / prm.eps;
  a.gc_times_l = prm.Gc * prm.eps;
}

void leaf_modulus(const pff_problem& pb, int precision, ApplyArgs& a) {
  fill_material(pb.prm, a, pb.has_ecell);
  a.ecell = !pb.has_ecell ? nullptr
            : precision == PFF_F64 ? static_cast<const void*>(pb.ecell64) : static_cast<const void*>(pb.ecell32);
}

cudaError_t leaf_apply(pff_problem& pb, int precision, int op, const void* xu, const void* xp, void* yu,
                       void* yp, cudaStream_t s) {
  const Mesh& M = pb.mesh->m;
  const DevMesh& D = pb.mesh->dev;
  ApplyArgs a;
  std::memset(&a, 0, sizeof(a));
  a.lay = D.leaf;
  a.lc = D.cells;
  std::unique_lock<std::mutex> lk(pb.cells_mu, std::defer_lock);
  if (precision == PFF_F32) {
    a.lc.out = pb.cells32;
  } else if (refinement_edges(D)) {
    a.lc.out = leaf_contributions64(pb);
  } else if (M.k == 2 || pb.sweep_sh == 0) {
    lk.lock();
    a.lc.out = stream_contributions(pb, s);
  }
  a.hang = D.hang;
  a.cmask = pb.cmask;
  a.lin = precision == PFF_F64 ? static_cast<const void*>(pb.lin64) : static_cast<const void*>(pb.lin32);
  a.xu = xu; a.xp = xp; a.yu = yu; a.yp = yp;
  a.ibuf = precision == PFF_F64 ? static_cast<void*>(pb.ibuf64) : static_cast<void*>(pb.ibuf32);
  a.hlin = precision == PFF_F64 ? static_cast<const void*>(pb.hlin64) : static_cast<const void*>(pb.hlin32);
  a.hang_x = precision == PFF_F64 ? static_cast<void*>(pb.hx64) : static_cast<void*>(pb.hx32);
  a.nhang = D.nhang;
  a.n_slots = M.lay.n_slots;
  for (int l = 0; l <= M.Lf && l < kMaxLevels; ++l) {
    a.hx[l] = M.tree.hx(l);
    a.hy[l] = M.tree.hy(l);
  }
  leaf_modulus(pb, precision, a);
  fill_cell_constants(a, M.Lf + 1);
  a.fe_degree = M.k;
  a.sweep_sh = pb.sweep_sh;
  int kop = OP_FULL;
  if (op == PFF_OP_JACOBIAN) { kop = OP_FULL; a.mode = MODE_MASK_INPUT | MODE_IDENTITY; }
  else if (op == PFF_OP_TRANSPOSE) { kop = OP_FULL_T; a.mode = MODE_MASK_INPUT | MODE_IDENTITY; }
  else { kop = OP_FULL; a.mode = 0; }
  FixupArgs f;
  f.n = D.nfix; f.n_slots = M.lay.n_slots; f.slot = D.fix_slot; f.ptr = D.fix_ptr; f.part = D.fix_part; f.w = D.fix_w;
  f.cmask = pb.cmask; f.xu = xu; f.xp = xp; f.yu = yu; f.yp = yp; f.ibuf = a.ibuf; f.mode = a.mode;
  return precision == PFF_F64 ? launch_leaf<double>(a, f, kop, s) : launch_leaf<float>(a, f, kop, s);
}

}  // namespace pff
