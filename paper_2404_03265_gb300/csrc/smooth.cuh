// Tiled level kernels of the Q1 V-cycle: the FP32 smoothers (smooth.cu) and the set-up of
// all levels (setup.cu).
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

#include "kernels.cuh"

namespace pff {

// A tile of node positions of a level brick: tile x tile nodes, tile in {6, 10, 15}
// (25, 9 or 4 tiles per brick; only tiles that hold a node are listed).  Node (n, r)
// of the window around the tile lies in one of the brick's 3x3 neighbours; the coarser
// level's nodes under the window lie in the 3x3 neighbours of the parent brick.
struct SmoothTile {
  int32_t fb[9];   // storage bases of the brick's 3x3 neighbours on this level (-1 absent)
  int32_t cb[9];   // the same of the parent brick (bx / 2, by / 2) on the next coarser level
  int32_t pos;     // tile column | tile row << 3 | (bx & 1) << 6 | (by & 1) << 7
  int32_t pad;     // the level (set-up tiles)
};

// A brick of the concatenated level storage (900 slots): its level's slot offset
// and slot count, and the brick's first slot on its level.
struct LevBrick {
  int32_t off, n, base;
};

// One level and block of the V-cycle.  Vectors: ncomp blocks of n (coarse: nc) floats.
struct SmoothArgs {
  const SmoothTile* tiles;
  int32_t ntiles, tile;    // tiles, and nodes per tile side
  int32_t n, nc;           // slots of this level, of the next coarser one
  const uint8_t* flags;    // level slot flags: bit0 node, bit5 the cell whose lower-left node this is exists
  const uint8_t* cmask;
  const uint8_t* cmask_c;
  const float* lin;        // 4 blocks of n
  const float* ecell;      // per-cell modulus at cell slots, or nullptr
  const float* dinv;
  const float* d;          // level defect
  float* dc;               // down: coarse defect, the restricted residual is added
  const float* x;          // up: the pre-smoothed iterate
  const float* xc;         // up: the coarse correction
  float* xout;             // down: the pre-smoothed iterate; up: the level's result
  MatConst<float> m;
  LevGeom<float> g;
  float c0, a1, b1, a2, b2;   // Chebyshev steps: c0 D^-1, then (a, b) of cheb_next twice; all 0: no smoothing
};

// Down: x = p(D^-1 A) D^-1 d (Chebyshev degree 3 from zero), then dc += P^T (d - A x).
// Up: x += P xc, then x += p(D^-1 A) D^-1 (d - A x).
// op: OP_UU or OP_PP.  Launched programmatically dependent on the preceding kernel of
// the stream (up: when pdl is set).  Up reads d and x before it waits for that kernel,
// so with pdl that kernel must let it start (pdl_trigger) only after the one that
// wrote d and x has completed.
cudaError_t launch_smooth_down(const SmoothArgs& a, int op, cudaStream_t s);
cudaError_t launch_smooth_up(const SmoothArgs& a, int op, cudaStream_t s, bool pdl);

// ---- set-up of all levels at once (Q1): the inverse diagonals, and the CG runs of the
// eigenvalue estimate with FP32 applies.  Tiles of kSetupTile nodes of every level,
// level by level (SmoothTile::pad: the level); vectors of level l at ncomp off_l in the
// concatenated level storage.
constexpr int kSetupTile = 15;
struct SetupArgs {
  const SmoothTile* tiles;
  int32_t ntiles;
  const uint8_t* flags;      // concatenated level flags and masks
  const uint8_t* cmask;
  const double* lin64;       // per level 4 blocks
  const float* lin32;
  const double* ecell64;     // concatenated cell modulus, or nullptr
  const float* ecell32;
  const int32_t* gx;         // concatenated level-grid coordinates
  const int32_t* gy;
  double* dinv64;
  float* dinv32;
  double *r, *z, *p[2];      // CG vectors; p of step j in p[j % 2]
  float* q;
  double *sc, *hist;         // per level 8 scalars; hist_stride doubles (alpha_j, beta_j per step)
  int32_t hist_stride;
  double* partial;           // dot0[kMaxLevels] doubles
  unsigned* count;           // per level, 0 between launches
  int32_t off[kMaxLevels], n[kMaxLevels];   // per level: slot offset and count,
  int32_t dot0[kMaxLevels + 1];             // its first block of a dot (level 0: none; see setup_dot_blocks)
  int32_t tile1;                            // first tile of level 1
  MatConst<float> mf;
  MatConst<double> md;
  LevGeom<float> gf[kMaxLevels];
  LevGeom<double> gd[kMaxLevels];
};
// blocks of a dot over nn entries
inline int32_t setup_dot_blocks(int64_t nn) { return int32_t(nn <= 0 ? 1 : nn >= 512 * 256 ? 512 : (nn + 255) / 256); }
// op: OP_UU or OP_PP
cudaError_t launch_setup_diag(const SetupArgs& a, int op, cudaStream_t s);
cudaError_t launch_setup_cg(const SetupArgs& a, int op, int steps, cudaStream_t s);

}  // namespace pff
