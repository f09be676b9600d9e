// The dense level-0 blocks of the direct coarse solve: assembly and inversion (coarse.cu).
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

namespace pff {

// One block (0: u-u, 1: phi-phi) of the level-0 matrix.  Entries: the block's components
// on the level-0 nodes, without Dirichlet ones, free entries first (coarse_order); fixed
// ones (active phi) are identity rows and columns.
struct CoarseBlock {
  int32_t n;             // entries
  int nc, fix0;          // components; constraint-mask bit of component 0 (1 or 4)
  const int32_t* all;    // the entries by slot: comp * n_0 + slot
  int32_t* idx;          // in the order of the matrix
  int32_t* ent;          // its inverse: per comp * n_0 + slot the entry or -1
  double* Ke;            // per cell its element matrix, [row][column], dof = node * nc + comp
  double* A;             // n x n
  double* scr;           // scratch of the inversion (coarse_scratch(n) doubles)
};
struct CoarseArgs {
  CoarseBlock b[2];
  int k, ncx, ncy;         // element degree, coarse cells
  int32_t n0;              // level-0 slots
  const int32_t* node_slot;   // slot of level-0 grid node (gx, gy) at gx + (k ncx + 1) gy
  const int32_t* gx;
  const int32_t* gy;
  const uint8_t* cmask;    // level-0 constraint mask
  int32_t* bad;            // per block: set to 1 when a pivot is not positive
};

int64_t coarse_scratch(int32_t n);
// the entries' order (idx, ent), and A of both blocks from the element matrices
cudaError_t coarse_fill(const CoarseArgs& a, cudaStream_t s);
// A <- A^-1 of both blocks (SPD), side by side in the same launches
cudaError_t coarse_invert(const CoarseArgs& a, cudaStream_t s);

}  // namespace pff
