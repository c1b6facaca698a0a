// The cooperative solve kernel of persist.cu.
#pragma once

#include "sph_internal.cuh"
#include "tiles.cuh"

namespace sph {

// what the host reads back
struct PersistResult {
  double rr[3];        // squared norms of r64 (updated, not recomputed from x)
  int32_t passes, iters, last_iter;
  int32_t stuck;       // the last pass ran no iteration
  int32_t stalled;     // bit c: component c stalled in some pass
  int32_t state[3];    // of the last pass
  int32_t done;        // the kernel came to its end
  int32_t fault;       // a grid barrier gave up
};

// Whether the handle's tiles fit one block per SM (persist.cu), and the launch for it
struct PersistPlan {
  bool ok = false;
  int grid = 0, tiles_per_block = 0, splits = 1, ucap = 0, rcap = 0;
  size_t smem = 0;
};
PersistPlan persist_plan(const sph_neighbors* H);

// Refinement passes from the residual r64 (squared norms rr0) until its updated norm
// is at most tol, max_pass passes or maxit iterations have run, or nothing moves.
// x64 and r64 follow.  view: the tile form with the preconditioner's 1/D; D64 its
// diagonal.  Synchronises.
sph_status persist_solve(sph_neighbors* H, const PersistPlan& plan, const TileView& view, const double* D64, double tol,
                         double eps_floor, const double rr0[3], int maxit, int max_pass, PersistResult* out,
                         cudaStream_t st);

}  // namespace sph
