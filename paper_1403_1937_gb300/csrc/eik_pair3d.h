// Two-pass FP32 inner CG of the 3D mixed solve (internal; csrc/eik_pair3d.cu).
#pragma once

#include "eik_cg32.h"

namespace eik {

struct PairCtl;

struct Pair3Plan {
  bool ok = false;
  int tiles_x = 0, tiles_y = 0, zc = 0, ntiles = 0, nblk_dir = 0;
  int step_x = 0, step_y = 0, nblk_step = 0;   // block shape and count of the step pass
  PairCtl *ctl = nullptr;
  double *part = nullptr;
};

// Fills *pl; pl->ok stays false for 2D grids and when the device refuses a
// resource (the one-pass kernels serve those).
void pair3_plan(Pair3Plan *pl, const Grid &g, const CellGrid &cg, int num_sms, cudaStream_t s);
void pair3_destroy(Pair3Plan *pl);
// One inner iteration; r in b.r[0], directions read from b.p[set] and written
// to b.p[1 - set], A p in b.r[1].  The inner solve starts with r and p = 0 as
// the residual kernel leaves them, MixCtl.iter = 0, and r to be moved to frame
// MixCtl.F + MixCtl.dF.
void pair3_iter(const Pair3Plan &pl, const Grid &g, const CellGrid &cg, const Cg32Buffers &b,
                int set, cudaStream_t s);

}  // namespace eik
