// Resident FP32 inner CG of the 2D mixed solve: many iterations per launch
// with r, p and sigma held on chip (internal; see eik_res32.cu).
#pragma once

#include "eik_cg32.h"

namespace eik {

// How one 2D grid is split over the blocks: tx x ty tiles, tile i of x
// covering the four-column chunks [i n4 / tx, (i + 1) n4 / tx), n4 = ceil(nx / 4),
// tile j of y the rows [j ny / ty, (j + 1) ny / ty).
struct Res32Plan {
  bool ok = false;
  int tx = 1, ty = 1, nblk = 0;
  int pw = 0, ht = 0;            // widest tile (columns, a multiple of 4) and tallest
  int instance = 0;              // template instance (by tile height)
  size_t smem = 0, inbox_words = 0;
  unsigned epoch = 0;            // tags used so far
  unsigned long long *msg = nullptr;   // message buffer, then the inboxes; zeroed
};

// Plans the kernel for a 2D grid (ok = false where it does not fit on chip or
// the device cannot run it), allocating and zeroing the message buffer on s.
void res32_plan(Res32Plan *pl, const Grid &g, const CellGrid &cg, int num_sms, cudaStream_t s);
void res32_destroy(Res32Plan *pl);
// Runs a few hundred inner iterations at most from (r, p)[0], d and *st (as
// left by the FP64 residual kernel, or by the launch before), and writes them
// back.
cudaError_t launch_res32(Res32Plan *pl, const Grid &g, const CellGrid &cg, const Cg32Buffers &b,
                         cudaStream_t s);

}  // namespace eik
