// Resident FP64 CG: many iterations per launch with the CG vectors held on
// chip (internal; see eik_res64.cu).
#pragma once

#include "eik_internal.cuh"

namespace eik {

// How one grid is split over the blocks: cx x cy x cz bricks, brick i of an
// axis covering nodes [i n / c, (i + 1) n / c).
struct Res64Plan {
  bool ok = false;
  int cx = 1, cy = 1, cz = 1, nblk = 0;
  int bx = 1, by = 1, bz = 1;   // largest brick
  int halo = 0;                 // most halo nodes of a brick
  int per_thread = 0;           // nodes per thread (template instance)
  size_t smem = 0, inbox_words = 0;
  unsigned epoch = 0;           // tags used so far
};

// Plans the resident kernel for g (ok = false where the grid does not fit on
// chip or the device cannot run it).
void res64_plan(Res64Plan *pl, const Grid &g, int num_sms);
// Runs up to a few hundred CG iterations from (x, r, p) and *st, as the two
// passes of eik_cg64.cu do, and writes them back.  msg: the solver's message
// buffer (kSyncBytes) and inbox the halo buffer (inbox_words), both zeroed
// when they were allocated.  withhold: test hook, one block does not arrive in
// the launch's first grid-wide sum, so that the waits run out (EIK_ERR_TIMEOUT).
cudaError_t launch_res64(Res64Plan *pl, const Grid &g, const double *sig, double *x, double *r,
                         double *p, const double *cw_weight, CgState *st,
                         unsigned long long *msg, unsigned long long *inbox, bool withhold,
                         cudaStream_t s);

}  // namespace eik
