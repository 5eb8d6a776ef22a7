// lbm_pair_host.h -- host side of the two-step kernel: the cells its warps work
// on, shared by single lattices and batches.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>
#include <vector>

#include "lbm_ctx.h"
#include "lbm_internal.h"

namespace gblbm {

// Capacities of a workspace region for `cases` lattices; a plan that needs more
// leaves its lattices to the one-step kernels.
constexpr int kPairCellsSingle = 8192, kPairSlotsSingle = 512;
constexpr int kPairCellsBatch = 8192, kPairSlotsBatch = 4096;
size_t pair_region_bytes(int cells, int slots, int cases);

struct PairLattice {
  int nx, ny, bc;
  const Geometry *geo;
};

// Split the lattices over the warps of `sms` SMs, upload the tables into `region`
// (pair_region_bytes() of it) on `st` and fill q (q->pairs: the most passes of a
// launch) and *grid.  LBM_OK with *grid = 0
// where the kernel does not take them.
int pair_plan(const std::vector<PairLattice> &lattices, int sms, void *region, int cells_cap, int slots_cap,
              cudaStream_t st, PairParams *q, int *grid);
// Of n steps, those to take in pairs: all but an odd one.  Under a caller's stream
// capture a multiple of four, so that an even number of steps ends in the buffer it
// began in (each pass changes it) and the graph can be launched again.
int64_t pair_steps_of(cudaStream_t st, int64_t n);
// False where a fault is injected but no cell of these n steps would wait for another
// (a launch of one pass): the one-step kernel, whose tiles wait for their copies, then
// takes them.
inline bool pair_waits(const StepParams &p, const PairParams &q, int64_t n) {
  return p.fault_tile < 0 || (n >= 4 && q.pairs >= 2);
}

}  // namespace gblbm
