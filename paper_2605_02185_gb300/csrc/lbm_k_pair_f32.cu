// lbm_k_pair_f32.cu -- the two-step kernel for float storage.
#include "../../include/gblbm.h"
#include "lbm_pair.cuh"

namespace gblbm {

cudaError_t pair_f32(int grid, void *buf0, void *buf1, const StepParams &p, const PairParams &q, cudaStream_t st,
                     int mode, int *occ) {
  float *a = (float *)buf0, *b = (float *)buf1;
  return p.qmap ? pair_one<kPairWarps, kPairStages, true, false>(grid, a, b, p, nullptr, 1, p.mrt, q, st, mode, occ)
                : pair_one<kPairWarps, kPairStages, false, false>(grid, a, b, p, nullptr, 1, p.mrt, q, st, mode, occ);
}

cudaError_t pair_batch_f32(int grid, const CaseDesc *cases, int ncases, int mrt, const PairParams &q, cudaStream_t st,
                           int mode, int *occ) {
  return pair_one<kPairWarps, kPairStages, false, true>(grid, nullptr, nullptr, StepParams{}, cases, ncases, mrt, q, st,
                                                        mode, occ);
}

}  // namespace gblbm
