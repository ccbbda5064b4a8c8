// 2D stage kernels compiled for one tile shape and thread count each (minmod):
// every shared-memory offset of the face loops is a constant.
#include "fv_stage.cuh"

namespace fvk {

// 48x13 cells: 91 and 96 runs of 7 faces for the 96 threads (93% and 97% of
// their steps), 57 KB of shared memory: four CTAs, 12 warps, per SM, which mix
// their load and face phases better than two CTAs of 192 threads (KH 2048^2:
// 1.83 ms per step; 32x19 and 96: 1.84, 24x19 and 96: 1.85, 64x14 and 128: 1.89,
// 48x27 and 192: 1.91, 64x17 and 192: 2.08).
bool launch_stage_fixed_2d(int mode, const CUtensorMap *tmap, const StageArgs &a, int threads, cudaStream_t st,
                           cudaError_t *e) {
  return launch_shape<2, FV_LIM_MINMOD, 4, Shape<48, 13, 1, 96>>(mode, tmap, a, threads, st, e) ||
         launch_shape<2, FV_LIM_MINMOD, 4, Shape<24, 19, 1, 96>>(mode, tmap, a, threads, st, e);
}

// (the 24x19 CTAs stay below 48 KB)
cudaError_t set_stage_attributes_fixed_2d(size_t smem) {
  return StageKernels<2, FV_LIM_MINMOD, 96, 4, Shape<48, 13, 1, 96>>::set_attributes(smem);
}
}  // namespace fvk
