// 3D stage kernels compiled for one tile shape and thread count each (minmod):
// every shared-memory offset of the face loops is a constant.
#include "fv_stage.cuh"

namespace fvk {

// 8x8x8 cells: 9 faces on each of 64 lines per axis, 192 runs of 3 for the 192
// threads (TGV 192^3: 6.85 ms per step; with run-time offsets 7.80); 4x4x4 for
// grids that would leave SMs idle.
bool launch_stage_fixed_3d(int mode, const CUtensorMap *tmap, const StageArgs &a, int threads, cudaStream_t st,
                           cudaError_t *e) {
  return launch_shape<3, FV_LIM_MINMOD, 2, Shape<8, 8, 8, 192>>(mode, tmap, a, threads, st, e) ||
         launch_shape<3, FV_LIM_MINMOD, 4, Shape<4, 4, 4, 96>>(mode, tmap, a, threads, st, e);
}

// (the 4x4x4 CTAs stay below 48 KB)
cudaError_t set_stage_attributes_fixed_3d(size_t smem) {
  return StageKernels<3, FV_LIM_MINMOD, 192, 2, Shape<8, 8, 8, 192>>::set_attributes(smem);
}
}  // namespace fvk
