// 2D stage kernels compiled for one tile shape and thread count each (minmod):
// every shared-memory offset of the face loops is a constant.
#include "fv_stage.cuh"

namespace fvk {

// Tiles for grids that larger ones would leave SMs idle on (auto_launch in
// fv_api.cu): one, two or three faces per thread and axis.
bool launch_stage_small_2d(int mode, const CUtensorMap *tmap, const StageArgs &a, int threads, cudaStream_t st,
                           cudaError_t *e) {
  return launch_shape<2, FV_LIM_MINMOD, 4, Shape<16, 8, 1, 96>>(mode, tmap, a, threads, st, e) ||
         launch_shape<2, FV_LIM_MINMOD, 4, Shape<16, 4, 1, 96>>(mode, tmap, a, threads, st, e) ||
         launch_shape<2, FV_LIM_MINMOD, 4, Shape<16, 16, 1, 96>>(mode, tmap, a, threads, st, e);
}
}  // namespace fvk
