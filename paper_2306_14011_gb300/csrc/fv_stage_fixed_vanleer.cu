// The stage kernels of the main tile shapes for the van Leer limiter, every
// shared-memory offset of the face loops a constant (as fv_stage2d_fixed.cu and
// fv_stage3d_fixed.cu for minmod).
// 1021x767, van Leer on primitive variables, 24x19 tiles, 4 steps: 2.93 ms; with
// run-time offsets 3.11 (both with a slope of three roundings; 2.72 now).
#include "fv_stage.cuh"

namespace fvk {

bool launch_stage_fixed_vanleer(int dim, int mode, const CUtensorMap *tmap, const StageArgs &a, int threads,
                           cudaStream_t st, cudaError_t *e) {
  if (dim == 3) return launch_shape<3, FV_LIM_VANLEER, 2, Shape<8, 8, 8, 192>>(mode, tmap, a, threads, st, e);
  return launch_shape<2, FV_LIM_VANLEER, 4, Shape<48, 13, 1, 96>>(mode, tmap, a, threads, st, e) ||
         launch_shape<2, FV_LIM_VANLEER, 4, Shape<24, 19, 1, 96>>(mode, tmap, a, threads, st, e);
}

// (the 24x19 CTAs stay below 48 KB)
cudaError_t set_stage_attributes_fixed_vanleer(int dim, size_t smem) {
  return dim == 3 ? StageKernels<3, FV_LIM_VANLEER, 192, 2, Shape<8, 8, 8, 192>>::set_attributes(smem)
                  : StageKernels<2, FV_LIM_VANLEER, 96, 4, Shape<48, 13, 1, 96>>::set_attributes(smem);
}
}  // namespace fvk
