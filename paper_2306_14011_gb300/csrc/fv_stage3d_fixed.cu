// 3D stage kernels compiled for one tile shape and thread count each (minmod):
// every shared-memory offset of the face loops is a constant.
#include "fv_stage.cuh"

namespace fvk {
namespace {
// 8x8x8 cells: 9 faces on each of 64 lines per axis, 192 runs of 3 for the 192
// threads (TGV 192^3: 6.85 ms per step; with run-time offsets 7.80); 4x4x4 for
// grids that would leave SMs idle.
template <int TX, int TY, int TZ, int THREADS, int MINB>
using Kernels = StageKernels<3, FV_LIM_MINMOD, THREADS, MINB, Shape<TX, TY, TZ, THREADS>>;

template <class SH, class K>
bool take(int mode, const CUtensorMap *tmap, const StageArgs &a, int threads, cudaStream_t st, cudaError_t *e) {
  if (a.limiter != FV_LIM_MINMOD || threads != SH::THREADS || a.tile[0] != SH::TX || a.tile[1] != SH::TY ||
      a.tile[2] != SH::TZ)
    return false;
  *e = K::launch(mode, tmap, a, threads, st);
  return true;
}
}  // namespace

bool launch_stage_fixed_3d(int mode, const CUtensorMap *tmap, const StageArgs &a, int threads, cudaStream_t st,
                     cudaError_t *e) {
  return take<Shape<8, 8, 8, 192>, Kernels<8, 8, 8, 192, 2>>(mode, tmap, a, threads, st, e) ||
         take<Shape<4, 4, 4, 96>, Kernels<4, 4, 4, 96, 4>>(mode, tmap, a, threads, st, e);
}

// (the 4x4x4 CTAs stay below 48 KB)
cudaError_t set_stage_attributes_fixed_3d(size_t smem) { return Kernels<8, 8, 8, 192, 2>::set_attributes(smem); }
}  // namespace fvk
