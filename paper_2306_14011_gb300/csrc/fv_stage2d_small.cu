// 2D stage kernels compiled for one tile shape and thread count each (minmod):
// every shared-memory offset of the face loops is a constant.
#include "fv_stage.cuh"

namespace fvk {
namespace {
// Tiles for grids that larger ones would leave SMs idle on (auto_launch in
// fv_api.cu): one, two or three faces per thread and axis.
template <int TX, int TY, int TZ, int THREADS, int MINB>
using Kernels = StageKernels<2, FV_LIM_MINMOD, THREADS, MINB, Shape<TX, TY, TZ, THREADS>>;

template <class SH, class K>
bool take(int mode, const CUtensorMap *tmap, const StageArgs &a, int threads, cudaStream_t st, cudaError_t *e) {
  if (a.limiter != FV_LIM_MINMOD || threads != SH::THREADS || a.tile[0] != SH::TX || a.tile[1] != SH::TY ||
      a.tile[2] != SH::TZ)
    return false;
  *e = K::launch(mode, tmap, a, threads, st);
  return true;
}
}  // namespace

bool launch_stage_small_2d(int mode, const CUtensorMap *tmap, const StageArgs &a, int threads, cudaStream_t st,
                     cudaError_t *e) {
  return take<Shape<16, 8, 1, 96>, Kernels<16, 8, 1, 96, 4>>(mode, tmap, a, threads, st, e) ||
         take<Shape<16, 4, 1, 96>, Kernels<16, 4, 1, 96, 4>>(mode, tmap, a, threads, st, e) ||
         take<Shape<16, 16, 1, 96>, Kernels<16, 16, 1, 96, 4>>(mode, tmap, a, threads, st, e);
}
}  // namespace fvk
