// 2D stage kernels compiled for one tile shape and thread count each (minmod):
// every shared-memory offset of the face loops is a constant.
#include "fv_stage.cuh"

namespace fvk {
namespace {
// 48x13 cells: 91 and 96 runs of 7 faces for the 96 threads (93% and 97% of
// their steps), 57 KB of shared memory: four CTAs, 12 warps, per SM, which mix
// their load and face phases better than two CTAs of 192 threads (KH 2048^2:
// 1.83 ms per step; 32x19 and 96: 1.84, 24x19 and 96: 1.85, 64x14 and 128: 1.89,
// 48x27 and 192: 1.91, 64x17 and 192: 2.08).
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

bool launch_stage_fixed_2d(int mode, const CUtensorMap *tmap, const StageArgs &a, int threads, cudaStream_t st,
                     cudaError_t *e) {
  return take<Shape<48, 13, 1, 96>, Kernels<48, 13, 1, 96, 4>>(mode, tmap, a, threads, st, e) ||
         take<Shape<24, 19, 1, 96>, Kernels<24, 19, 1, 96, 4>>(mode, tmap, a, threads, st, e);
}

// (the 24x19 CTAs stay below 48 KB)
cudaError_t set_stage_attributes_fixed_2d(size_t smem) { return Kernels<48, 13, 1, 96, 4>::set_attributes(smem); }
}  // namespace fvk
