// FP32 fused step, 12 nodes per axis (storage and arithmetic in float): velocity slices NS per nodes M an axis.
// (instantiation list; the kernel is in step_tile.cuh)
#include "step_tile.cuh"

using namespace lbmk;

#define LBM_TILE_LIST(X) X(12, 2) X(12, 3) X(12, 4) X(12, 6)

cudaError_t launch_step_f32_large(int m, int ns, bool resid, const StepArgs &a, cudaStream_t s)
{
#define LBM_TILE_LAUNCH(M_, NS_)                                                                   \
    if (m == M_ && ns == NS_)                                                                      \
        return resid ? launch_tile<float, float, M_, NS_, true, false, false>(a, s)              \
                     : launch_tile<float, float, M_, NS_, false, false, false>(a, s);
    LBM_TILE_LIST(LBM_TILE_LAUNCH)
#undef LBM_TILE_LAUNCH
    return cudaErrorInvalidValue;
}
