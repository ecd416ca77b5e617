// FP64 fused step, 3/4/6 nodes per axis (storage and arithmetic in double): velocity slices NS per nodes M an axis.
// (instantiation list; the kernel is in step_tile.cuh)
#include "step_tile.cuh"

using namespace lbmk;

#define LBM_TILE_LIST(X) X(3, 1) X(4, 1) X(4, 2) X(4, 4) X(6, 1) X(6, 2) X(6, 6)

cudaError_t launch_step_f64_small(int m, int ns, bool resid, const StepArgs &a, cudaStream_t s)
{
#define LBM_TILE_LAUNCH(M_, NS_)                                                                   \
    if (m == M_ && ns == NS_)                                                                      \
        return resid ? launch_tile<double, double, M_, NS_, true, false, false>(a, s)              \
                     : launch_tile<double, double, M_, NS_, false, false, false>(a, s);
    LBM_TILE_LIST(LBM_TILE_LAUNCH)
#undef LBM_TILE_LAUNCH
    return cudaErrorInvalidValue;
}
