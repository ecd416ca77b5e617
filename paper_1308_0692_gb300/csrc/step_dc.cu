// Kernels of the mixed-precision refinement of the FP32 march:
//   defect  : one step evaluated in FP64 arithmetic on the FP32 state, storing the
//             change M(h) - h (the defect) as float, with its norms;
//   correct : the FP32 step of the homogeneous problem (wall driving removed) plus a
//             source array -- the correction equation delta = L(delta) + defect.
// The slices are those tile_plan (lbm_api.cu) picks for either arithmetic.
// (instantiation list; the kernel is in step_tile.cuh)
#include "step_tile.cuh"

using namespace lbmk;

cudaError_t launch_defect_f32_large(int ns, const StepArgs &a, cudaStream_t s);                  // step_dc_large.cu
cudaError_t launch_correct_f32_large(int ns, bool resid, const StepArgs &a, cudaStream_t s);

cudaError_t launch_defect_f32(int m, int ns, const StepArgs &a, cudaStream_t s)
{
#define LBM_DEFECT(M_, NS_) \
    if (m == M_ && ns == NS_) return launch_tile<float, double, M_, NS_, false, false, true>(a, s);
    LBM_DEFECT(3, 1) LBM_DEFECT(4, 1) LBM_DEFECT(4, 4) LBM_DEFECT(6, 2) LBM_DEFECT(6, 6) LBM_DEFECT(8, 4) LBM_DEFECT(8, 8)
#undef LBM_DEFECT
    return m == 12 ? launch_defect_f32_large(ns, a, s) : cudaErrorInvalidValue;
}

cudaError_t launch_correct_f32(int m, int ns, bool resid, const StepArgs &a, cudaStream_t s)
{
#define LBM_CORRECT(M_, NS_)                                                                       \
    if (m == M_ && ns == NS_)                                                                      \
        return resid ? launch_tile<float, float, M_, NS_, true, true, false>(a, s)                 \
                     : launch_tile<float, float, M_, NS_, false, true, false>(a, s);
    LBM_CORRECT(3, 1) LBM_CORRECT(4, 1) LBM_CORRECT(4, 4) LBM_CORRECT(6, 2) LBM_CORRECT(6, 6) LBM_CORRECT(8, 4) LBM_CORRECT(8, 8)
#undef LBM_CORRECT
    return m == 12 ? launch_correct_f32_large(ns, resid, a, s) : cudaErrorInvalidValue;
}
