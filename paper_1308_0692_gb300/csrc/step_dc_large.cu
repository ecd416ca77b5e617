// The refinement's defect and correction kernels (step_dc.cu) of the 144-velocity set: a
// translation unit of their own, since a kernel's first launch loads its whole unit.
#include "step_tile.cuh"

using namespace lbmk;

cudaError_t launch_defect_f32_large(int ns, const StepArgs &a, cudaStream_t s)
{
    if (ns == 4) return launch_tile<float, double, 12, 4, false, false, true>(a, s);
    if (ns == 12) return launch_tile<float, double, 12, 12, false, false, true>(a, s);
    return cudaErrorInvalidValue;
}

cudaError_t launch_correct_f32_large(int ns, bool resid, const StepArgs &a, cudaStream_t s)
{
#define LBM_CORRECT(NS_)                                                                           \
    if (ns == NS_)                                                                                 \
        return resid ? launch_tile<float, float, 12, NS_, true, true, false>(a, s)                 \
                     : launch_tile<float, float, 12, NS_, false, true, false>(a, s);
    LBM_CORRECT(2) LBM_CORRECT(4) LBM_CORRECT(6)
#undef LBM_CORRECT
    return cudaErrorInvalidValue;
}
