// The marching kernels for FP16 deviation storage, periodic boundary: two steps per
// launch with the level between them in FP32 (each_level = false), or three steps
// each rounded to the format as one step per launch rounds it.
#include "lbm_march.cuh"

namespace lbm {

cudaError_t launch_march_f16_periodic(const void* src, void* dst, const Geometry& g,
                                   const StepConst<F2>& k, const AxisCoef<float>* tx,
                                   const AxisCoef<float>* ty, int variant, bool each_level,
                                   int seg, cudaStream_t st, int pdl) {
    if (each_level)
        return launch_march_t<__half, kPeriodic, 3, true>(src, dst, g, k, tx, ty, variant, seg, st, pdl);
    return launch_march_t<__half, kPeriodic, 2, false>(src, dst, g, k, tx, ty, variant, seg, st, pdl);
}

}  // namespace lbm
