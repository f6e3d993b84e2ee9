// The marching kernels for float population storage, periodic boundary.
#include "lbm_march.cuh"

namespace lbm {

cudaError_t launch_march_f32_periodic(const void* src, void* dst, const Geometry& g,
                                      const StepConst<F2>& k, const AxisCoef<float>* tx,
                                      const AxisCoef<float>* ty, int variant, int seg,
                                      cudaStream_t st, int pdl) {
    return launch_march_t<float, kPeriodic, 3, false>(src, dst, g, k, tx, ty, variant, seg, st,
                                                      pdl);
}

}  // namespace lbm
