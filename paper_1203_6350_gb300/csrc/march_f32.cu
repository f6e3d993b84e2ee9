// The marching kernels (several time steps per launch) for float population
// storage, Dirichlet boundary: three steps per launch.
#include "lbm_march.cuh"

namespace lbm {

cudaError_t launch_march_f32_dirichlet(const void* src, void* dst, const Geometry& g,
                                       const StepConst<F2>& k, const AxisCoef<float>* tx,
                                       const AxisCoef<float>* ty, int variant, int seg,
                                       cudaStream_t st, int pdl) {
    return launch_march_t<float, kDirichlet, 3, false>(src, dst, g, k, tx, ty, variant, seg, st,
                                                       pdl);
}

}  // namespace lbm
