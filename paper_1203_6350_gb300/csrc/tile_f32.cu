// The tile kernels (several time steps per launch on small lattices) for float storage.
#include "lbm_tile.cuh"

namespace lbm {

cudaError_t launch_tile_f32(const void* src, void* dst, const Geometry& g, const StepConst<F2>& k,
                            const AxisCoef<float>* tx, const AxisCoef<float>* ty, int variant,
                            int bc, int h, int levels, cudaStream_t st, int pdl,
                            const LineSource& ls) {
    return launch_tile_t<float>(src, dst, g, k, tx, ty, variant, bc, tile_shape(h, levels), st,
                                pdl, ls);
}

cudaError_t prepare_tile_f32(int variant, int bc, int h, int levels) {
    return prepare_tile_t<float>(variant, bc, tile_shape(h, levels));
}

}  // namespace lbm
