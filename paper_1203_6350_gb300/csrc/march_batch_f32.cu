// The batched marching kernels for float storage.
#include "lbm_march_batch.cuh"

namespace lbm {

cudaError_t launch_march_batch_f32(const MarchBatch& p, int variant, cudaStream_t st, int pdl) {
    return launch_march_batch_t<float, 3>(p, variant, st, pdl);
}

}  // namespace lbm
