// The batched marching kernels for __half storage.
#include "lbm_march_batch.cuh"

namespace lbm {

cudaError_t launch_march_batch_f16(const MarchBatch& p, int variant, cudaStream_t st, int pdl) {
    return launch_march_batch_t<__half, 2>(p, variant, st, pdl);
}

}  // namespace lbm
