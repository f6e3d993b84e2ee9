// The batched marching kernels for __nv_bfloat16 storage.
#include "lbm_march_batch.cuh"

namespace lbm {

cudaError_t launch_march_batch_bf16(const MarchBatch& p, int variant, cudaStream_t st, int pdl) {
    return launch_march_batch_t<__nv_bfloat16, 2>(p, variant, st, pdl);
}

}  // namespace lbm
