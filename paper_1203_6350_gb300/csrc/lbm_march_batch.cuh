// The marching kernel over many lattices: one launch advances up to kMarchItems
// Dirichlet instances of one variant.  The instances' constants, buffers and cuts are the
// kernel's parameters, so they come through the constant path and stay in uniform
// registers (the batched tile kernels read them from shared memory at each use).
//
// What bounds it beside the walks themselves (lbm_march.cuh) is that path: the blocks an SM
// holds together should share an instance's constants, hence the order of the walks over
// the blocks (64 lattices of sides 64-1024 in FP32: 72 us per step in plain order, 61
// in this one, 86 with the TMA-staged tiles; FP16: 161, 81 and 109).  One kernel over all
// variants does not fit the instruction cache: 360 us.
#pragma once

#include "lbm_march.cuh"

namespace lbm {

template <typename T, int VAR, int NL>
__global__ void __launch_bounds__(32, march_per_sm(NL))
    march_batch_kernel(const __grid_constant__ MarchBatch p) {
    __shared__ __align__(16) T ring[kMarchSlots * 4 * kMarchStage];
    __shared__ float4 rows_y[VAR == kNone ? 1 : kMarchMaxSeg + 2 * (NL - 1)];
    // blocks that an SM is likely to hold at the same time take neighbouring walks, of
    // one instance where it is large enough
    const int per_sm = (p.blocks + p.sms - 1) / p.sms;
    const int b = blockIdx.x % p.sms * per_sm + blockIdx.x / p.sms;
    int i = 0;  // the last instance that starts at or before walk b
    for (int step = kMarchItems / 2; step > 0; step /= 2)
        if (i + step < p.count && p.item[i + step].block0 <= b) i += step;
    const MarchItem& it = p.item[i];
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (b >= p.blocks) {
        asm volatile("griddepcontrol.launch_dependents;");
        return;
    }
    const MarchWalk w = march_walk(it.grid, b - it.block0, it.ny);
    const T* src = static_cast<const T*>(it.src);
    T* dst = static_cast<T*>(it.dst);
    const size_t plane_bytes = static_cast<size_t>(it.plane) * sizeof(T);
    const int xw = w.strip * march_width(NL);
    const StepConst<F2>& k = it.k;
    if (w.fast)
        march<T, VAR, kDirichlet, NL, false, true>(src, dst, it.nx, it.ny, it.pitch, plane_bytes,
                                                   k, it.tx, it.ty, xw, w.ya, w.yb, ring, rows_y);
    else
        march<T, VAR, kDirichlet, NL, false, false>(src, dst, it.nx, it.ny, it.pitch, plane_bytes,
                                                    k, it.tx, it.ty, xw, w.ya, w.yb, ring, rows_y);
    asm volatile("griddepcontrol.launch_dependents;");
}

template <typename T, int NL>
cudaError_t launch_march_batch_t(const MarchBatch& p, int variant, cudaStream_t st, int pdl) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((p.blocks + p.sms - 1) / p.sms * p.sms);
    cfg.blockDim = dim3(32);
    cfg.dynamicSmemBytes = 0;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = pdl ? 1 : 0;
    switch (variant) {
        case kNone: return cudaLaunchKernelEx(&cfg, march_batch_kernel<T, kNone, NL>, p);
        case kTypeI: return cudaLaunchKernelEx(&cfg, march_batch_kernel<T, kTypeI, NL>, p);
        case kTypeII: return cudaLaunchKernelEx(&cfg, march_batch_kernel<T, kTypeII, NL>, p);
        case kTypeIII: return cudaLaunchKernelEx(&cfg, march_batch_kernel<T, kTypeIII, NL>, p);
        case kViscous: return cudaLaunchKernelEx(&cfg, march_batch_kernel<T, kViscous, NL>, p);
    }
    return cudaErrorInvalidValue;
}

}  // namespace lbm
