// Several time steps per launch on lattices too small to fill the GPU.
//
// A step of such a lattice costs little more than its launch (1.5 us of the 1.7 us of
// a 100^2 step), so a block takes several steps on a tile: level 1 pulls time t from
// memory and collides the tile widened by levels - 1 cells on every side into
// shared memory; each further level pulls the one before it from there, on a region
// one cell narrower per side, and the last stores the tile.  The cells around the
// tile are computed by several blocks, which is free while the GPU is not full.
// Levels are held in FP32; for 16-bit storage each is rounded to the format, as a
// launch per step rounds it, so the result does not depend on the grouping.
//
// What bounds it: the latency of a level (about 0.7 us: the chain of one collision, its
// 15 + 9 shared-memory accesses and the block's barrier, at one or two warps per
// scheduler, 24 % of issue slots busy).  Measured, us per step with a launch per step and
// with tiles: FP32 64^2 1.66 / 0.87, 100^2 1.71 / 0.89, 200^2 1.61 / 1.31, 300^2 1.97 /
// 2.37; FP16 200^2 2.08 / 1.38; 800 x 200 channel 2.63 / 2.85.
#pragma once

#include "lbm_march.cuh"
#include "lbm_step_tb.cuh"

namespace lbm {

constexpr int kTileThreads = 512;  // at most
constexpr int kTilePad = 4;  // elements in front of and behind the planes of a level

// Region and tile of a launch: the region is rw = 32 or 64 columns wide (launched with 32),
// starts hx columns left of the tile (even, so that pairs stay aligned) and levels - 1 rows
// above it.
struct TileShape {
    int rw, rh, hx;  // region, halo along x
    int w, h;        // tile
    int levels;
};
inline TileShape tile_shape(int h, int levels) {
    return TileShape{kTileRegion, h + 2 * (levels - 1), tile_halo(levels), tile_width(levels), h,
                     levels};
}
inline size_t tile_smem_bytes(const TileShape& s) {
    return 2 * sizeof(float) * (9 * s.rw * s.rh + 2 * kTilePad);
}

// A warp owns two rows of 16 pairs.  A thread keeps its K pairs through all levels (one: the
// regions are at most 22 rows high), so what depends on their place only -- the boundary, the
// layer's coefficients -- is worked out once.  Written out for one pair and a fixed region
// width the kernels compile to other schedules: up to 14 % faster without a layer, up to 9 %
// slower with one (FP32 periodic type III at 100^2-226^2).
template <typename T, int VAR, int BC, int K = 1>
__global__ void __launch_bounds__(kTileThreads, 1)
    tile_kernel(const T* __restrict__ src, T* __restrict__ dst, int nx, int ny, int pitch,
                unsigned plane, StepConst<F2> k, const AxisCoef<float>* __restrict__ tx,
                const AxisCoef<float>* __restrict__ ty, TileShape t, LineSource ls) {
    extern __shared__ __align__(16) float tile_raw[];
    constexpr bool UB = UnbiasedScale<T>::value;
    const unsigned rw = t.rw, rplane = t.rw * t.rh;
    const int lane = threadIdx.x & 31, warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0);
    const int shift = t.rw == 64 ? 5 : 4, rows_per_warp = 32 >> shift;
    const int c = 2 * (lane & ((1 << shift) - 1));
    const int x = blockIdx.x * t.w - t.hx + c;
    float* const level[2] = {tile_raw + kTilePad, tile_raw + 9 * rplane + 3 * kTilePad};
    const bool in_a = x >= 0 && x < nx, in_b = x + 1 >= 0 && x + 1 < nx;
    const int ca = BC == kPeriodic ? wrapped(x, nx) : min(max(x, 0), nx - 1);
    const int cb = BC == kPeriodic ? wrapped(x + 1, nx) : min(max(x + 1, 0), nx - 1);
    int row[K], y[K];  // row of the region, row of the lattice
    F2 chi[K], rn[K], rm[K];
    bool layer[K];
#pragma unroll
    for (int i = 0; i < K; ++i) {
        row[i] = (warp + i * static_cast<int>(blockDim.x >> 5)) * rows_per_warp + (lane >> shift);
        y[i] = blockIdx.y * t.h - (t.levels - 1) + row[i];
        layer[i] = false;
        if constexpr (VAR != kNone) {
            const int cy = BC == kDirichlet ? min(max(y[i], 0), ny - 1) : wrapped(y[i], ny);
            const AxisCoef<float> a0 = load_coef(tx, ca), a1 = load_coef(tx, cb);
            const AxisCoef<float> ay = load_coef(ty, cy);
            chi[i] = f2(fmaxf(a0.chi, ay.chi), fmaxf(a1.chi, ay.chi));
            rn[i] = f2(fminf(a0.rn, ay.rn), fminf(a1.rn, ay.rn));
            rm[i] = f2(fminf(a0.rm, ay.rm), fminf(a1.rm, ay.rm));
            layer[i] = __any_sync(0xffffffffu, f2_lo(chi[i]) > 0.0f || f2_hi(chi[i]) > 0.0f);
        }
    }
    asm volatile("griddepcontrol.wait;" ::: "memory");
    for (int l = 0; l < t.levels; ++l) {
        const float* from = level[(l + 1) & 1];
        float* to = level[l & 1];
        const float* src_pop = BC == kChannel ? ls.pop + 9 * (ls.t_off + l) : nullptr;
#pragma unroll
        for (int i = 0; i < K; ++i) {
            // the level is complete on rows l .. rh - l - 1; pairs outside the columns
            // l .. rw - l - 1 hold values that nothing reads
            const bool own = row[i] >= l && row[i] < t.rh - l;
            if (!__any_sync(0xffffffffu, own)) continue;
            F2 v[9];
            if (l == 0) {
                const int yy = y[i];
                if (x > 0 && x + 2 < nx && yy > 0 && yy + 1 < ny)
                    pull_pair_interior<T>(src, plane, static_cast<unsigned>(pitch),
                                          static_cast<unsigned>(yy * pitch + x), v);
                else
                    pull_lanes<T, BC>(src, plane, pitch, ca, cb,
                                      BC == kDirichlet ? min(max(yy, 0), ny - 1) : wrapped(yy, ny),
                                      nx, ny, v, src_pop);
            } else {
                const int r = own ? row[i] : l;  // (a row that is there)
                pull_pair_interior<float, true>(from, rplane, rw, r * rw + c, v);
                if (BC == kChannel) {
                    if (x == 0) {  // the source column's populations at this level
                        v[1] = f2(src_pop[1], f2_hi(v[1]));
                        v[5] = f2(src_pop[5], f2_hi(v[5]));
                        v[8] = f2(src_pop[8], f2_hi(v[8]));
                    }
                    if (x == nx - 1 || x + 1 == nx - 1) {  // outflow: the last column's own values
                        const float* s = from + r * rw + c + (nx - 1 - x);
                        const float o3 = s[3 * rplane], o6 = *(s + 6 * rplane - rw),
                                    o7 = s[7 * rplane + rw];
                        const bool lo = x == nx - 1;
                        v[3] = f2(lo ? o3 : f2_lo(v[3]), lo ? f2_hi(v[3]) : o3);
                        v[6] = f2(lo ? o6 : f2_lo(v[6]), lo ? f2_hi(v[6]) : o6);
                        v[7] = f2(lo ? o7 : f2_lo(v[7]), lo ? f2_hi(v[7]) : o7);
                    }
                }
            }
            if (VAR == kNone || !layer[i]) {
                collide_bulk<F2, UB>(v, k);
            } else {
                if constexpr (VAR == kViscous)
                    collide_viscous<F2, UB>(v, chi[i], k);
                else if constexpr (VAR != kNone)
                    collide_layer<F2, VAR, UB>(v, chi[i], rn[i], rm[i], k);
            }
            if (!own) continue;
            if (l + 1 < t.levels) {
                if (BC == kDirichlet) {  // outside: the wall value 0
                    const bool row_in = y[i] >= 0 && y[i] < ny;
                    const bool ka = row_in && in_a, kb = row_in && in_b;
                    if (!(ka && kb)) {
#pragma unroll
                        for (int q = 0; q < 9; ++q)
                            v[q] = f2(ka ? f2_lo(v[q]) : 0.0f, kb ? f2_hi(v[q]) : 0.0f);
                    }
                }
                if constexpr (sizeof(T) == 2) {
                    for_planes([&](auto plane_index) {
                        constexpr int q = decltype(plane_index)::value;
                        v[q] = through_storage<T, q>(v[q]);
                    });
                }
                store_pair<float>(to, rplane, row[i] * rw + c, v);
            } else if (c >= t.hx && c < t.hx + t.w && in_a && y[i] < ny) {
                const unsigned o = static_cast<unsigned>(y[i] * pitch + x);
                if (in_b)
                    store_pair<T>(dst, plane, o, v);
                else
                    store_lo<T>(dst, plane, o, v);
            }
        }
        __syncthreads();
    }
    asm volatile("griddepcontrol.launch_dependents;");
}

// f(kernel) for the kernel of a variant and boundary; cudaErrorInvalidValue if there is none.
template <typename T, typename F>
cudaError_t with_tile_kernel(int variant, int bc, F f) {
#define LBM_TILE_CASE(V)                                             \
    if (variant == V && bc == kDirichlet) return f(tile_kernel<T, V, kDirichlet>); \
    if (variant == V && bc == kPeriodic) return f(tile_kernel<T, V, kPeriodic>);   \
    if (variant == V && bc == kChannel) return f(tile_kernel<T, V, kChannel>);
    LBM_TILE_CASE(kNone)
    LBM_TILE_CASE(kTypeI)
    LBM_TILE_CASE(kTypeII)
    LBM_TILE_CASE(kTypeIII)
    LBM_TILE_CASE(kViscous)
#undef LBM_TILE_CASE
    return cudaErrorInvalidValue;
}

// Raise the kernel's dynamic shared-memory limit (outside any stream capture, before its
// first launch).  The limit is the kernel's, not the handle's: it is the same for
// every tile, so that a handle with small tiles does not lower it for one with large.
constexpr int kTileSmem = 96 * 1024;
template <typename T>
cudaError_t prepare_tile_t(int variant, int bc, const TileShape& t) {
    if (tile_smem_bytes(t) > kTileSmem) return cudaErrorInvalidValue;
    return with_tile_kernel<T>(variant, bc, [](auto kernel) {
        return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    kTileSmem);
    });
}

// Advance t.levels >= 2 steps.  cudaErrorInvalidValue when the nine planes exceed
// 32-bit element offsets.
template <typename T>
cudaError_t launch_tile_t(const void* src, void* dst, const Geometry& g, const StepConst<F2>& k,
                          const AxisCoef<float>* tx, const AxisCoef<float>* ty, int variant, int bc,
                          const TileShape& t, cudaStream_t st, int pdl, const LineSource& ls) {
    if (9 * g.plane >= (1ll << 32)) return cudaErrorInvalidValue;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((g.nx + t.w - 1) / t.w, (g.ny + t.h - 1) / t.h);
    const int warps = (t.rh + 1) / 2;
    if (32 * warps > kTileThreads) return cudaErrorInvalidValue;
    cfg.blockDim = dim3(32 * warps);
    cfg.dynamicSmemBytes = tile_smem_bytes(t);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = pdl ? 1 : 0;
    const T* s = static_cast<const T*>(src);
    T* d = static_cast<T*>(dst);
    const int pitch = static_cast<int>(g.pitch);
    const unsigned plane = static_cast<unsigned>(g.plane);
    const auto launch = [&](auto kernel) {
        return cudaLaunchKernelEx(&cfg, kernel, s, d, g.nx, g.ny, pitch, plane, k, tx, ty, t, ls);
    };
    return with_tile_kernel<T>(variant, bc, launch);
}

}  // namespace lbm
