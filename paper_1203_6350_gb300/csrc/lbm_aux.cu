// Auxiliary kernels: time-0 store at equilibrium, macroscopic fields, and FP64
// diagnostics reductions.  They read the same pull-stored state as the step.
#include "lbm_read.cuh"

namespace lbm {

namespace {

template <typename CT>
__device__ __forceinline__ CT weight(int i) {
    return i == 0 ? CT(4) / CT(9) : i < 5 ? CT(1) / CT(9) : CT(1) / CT(36);
}

// f^eq_i(rho, u) - f^eq_i(rho0, u0) of the second-order D2Q9 equilibrium, from
// rho' = rho - rho0 and du = u - u0 without cancellation:
//   w_i [rho' (1 + 3 c.u + 9/2 (c.u)^2 - 3/2 u.u)
//        + rho0 (3 c.du + 9/2 (c.du)(c.u + c.u0) - 3/2 du.(u + u0))].
template <typename CT>
__device__ __forceinline__ CT feq_dev(int i, CT dr, CT ux, CT uy, CT dux, CT duy, CT rho0, CT ux0,
                                      CT uy0) {
    const CT cu = cx(i) * ux + cy(i) * uy;
    const CT cu0 = cx(i) * ux0 + cy(i) * uy0;
    const CT cdu = cx(i) * dux + cy(i) * duy;
    const CT a = CT(1) + CT(3) * cu + CT(4.5) * cu * cu - CT(1.5) * (ux * ux + uy * uy);
    const CT b = CT(3) * cdu + CT(4.5) * cdu * (cu + cu0) - CT(1.5) * (dux * (ux + ux0) + duy * (uy + uy0));
    return weight<CT>(i) * (dr * a + rho0 * b);
}

// The base state in the compute precision, converted once on the host (FP64 and the
// conversions to and from it run at 1/64 of the FP32 rate on GB300, so a kernel that
// should be bound by memory can afford a few of them per cell, not dozens).
template <typename CT>
struct BaseCt {
    CT rho0, ux0, uy0;
};
template <typename T>
BaseCt<typename Codec<T>::CT> base_ct(const BaseState& b) {
    using CT = typename Codec<T>::CT;
    return {CT(b.rho0), CT(b.ux0), CT(b.uy0)};
}

template <typename T, int BC, int I>
__device__ __forceinline__ void put_plane(const PlanePtrs<T>& dst, const Geometry& g, int x, int y,
                                          typename Codec<T>::CT v, bool interior) {
    using CT = typename Codec<T>::CT;
    int tx = x - cx(I), ty = y - cy(I);  // the cell that pulls this population reads slot (tx, ty)
    if (!interior) {
        int sx = x + cx(I), sy = y + cy(I);  // the cell whose population this cell's slot holds
        if (BC != kDirichlet) {  // periodic in y
            ty = ty < 0 ? g.ny - 1 : ty >= g.ny ? 0 : ty;
            sy = sy < 0 ? g.ny - 1 : sy >= g.ny ? 0 : sy;
        }
        if (BC == kPeriodic) {
            tx = tx < 0 ? g.nx - 1 : tx >= g.nx ? 0 : tx;
            sx = sx < 0 ? g.nx - 1 : sx >= g.nx ? 0 : sx;
        }
        if (sx < 0 || sx >= g.nx || sy < 0 || sy >= g.ny)
            dst.p[I][(long long)y * g.pitch + x] = Codec<T>::template enc<I>(CT(0));
        if (tx < 0 || tx >= g.nx || ty < 0 || ty >= g.ny) return;
    }
    dst.p[I][(long long)ty * g.pitch + tx] = Codec<T>::template enc<I>(v);
}

// Store the equilibrium populations f of cell (x, y) where the first pull reads them,
// and zero (the far field) in the cell's own slots whose source lies outside the
// lattice.  Every slot is written once.
template <typename T, int BC>
__device__ __forceinline__ void put_cell(const PlanePtrs<T>& dst, const Geometry& g, int x, int y,
                                         const typename Codec<T>::CT (&f)[9]) {
    const bool interior = x > 0 && x < g.nx - 1 && y > 0 && y < g.ny - 1;
    put_plane<T, BC, 0>(dst, g, x, y, f[0], interior);
    put_plane<T, BC, 1>(dst, g, x, y, f[1], interior);
    put_plane<T, BC, 2>(dst, g, x, y, f[2], interior);
    put_plane<T, BC, 3>(dst, g, x, y, f[3], interior);
    put_plane<T, BC, 4>(dst, g, x, y, f[4], interior);
    put_plane<T, BC, 5>(dst, g, x, y, f[5], interior);
    put_plane<T, BC, 6>(dst, g, x, y, f[6], interior);
    put_plane<T, BC, 7>(dst, g, x, y, f[7], interior);
    put_plane<T, BC, 8>(dst, g, x, y, f[8], interior);
}

// Time 0 from FP64 fields.  Each thread takes one cell, converts its three fields
// once and stores its nine populations; taking each population's source cell instead
// converted every field nine times.  4096^2 FP32, 24 + 36 B per cell: 2898 us before,
// 303 us now (3.3 TB/s; the floor at the copy rate is 150 us).
template <typename T, int BC>
__global__ void __launch_bounds__(256)
    init_kernel(PlanePtrs<T> dst, Geometry g, BaseState b, BaseCt<typename Codec<T>::CT> c0,
                const double* __restrict__ rho, const double* __restrict__ ux,
                const double* __restrict__ uy) {
    using CT = typename Codec<T>::CT;
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y * blockDim.y + threadIdx.y;
    if (x >= g.nx || y >= g.ny) return;
    const long long c = (long long)y * g.nx + x;
    const double u = ux[c], w = uy[c];
    const CT dr = CT(rho[c] - b.rho0), cu = CT(u), cw = CT(w);
    const CT du = b.ux0 == 0.0 ? cu : CT(u - b.ux0), dw = b.uy0 == 0.0 ? cw : CT(w - b.uy0);
    CT f[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) f[i] = feq_dev<CT>(i, dr, cu, cw, du, dw, c0.rho0, c0.ux0, c0.uy0);
    put_cell<T, BC>(dst, g, x, y, f);
}

// Time 0 of the acoustic pulse of Sec. 4.1 (Eqs. pulseprofile, 3:para0) without
// any input field: rho = rho0 + eps exp(-alpha |x - x_c|^2), u = u0 at every cell.
// A block takes 128 columns and `rows` <= kPulseRows rows.  SEP: the exponential as
// the product of its two factors, one FP64 exp per column and row of the block and one
// FP64 product per cell in place of an exp per population; its error of two FP64
// roundings is far below the FP32 value it is rounded to.  Otherwise (FP64 storage, or
// alpha not finite) one exp per cell.  4096^2 FP32, 36 B per cell: 8455 us with an exp
// per population, 184 us now (3.3 TB/s; floor 90 us); 8192^2 BF16 33.8 ms, now 0.45 ms.
constexpr int kPulseRows = 64;
template <typename T, int BC, bool SEP>
__global__ void __launch_bounds__(128)
    pulse_kernel(PlanePtrs<T> dst, Geometry g, BaseCt<typename Codec<T>::CT> c0, double eps,
                 double alpha, double xc, double yc, int rows) {
    using CT = typename Codec<T>::CT;
    __shared__ double along_y[SEP ? kPulseRows : 1];
    const int x = blockIdx.x * 128 + threadIdx.x;
    const int y0 = blockIdx.y * rows, y1 = min(y0 + rows, g.ny);
    const double dx = x - xc;
    double along_x = 0.0;
    if (SEP) {
        if (threadIdx.x < rows) {
            const double dy = static_cast<int>(y0 + threadIdx.x) - yc;
            along_y[threadIdx.x] = exp(-alpha * (dy * dy));
        }
        along_x = eps * exp(-alpha * (dx * dx));
        __syncthreads();
    }
    if (x >= g.nx) return;
    for (int y = y0; y < y1; ++y) {
        double dr;
        if (SEP) {
            dr = along_x * along_y[y - y0];
        } else {
            const double dy = y - yc;
            dr = eps * exp(-alpha * (dx * dx + dy * dy));
        }
        CT f[9];
#pragma unroll
        for (int i = 0; i < 9; ++i)
            f[i] = feq_dev<CT>(i, CT(dr), c0.ux0, c0.uy0, CT(0), CT(0), c0.rho0, c0.ux0, c0.uy0);
        put_cell<T, BC>(dst, g, x, y, f);
    }
}

template <typename T, int BC>
cudaError_t pulse_bc(void* dst, const Geometry& g, const BaseState& b, double eps, double alpha,
                     double xc, double yc, cudaStream_t st) {
    const PlanePtrs<T> d = plane_ptrs<T>(dst, g.plane);
    const BaseCt<typename Codec<T>::CT> c0 = base_ct<T>(b);
    // tall blocks share the exponentials, short ones fill the device on small lattices
    const int columns = (g.nx + 127) / 128;
    int rows = kPulseRows;
    while (rows > 4 && static_cast<long long>(columns) * ((g.ny + rows - 1) / rows) < 608) rows /= 2;
    const dim3 grid(columns, (g.ny + rows - 1) / rows);
    if (std::is_same<T, double>::value || !std::isfinite(alpha))
        pulse_kernel<T, BC, false><<<grid, 128, 0, st>>>(d, g, c0, eps, alpha, xc, yc, rows);
    else
        pulse_kernel<T, BC, true><<<grid, 128, 0, st>>>(d, g, c0, eps, alpha, xc, yc, rows);
    return cudaGetLastError();
}

template <typename T>
cudaError_t pulse_t(void* dst, const Geometry& g, const BaseState& b, double eps, double alpha,
                    double xc, double yc, int bc, cudaStream_t st) {
    if (bc == kPeriodic) return pulse_bc<T, kPeriodic>(dst, g, b, eps, alpha, xc, yc, st);
    if (bc == kChannel) return pulse_bc<T, kChannel>(dst, g, b, eps, alpha, xc, yc, st);
    return pulse_bc<T, kDirichlet>(dst, g, b, eps, alpha, xc, yc, st);
}

// rho', j' of the pulled populations at (x, y), summed in the compute precision.
template <typename T, int BC>
__device__ __forceinline__ void cell_moments(const PlanePtrs<T>& src, const Geometry& g, int x,
                                             int y, typename Codec<T>::CT& r,
                                             typename Codec<T>::CT& jx,
                                             typename Codec<T>::CT& jy, const LineSource& ls) {
    using CT = typename Codec<T>::CT;
    PullSites ps;
    ps.edge<BC>(x, y, g.nx, g.ny, static_cast<int>(g.pitch));
    CT v[9];
    const double src_s = (BC == kChannel && x == 0) ? line_source_scale(ls) : 0.0;
    pull_all<T, BC, true>(src, y * static_cast<int>(g.pitch) + x, ps, v, src_s, ls.e);
    CT m[9];
    moments9(v, m);
    r = m[0];
    jx = m[1];
    jy = m[2];
}

// rho', u of every cell.  States held in FP32 or less: one reciprocal per cell (two FP64
// instructions) in place of two divisions, and no conversion instructions: eleven FP64
// instructions per cell, which bound it.  4096^2 FP32, 36 + 24 B per cell: 1143 us
// with divisions, 409 us now (2.5 TB/s; floor 150 us), the same bits.
template <typename T, int BC>
__global__ void __launch_bounds__(256)
    moments_kernel(PlanePtrs<T> src, Geometry g, BaseState b, double* rho_dev, double* ux,
                   double* uy, LineSource ls) {
    using CT = typename Codec<T>::CT;
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y * blockDim.y + threadIdx.y;
    if (x >= g.nx || y >= g.ny) return;
    CT r, jx, jy;
    cell_moments<T, BC>(src, g, x, y, r, jx, jy, ls);
    const long long c = (long long)y * g.nx + x;
    const double dr = widen(r);
    if (rho_dev) rho_dev[c] = dr;
    const double rho = b.rho0 + dr;
    if constexpr (std::is_same<CT, double>::value) {
        if (ux) ux[c] = __fma_rn(b.rho0, b.ux0, jx) / rho;
        if (uy) uy[c] = __fma_rn(b.rho0, b.uy0, jy) / rho;
    } else {
        const Reciprocal inv = reciprocal(rho);
        if (ux) ux[c] = quotient(__fma_rn(b.rho0, b.ux0, widen(jx)), inv);
        if (uy) uy[c] = quotient(__fma_rn(b.rho0, b.uy0, widen(jy)), inv);
    }
}

constexpr int kDiagThreads = 256;

// First pass: block (bx, by) of a gx x gy grid takes the rows y0 + by, + gy, ...
// and the columns x0 + bx * 256 + t, + gx * 256, ... of the region, and writes
// its kDiag sums (FP64) to partial[by * gx + bx].  4096^2
// FP32, 36 B per cell: 1020 us with eleven FP64 operations and nine conversions per
// cell, 414 us now (floor 90 us).
template <typename T, int BC>
__global__ void __launch_bounds__(kDiagThreads)
    diag_partial_kernel(PlanePtrs<T> src, Geometry g, BaseState b, int x0, int y0, int x1, int y1,
                        double* partial, LineSource ls) {
    using CT = typename Codec<T>::CT;
    DiagSums sums;
    const CT rho0 = CT(b.rho0), ux0 = CT(b.ux0), uy0 = CT(b.uy0);
    for (int y = y0 + blockIdx.y; y < y1; y += gridDim.y) {
        for (int x = x0 + blockIdx.x * kDiagThreads + threadIdx.x; x < x1;
             x += gridDim.x * kDiagThreads) {
            CT r, jx, jy;
            cell_moments<T, BC>(src, g, x, y, r, jx, jy, ls);
            sums.add(r, jx, jy, rho0, ux0, uy0);
        }
    }
    write_diag_partial<kDiagThreads>(sums, b.rho0,
                                     partial + (blockIdx.y * gridDim.x + blockIdx.x) * kDiag);
}

// Second pass: one block adds the partials in a fixed order.
__global__ void __launch_bounds__(kDiagThreads)
    diag_final_kernel(const double* partial, int blocks, double* out) {
    sum_diag_partials<kDiagThreads>(partial, blocks, out);
}

template <typename T>
cudaError_t init_t(void* dst, const Geometry& g, const BaseState& b, const double* rho,
                   const double* ux, const double* uy, int bc, cudaStream_t st) {
    const dim3 block(128, 2), grid((g.nx + 127) / 128, (g.ny + 1) / 2);
    const PlanePtrs<T> d = plane_ptrs<T>(dst, g.plane);
    const BaseCt<typename Codec<T>::CT> c0 = base_ct<T>(b);
    if (bc == kPeriodic)
        init_kernel<T, kPeriodic><<<grid, block, 0, st>>>(d, g, b, c0, rho, ux, uy);
    else if (bc == kChannel)
        init_kernel<T, kChannel><<<grid, block, 0, st>>>(d, g, b, c0, rho, ux, uy);
    else
        init_kernel<T, kDirichlet><<<grid, block, 0, st>>>(d, g, b, c0, rho, ux, uy);
    return cudaGetLastError();
}

template <typename T>
cudaError_t moments_t(const void* src, const Geometry& g, const BaseState& b, int bc, double* r,
                      double* ux, double* uy, cudaStream_t st, const LineSource& ls) {
    const dim3 block(128, 2), grid((g.nx + 127) / 128, (g.ny + 1) / 2);
    const PlanePtrs<T> s = plane_ptrs<T>(const_cast<void*>(src), g.plane);
    if (bc == kPeriodic)
        moments_kernel<T, kPeriodic><<<grid, block, 0, st>>>(s, g, b, r, ux, uy, ls);
    else if (bc == kChannel)
        moments_kernel<T, kChannel><<<grid, block, 0, st>>>(s, g, b, r, ux, uy, ls);
    else
        moments_kernel<T, kDirichlet><<<grid, block, 0, st>>>(s, g, b, r, ux, uy, ls);
    return cudaGetLastError();
}

template <typename T>
cudaError_t diag_t(const void* src, const Geometry& g, const BaseState& b, int bc, int x0, int y0,
                   int x1, int y1, double* partial, double* out, cudaStream_t st,
                   const LineSource& ls) {
    const PlanePtrs<T> s = plane_ptrs<T>(const_cast<void*>(src), g.plane);
    const int w = x1 - x0, h = y1 - y0;
    const int gx = w <= 0 ? 1 : (w + kDiagThreads - 1) / kDiagThreads < 4 ? (w + kDiagThreads - 1) / kDiagThreads : 4;
    int gy = kDiagBlocks / gx;
    if (h > 0 && h < gy) gy = h;
    if (gy < 1) gy = 1;
    const dim3 grid(gx, gy);
    if (bc == kPeriodic)
        diag_partial_kernel<T, kPeriodic><<<grid, kDiagThreads, 0, st>>>(s, g, b, x0, y0, x1, y1, partial, ls);
    else if (bc == kChannel)
        diag_partial_kernel<T, kChannel><<<grid, kDiagThreads, 0, st>>>(s, g, b, x0, y0, x1, y1, partial, ls);
    else
        diag_partial_kernel<T, kDirichlet><<<grid, kDiagThreads, 0, st>>>(s, g, b, x0, y0, x1, y1, partial, ls);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    diag_final_kernel<<<1, kDiagThreads, 0, st>>>(partial, gx * gy, out);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_init(int storage, void* dst, const Geometry& g, const BaseState& b,
                        const double* rho, const double* ux, const double* uy, int bc,
                        cudaStream_t st) {
    switch (storage) {
        case kF64: return init_t<double>(dst, g, b, rho, ux, uy, bc, st);
        case kF32: return init_t<float>(dst, g, b, rho, ux, uy, bc, st);
        case kF16: return init_t<__half>(dst, g, b, rho, ux, uy, bc, st);
        case kBF16: return init_t<__nv_bfloat16>(dst, g, b, rho, ux, uy, bc, st);
    }
    return cudaErrorInvalidValue;
}

cudaError_t launch_init_pulse(int storage, void* dst, const Geometry& g, const BaseState& b,
                              double eps, double half_width, double xc, double yc, int bc,
                              cudaStream_t st) {
    const double alpha = 0.69314718055994530942 / (half_width * half_width);  // ln 2 / b^2
    switch (storage) {
        case kF64: return pulse_t<double>(dst, g, b, eps, alpha, xc, yc, bc, st);
        case kF32: return pulse_t<float>(dst, g, b, eps, alpha, xc, yc, bc, st);
        case kF16: return pulse_t<__half>(dst, g, b, eps, alpha, xc, yc, bc, st);
        case kBF16: return pulse_t<__nv_bfloat16>(dst, g, b, eps, alpha, xc, yc, bc, st);
    }
    return cudaErrorInvalidValue;
}

cudaError_t launch_moments(int storage, const void* src, const Geometry& g, const BaseState& b,
                           int bc, double* rho_dev, double* ux, double* uy, cudaStream_t st,
                           const LineSource& ls) {
    switch (storage) {
        case kF64: return moments_t<double>(src, g, b, bc, rho_dev, ux, uy, st, ls);
        case kF32: return moments_t<float>(src, g, b, bc, rho_dev, ux, uy, st, ls);
        case kF16: return moments_t<__half>(src, g, b, bc, rho_dev, ux, uy, st, ls);
        case kBF16: return moments_t<__nv_bfloat16>(src, g, b, bc, rho_dev, ux, uy, st, ls);
    }
    return cudaErrorInvalidValue;
}

cudaError_t launch_diagnostics(int storage, const void* src, const Geometry& g,
                               const BaseState& b, int bc, int x0, int y0, int x1, int y1,
                               double* partial, double* out, cudaStream_t st,
                               const LineSource& ls) {
    switch (storage) {
        case kF64: return diag_t<double>(src, g, b, bc, x0, y0, x1, y1, partial, out, st, ls);
        case kF32: return diag_t<float>(src, g, b, bc, x0, y0, x1, y1, partial, out, st, ls);
        case kF16: return diag_t<__half>(src, g, b, bc, x0, y0, x1, y1, partial, out, st, ls);
        case kBF16: return diag_t<__nv_bfloat16>(src, g, b, bc, x0, y0, x1, y1, partial, out, st, ls);
    }
    return cudaErrorInvalidValue;
}

}  // namespace lbm
