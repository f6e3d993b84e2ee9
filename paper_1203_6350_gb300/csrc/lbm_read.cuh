// Shared by the read-out kernels (macroscopic fields, diagnostics): FP64 results from
// states held in FP32 or less, with as few FP64 instructions per cell as they need.
// GB300 issues FP64 arithmetic, and the conversions to FP64, at 1/64 of the FP32 rate
// (2 per cycle and SM), so a read-out kernel is bound by them long before HBM.
#pragma once

#include "d2q9_cell.cuh"

namespace lbm {

// float -> double, exact, in integer instructions (subnormals, infinities and NaN by
// the conversion instruction).
__device__ __forceinline__ double widen(float v) {
    const unsigned u = __float_as_uint(v), t = u & 0x7fffffffu;
    if (t - 0x00800000u >= 0x7f000000u && t != 0u) return static_cast<double>(v);
    const unsigned hi = (u & 0x80000000u) | (t != 0u ? (t >> 3) + 0x38000000u : 0u);
    return __hiloint2double(static_cast<int>(hi), static_cast<int>(t << 29));
}
__device__ __forceinline__ double widen(double v) { return v; }

// The float nearest to v towards zero, in integer instructions (v in the range of reciprocal).
__device__ __forceinline__ float narrow(double v) {
    const unsigned hi = static_cast<unsigned>(__double2hiint(v));
    const unsigned t = (hi & 0x7fffffffu) - 0x38000000u;
    return __uint_as_float((hi & 0x80000000u) |
                           __funnelshift_l(static_cast<unsigned>(__double2loint(v)), t, 3));
}

// 1/rho for quotients by one rho: an approximation y with relative error below 2^-42,
// from the FP32 reciprocal of rho cut to FP32 (each 2^-23 off at most) by one Newton step
// (two FP64 instructions).  It is rho itself that is cut: an FP32 sum of its terms loses all
// digits where they cancel, near vacuum.
struct Reciprocal {
    double rho, y;
    bool ok;  // |rho| in [2^-60, 2^60), where y is that good
};
__device__ __forceinline__ Reciprocal reciprocal(double rho) {
    Reciprocal r;
    r.rho = rho;
    const unsigned t = static_cast<unsigned>(__double2hiint(rho)) & 0x7fffffffu;
    r.ok = t - 0x3c300000u < 0x07800000u;  // (false for infinities and NaN)
    const double y0 = widen(rcp_eq(r.ok ? narrow(rho) : 1.0f));
    r.y = __fma_rn(__fma_rn(-rho, y0, 1.0), y0, y0);
    return r;
}
// a / rho: the quotient a y corrected by its exact remainder (P. Markstein, IBM J. Res.
// Dev. 34, 1990), three FP64 instructions; the remainder of a quotient good to 2^-42 is
// itself good to 2^-53, so the result is the correctly rounded quotient but for ties
// within 2^-30 of an ulp.  A zero keeps its sign.  Infinities, NaN and numbers outside
// [2^-900, 2^900), whose remainder may be neither exact nor finite, and rho out of range,
// take the division.
__device__ __forceinline__ double quotient(double a, const Reciprocal& r) {
    const unsigned t = static_cast<unsigned>(__double2hiint(a)) & 0x7fffffffu;
    if (!r.ok) return a / r.rho;
    if (t - 0x07b00000u >= 0x70800000u)
        return (t | static_cast<unsigned>(__double2loint(a))) == 0u ? a * r.y : a / r.rho;
    const double q = a * r.y;
    return __fma_rn(__fma_rn(-r.rho, q, a), r.y, q);
}

// The sums of one thread of a diagnostics pass: what the six results need per cell is
// five conversions and six FP64 instructions.
struct DiagSums {
    double mass = 0, jx = 0, jy = 0, speed2 = 0, mass2 = 0;
    int bad = 0;

    // rho', j' of a cell in the compute precision.
    template <typename CT>
    __device__ __forceinline__ void add(CT r, CT mx, CT my, CT rho0, CT ux0, CT uy0) {
        // u - u0 = (j' - rho' u0) / rho, with j' = j - rho0 u0
        const CT inv = CT(1) / (rho0 + r);
        const CT dux = (mx - r * ux0) * inv;
        const CT duy = (my - r * uy0) * inv;
        const double dr = widen(r), vx = widen(dux), vy = widen(duy);
        mass += dr;
        jx += widen(mx);
        jy += widen(my);
        speed2 = __fma_rn(vx, vx, speed2);
        speed2 = __fma_rn(vy, vy, speed2);
        mass2 = __fma_rn(dr, dr, mass2);
        bad += (isfinite(r) && isfinite(dux) && isfinite(duy)) ? 0 : 1;
    }
};

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;
}

// Sum a block of THREADS threads and write its kDiag partial sums: the acoustic energy
// is that of the block's sums, c_s^2 sum rho'^2 / (2 rho0) + rho0 sum |u - u0|^2 / 2.
template <int THREADS>
__device__ __forceinline__ void write_diag_partial(const DiagSums& s, double rho0, double* out) {
    __shared__ double red[kDiag][THREADS / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const double mine[kDiag] = {s.mass, s.jx, s.jy, s.speed2, s.mass2, static_cast<double>(s.bad)};
#pragma unroll
    for (int q = 0; q < kDiag; ++q) {
        const double v = warp_sum(mine[q]);
        if (lane == 0) red[q][warp] = v;
    }
    __syncthreads();
    if (threadIdx.x < kDiag) {
        double sum = 0.0;
        for (int k = 0; k < THREADS / 32; ++k) sum += red[threadIdx.x][k];
        if (threadIdx.x == 3) {
            double mass2 = 0.0;
            for (int k = 0; k < THREADS / 32; ++k) mass2 += red[4][k];
            sum = mass2 / (6.0 * rho0) + 0.5 * rho0 * sum;
        }
        out[threadIdx.x] = sum;
    }
}

// Add `blocks` partial rows in a fixed order (one block of THREADS threads).
template <int THREADS>
__device__ __forceinline__ void sum_diag_partials(const double* partial, int blocks, double* out) {
    __shared__ double red[kDiag][THREADS / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int q = 0; q < kDiag; ++q) {
        double s = 0.0;
        for (int k = threadIdx.x; k < blocks; k += THREADS) s += partial[k * kDiag + q];
        s = warp_sum(s);
        if (lane == 0) red[q][warp] = s;
    }
    __syncthreads();
    if (threadIdx.x < kDiag) {
        double s = 0.0;
        for (int k = 0; k < THREADS / 32; ++k) s += red[threadIdx.x][k];
        out[threadIdx.x] = s;
    }
}

}  // namespace lbm
