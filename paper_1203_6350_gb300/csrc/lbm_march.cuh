// Several time steps per launch by warps that march down the lattice
// (temporal blocking in registers) on the two-cells-per-thread arithmetic.
//
// A warp owns a strip of columns and a segment of rows.  Lane l holds the pair
// of cells (x, x + 1), x = strip start - kMarchHalo + 2 l, and the warp walks
// down its rows one at a time: level 1 collides row r of time t, level 2 then
// has the rows r - 2, r - 1, r of time t + 1 that it needs to collide row
// r - 1, and so on to level NL, which stores row r - NL + 1 of time t + NL.
//
//  - What a level still needs of the rows above stays in registers, nine pairs
//    between two levels: the planes pulled from the row above are kept for two
//    rows, those of the row itself for one, those of the row below for none.
//  - A plane that moves along x takes the one value that lies in the
//    neighbouring lane by a shuffle.  So the time levels cost no shared memory
//    and no barrier: 6 shuffles per pair and level in place of the 9 stores and
//    15 loads of a tile in shared memory.
//  - Level 1's input is copied ahead of its use by cp.async into a ring of
//    kMarchSlots rows in shared memory, private to the warp.  A ring slot holds
//    the nine plane-rows that one row of the walk pulls (each plane from its own
//    source row), in chunks of four elements from four columns left of the
//    strip; chunks outside the lattice are filled with zero, the Dirichlet
//    far-field deviation.
//  - Every level but the first loses one cell at each end of the warp's 64
//    columns, and every level one row at each end of its segment; those are
//    computed twice.
//
// The blocks (one warp each, so that the walk's control flow and the step's
// constants are uniform and the latter stay in uniform registers) are numbered so that
// the slower walks come first: the side strips, then the rows above and below
// the rectangle of the rest.  In that rectangle no cell touches the lattice's
// edge or the layer (chi = 0) and nothing is checked.
//
// What bounds it: HBM and the FMA pipe together (three levels at 4096^2: DRAM at 0.84 of
// its measured rate, the FMA pipe 65 % and the issue slots 59 % busy; a packed FMA takes
// the pipe for two cycles, so 95 of them per pair and level cap the chip at 391 GLUPS),
// and below 1.5 million cells the four rows that each short segment walks twice.
// It moves 24 B (FP32, three levels) or 18 B (16-bit, two) per cell-step to and from
// HBM.  Measured against the kernels it replaces, GLUPS, FP32 1024^2 / 2048^2 /
// 4096^2 / 8192^2: 146 / 129 / 148 / 150 before, 153 / 219 / 242 / 259 with it; BF16
// 4096^2: 183 before, 238 with it.
#pragma once

#include "lbm_march_cut.h"
#include "lbm_step2.cuh"

namespace lbm {

// What the next level needs of the rows that one level has produced.
struct MarchLine {
    F2 same[3];    // f_0, f_1, f_3 of the last row
    F2 above1[3];  // f_2, f_5, f_6 of the last row
    F2 above2[3];  // f_2, f_5, f_6 of the row before it
};

// The pair whose sources lie one column to the left, and to the right.
__device__ __forceinline__ F2 from_left(F2 p) {
    return f2(__shfl_up_sync(0xffffffffu, f2_hi(p), 1), f2_lo(p));
}
__device__ __forceinline__ F2 from_right(F2 p) {
    return f2(f2_hi(p), __shfl_down_sync(0xffffffffu, f2_lo(p), 1));
}

// A value rounded to the storage format, as a store and the next step's load do.
template <typename T, int I>
__device__ __forceinline__ F2 through_storage(F2 v) {
    return PairCodec<T>::template dec2<I>(PairCodec<T>::template enc2<I>(v));
}

// The periodic image of coordinate c in [0, n).
__device__ __forceinline__ int wrapped(int c, int n) {
    if (static_cast<unsigned>(c) < static_cast<unsigned>(n)) return c;
    c %= n;
    return c < 0 ? c + n : c;
}

// The row offset of the source of plane p: -c_y.
__device__ __forceinline__ int source_row(int p) {
    return (p == 2 || p == 5 || p == 6) ? -1 : (p == 4 || p == 7 || p == 8) ? 1 : 0;
}

template <int N>
using Plane = std::integral_constant<int, N>;
template <typename F>
__device__ __forceinline__ void for_planes(F f) {
    f(Plane<0>{}), f(Plane<1>{}), f(Plane<2>{}), f(Plane<3>{}), f(Plane<4>{}), f(Plane<5>{}),
        f(Plane<6>{}), f(Plane<7>{}), f(Plane<8>{});
}

// One warp's walk over the rows [ya, yb) of the strip at column xw.  FAST: every
// cell it touches is inside the lattice and in the bulk.  RND: each level is
// rounded to the storage format, as one step per launch rounds it; otherwise
// only the last.
template <typename T, int VAR, int BC, int NL, bool RND, bool FAST>
__device__ __forceinline__ void march(const T* __restrict__ src, T* __restrict__ dst, int nx,
                                      int ny, int pitch, size_t plane_bytes,
                                      const StepConst<F2>& k,
                                      const AxisCoef<float>* __restrict__ tx,
                                      const AxisCoef<float>* __restrict__ ty, int xw, int ya,
                                      int yb, T* ring, float4* rows_y) {
    using PC = PairCodec<T>;
    using Raw2 = typename PC::Raw2;
    constexpr bool UB = UnbiasedScale<T>::value;
    constexpr int ES = sizeof(T);
    constexpr int kPer = (kMarchStage + 31) / 32;  // chunks a lane copies per row
    constexpr int kMarchHalo = march_halo(NL);
    const int lane = threadIdx.x;
    const int x = xw - kMarchHalo + 2 * lane;
    const int xs = xw - 4;  // column of a slot's first element
    const unsigned pitch_b = static_cast<unsigned>(pitch) * ES;
    const int r0 = ya - (NL - 1), rows = yb - ya + 2 * (NL - 1);

    const bool in_a = x >= 0 && x < nx, in_b = x + 1 >= 0 && x + 1 < nx;
    // lanes outside the lattice compute on a clamped (or, periodic, the wrapped) cell
    const bool edge = !FAST && BC == kDirichlet && (xs < 0 || xs + kMarchRow > nx);
    F2 chi_x, rn_x, rm_x;
    if constexpr (!FAST && VAR != kNone) {
        const int ca = BC == kPeriodic ? wrapped(x, nx) : min(max(x, 0), nx - 1);
        const int cb = BC == kPeriodic ? wrapped(x + 1, nx) : min(max(x + 1, 0), nx - 1);
        const AxisCoef<float> a0 = load_coef(tx, ca), a1 = load_coef(tx, cb);
        chi_x = f2(a0.chi, a1.chi);
        rn_x = f2(a0.rn, a1.rn);
        rm_x = f2(a0.rm, a1.rm);
        for (int i = lane; i < rows; i += 32) {
            const int y = BC == kPeriodic ? wrapped(r0 + i, ny) : min(max(r0 + i, 0), ny - 1);
            rows_y[i] = __ldg(reinterpret_cast<const float4*>(ty) + y);
        }
    }

    // ---- staging of level 1's input ----
    const unsigned ring_addr = static_cast<unsigned>(__cvta_generic_to_shared(ring));
    const char* from[kPer];  // FAST: the lane's chunks of the next row; else of row 0
    int column[kPer];        // periodic: their columns
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
        const int q = i * 32 + lane, p = q / kMarchChunks;
        int c = xs + 4 * (q % kMarchChunks);
        if (!FAST && BC == kPeriodic) column[i] = c = wrapped(c, nx);
        from[i] = reinterpret_cast<const char*>(src) + p * plane_bytes + c * ES;
        if (FAST) from[i] += static_cast<size_t>(r0 + source_row(p)) * pitch_b;
    }
    int staged = 0;
    unsigned slot_in = 0;
    auto stage_row = [&]() {
#pragma unroll
        for (int i = 0; i < kPer; ++i) {
            const int q = i * 32 + lane;
            const unsigned to = ring_addr + (slot_in * kMarchStage + q) * (4 * ES);
            if (i + 1 == kPer && q >= kMarchStage) break;
            if constexpr (FAST) {
                asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(to), "l"(from[i]),
                             "n"(4 * ES)
                             : "memory");
                from[i] += pitch_b;
            } else {
                const int p = q / kMarchChunks;
                int y = r0 + staged + source_row(p);
                if constexpr (BC == kPeriodic) {
                    y = wrapped(y, ny);
                    const int cw = column[i];
                    const char* row = from[i] + static_cast<size_t>(y) * pitch_b;
                    // (16-bit rows are a multiple of 4 long, so every chunk is whole and aligned)
                    if (ES == 2 || (cw + 4 <= nx && (cw & 3) == 0)) {
                        asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(to),
                                     "l"(row), "n"(4 * ES)
                                     : "memory");
                    } else {  // a chunk across the seam, or shifted by a row length not a multiple of 4
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            const int past = cw + e >= nx ? e - nx : e;  // elements from the chunk's start
                            asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(to + e * ES),
                                         "l"(row + past * ES)
                                         : "memory");
                        }
                    }
                } else {
                    const int c = xs + 4 * (q - p * kMarchChunks);
                    const bool ok = c >= 0 && c < nx && y >= 0 && y < ny;
                    const char* row = from[i] + static_cast<long long>(y) * pitch_b;
                    asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;" ::"r"(to),
                                 "l"(ok ? row : reinterpret_cast<const char*>(src)), "n"(4 * ES),
                                 "r"(ok ? 4 * ES : 0)
                                 : "memory");
                }
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
        ++staged;
        slot_in = slot_in + 1 == kMarchSlots ? 0 : slot_in + 1;
    };

    MarchLine line[NL - 1];
#pragma unroll
    for (int i = 0; i < kMarchSlots - 1; ++i) stage_row();  // rows >= 2 NL - 1 > kMarchSlots - 1
    unsigned slot = 0;
    // Unrolled by two, the rectangle's walk keeps its lines without register moves
    // (2 % at 4096^2).  Not with 16-bit storage: there the code generator then fuses
    // other products into sums, and a store in ten thousand rounds the other way.
    constexpr int kUnroll = FAST && sizeof(T) == 4 ? 2 : 1;
#pragma unroll kUnroll
    for (int j = 0; j < rows; ++j) {
        // all groups but the newest kMarchSlots - 2 are done: row j is in its slot
        asm volatile("cp.async.wait_group %0;" ::"n"(kMarchSlots - 2) : "memory");
        __syncwarp();
        F2 v[9];
        {
            constexpr int P = kMarchRow;
            const T* s = ring + slot * (4 * kMarchStage) + (4 - kMarchHalo) + 2 * lane;
            v[0] = PC::template dec2<0>(ld_pair<T, true>(s));
            v[1] = PC::template dec11<1>(s[P - 1], s[P]);
            v[2] = PC::template dec2<2>(ld_pair<T, true>(s + 2 * P));
            v[3] = PC::template dec11<3>(s[3 * P + 1], s[3 * P + 2]);
            v[4] = PC::template dec2<4>(ld_pair<T, true>(s + 4 * P));
            v[5] = PC::template dec11<5>(s[5 * P - 1], s[5 * P]);
            v[6] = PC::template dec11<6>(s[6 * P + 1], s[6 * P + 2]);
            v[7] = PC::template dec11<7>(s[7 * P + 1], s[7 * P + 2]);
            v[8] = PC::template dec11<8>(s[8 * P - 1], s[8 * P]);
        }
        slot = slot + 1 == kMarchSlots ? 0 : slot + 1;
        __syncwarp();  // the slot filled next was read one row ago by every lane
        if (staged < rows)
            stage_row();
        else
            asm volatile("cp.async.commit_group;" ::: "memory");
        if (edge) {  // the last chunk of a row may reach into its padding
            const bool in_c = x + 2 < nx;
            auto keep = [](F2 p, bool a, bool b) {
                return f2(a ? f2_lo(p) : 0.0f, b ? f2_hi(p) : 0.0f);
            };
            v[0] = keep(v[0], in_a, in_b);
            v[2] = keep(v[2], in_a, in_b);
            v[4] = keep(v[4], in_a, in_b);
            v[1] = keep(v[1], x - 1 < nx, in_a);
            v[5] = keep(v[5], x - 1 < nx, in_a);
            v[8] = keep(v[8], x - 1 < nx, in_a);
            v[3] = keep(v[3], in_b, in_c);
            v[6] = keep(v[6], in_b, in_c);
            v[7] = keep(v[7], in_b, in_c);
        }
#pragma unroll
        for (int l = 0; l < NL; ++l) {
            if (l > 0) {  // v: row r0 + j - l + 1, as the level below has just produced it
                MarchLine& m = line[l - 1];
                const F2 w0 = v[0], w1 = v[1], w2 = v[2], w3 = v[3], w5 = v[5], w6 = v[6];
                v[0] = m.same[0];
                v[1] = m.same[1];
                v[3] = m.same[2];
                v[2] = m.above2[0];
                v[5] = m.above2[1];
                v[6] = m.above2[2];
                m.above2[0] = m.above1[0];
                m.above2[1] = m.above1[1];
                m.above2[2] = m.above1[2];
                m.same[0] = w0;
                m.same[1] = w1;
                m.same[2] = w3;
                m.above1[0] = w2;
                m.above1[1] = w5;
                m.above1[2] = w6;
                if (j < 2 * l) break;  // this level's first row is not complete yet
                v[1] = from_left(v[1]);
                v[5] = from_left(v[5]);
                v[8] = from_left(v[8]);
                v[3] = from_right(v[3]);
                v[6] = from_right(v[6]);
                v[7] = from_right(v[7]);
            }
            const int y = r0 + j - l;
            if constexpr (FAST || VAR == kNone) {
                collide_bulk<F2, UB>(v, k);
            } else {  // where chi = 0 this is the bulk collision bit for bit
                const float4 cy = rows_y[j - l];
                const F2 chi = f2(fmaxf(f2_lo(chi_x), cy.x), fmaxf(f2_hi(chi_x), cy.x));
                if constexpr (VAR == kViscous)
                    collide_viscous<F2, UB>(v, chi, k);
                else
                    collide_layer<F2, VAR, UB>(
                        v, chi, f2(fminf(f2_lo(rn_x), cy.y), fminf(f2_hi(rn_x), cy.y)),
                        f2(fminf(f2_lo(rm_x), cy.z), fminf(f2_hi(rm_x), cy.z)), k);
            }
            if (l + 1 < NL) {
                if constexpr (!FAST && BC == kDirichlet) {  // cells outside hold the wall value 0
                    if (edge || y < 0 || y >= ny) {
                        const bool row_in = y >= 0 && y < ny;
                        const bool ka = row_in && in_a, kb = row_in && in_b;
#pragma unroll
                        for (int i = 0; i < 9; ++i)
                            v[i] = f2(ka ? f2_lo(v[i]) : 0.0f, kb ? f2_hi(v[i]) : 0.0f);
                    }
                }
                if constexpr (RND)
                    for_planes([&](auto plane_index) {
                        constexpr int i = decltype(plane_index)::value;
                        v[i] = through_storage<T, i>(v[i]);
                    });
            } else if (lane >= kMarchHalo / 2 && lane < 32 - kMarchHalo / 2 && (FAST || in_a)) {
                char* o = reinterpret_cast<char*>(dst) +
                          (static_cast<size_t>(static_cast<unsigned>(y)) * pitch_b +
                           static_cast<unsigned>(x) * ES);
                if (FAST || in_b)
                    for_planes([&](auto plane_index) {
                        constexpr int i = decltype(plane_index)::value;
                        *reinterpret_cast<Raw2*>(o + i * plane_bytes) =
                            PC::template enc2<i>(v[i]);
                    });
                else  // the last column of an odd-width lattice
                    for_planes([&](auto plane_index) {
                        constexpr int i = decltype(plane_index)::value;
                        *reinterpret_cast<T*>(o + i * plane_bytes) = PC::template enc_lo<i>(v[i]);
                    });
            }
        }
    }
}

// Block b of a launch: its strip, its rows, and whether it lies in the rectangle.
struct MarchWalk {
    int strip, ya, yb;
    bool fast;
};
__device__ __forceinline__ MarchWalk march_walk(const MarchGrid& g, int b, int ny) {
    const int nm = g.s1 - g.s0;
    MarchWalk w;
    if (b >= g.n_side + g.n_middle) {
        b -= g.n_side + g.n_middle;
        w.strip = g.s0 + b % nm;
        w.ya = g.y0 + b / nm * g.seg;
        w.yb = min(w.ya + g.seg, g.y1);
        w.fast = true;
        return w;
    }
    int end = ny;
    if (b < g.n_side) {
        const int ns = g.s0 + g.strips - g.s1;
        w.strip = b % ns;
        if (w.strip >= g.s0) w.strip += nm;
        w.ya = b / ns * g.seg_gen;
    } else {
        b -= g.n_side;
        const int q = b / nm;
        w.strip = g.s0 + b % nm;
        w.ya = q < g.n_top ? q * g.seg_gen : g.y1 + (q - g.n_top) * g.seg_gen;
        if (q < g.n_top) end = g.y0;
    }
    w.yb = min(w.ya + g.seg_gen, end);
    w.fast = false;
    return w;
}

template <typename T, int VAR, int BC, int NL, bool RND>
__global__ void __launch_bounds__(32, march_per_sm(NL))
    march_kernel(const T* __restrict__ src, T* __restrict__ dst, int nx, int ny, int pitch,
                 unsigned plane, StepConst<F2> k, const AxisCoef<float>* __restrict__ tx,
                 const AxisCoef<float>* __restrict__ ty, MarchGrid g) {
    __shared__ __align__(16) T ring[kMarchSlots * 4 * kMarchStage];
    __shared__ float4 rows_y[VAR == kNone ? 1 : kMarchMaxSeg + 2 * (NL - 1)];
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const size_t plane_bytes = static_cast<size_t>(plane) * sizeof(T);
    const MarchWalk w = march_walk(g, blockIdx.x, ny);
    if (w.fast)
        march<T, VAR, BC, NL, RND, true>(src, dst, nx, ny, pitch, plane_bytes, k, tx, ty,
                                         w.strip * march_width(NL), w.ya, w.yb, ring, rows_y);
    else
        march<T, VAR, BC, NL, RND, false>(src, dst, nx, ny, pitch, plane_bytes, k, tx, ty,
                                          w.strip * march_width(NL), w.ya, w.yb, ring, rows_y);
    asm volatile("griddepcontrol.launch_dependents;");
}

// Advance NL steps: src holds time t, dst receives t + NL; pdl as for the one-step
// kernels.  cudaErrorInvalidValue when the nine planes exceed 32-bit offsets, and for periodic
// rows that the staging does not take: shorter than a chunk, or 16-bit and no multiple of it.
template <typename T, int BC, int NL, bool RND>
cudaError_t launch_march_t(const void* src, void* dst, const Geometry& g, const StepConst<F2>& k,
                           const AxisCoef<float>* tx, const AxisCoef<float>* ty, int variant,
                           int seg, cudaStream_t st, int pdl) {
    if (9 * g.plane >= (1ll << 32)) return cudaErrorInvalidValue;
    if (BC == kPeriodic && (g.nx < 4 || (sizeof(T) == 2 && g.nx % 4 != 0)))
        return cudaErrorInvalidValue;
    MarchGrid m = march_rectangle(g, k, variant, NL);
    march_cut(m, g.ny, seg);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(m.blocks);
    cfg.blockDim = dim3(32);
    cfg.dynamicSmemBytes = 0;
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
#define LBM_MARCH_CASE(V)                                                                       \
    if (variant == V)                                                                           \
        return cudaLaunchKernelEx(&cfg, march_kernel<T, V, BC, NL, RND>, s, d, g.nx, g.ny, pitch, \
                                  plane, k, tx, ty, m);
    LBM_MARCH_CASE(kNone)
    LBM_MARCH_CASE(kTypeI)
    LBM_MARCH_CASE(kTypeII)
    LBM_MARCH_CASE(kTypeIII)
    LBM_MARCH_CASE(kViscous)
#undef LBM_MARCH_CASE
    return cudaErrorInvalidValue;
}

}  // namespace lbm
