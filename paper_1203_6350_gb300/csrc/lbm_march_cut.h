// How the marching kernels (lbm_march.cuh) cut a lattice into strips and segments.
#pragma once

#include "lbm_internal.h"

namespace lbm {

// Columns computed twice at each end of a strip of NL levels (NL - 1, kept even).
__host__ __device__ constexpr int march_halo(int nl) { return nl / 2 * 2; }
// Columns a strip stores.
__host__ __device__ constexpr int march_width(int nl) { return 64 - 2 * march_halo(nl); }
// Resident warps per SM: two levels fit 128 registers, three fit 168 (at 128 they
// spill: 188 in place of 242 GLUPS at 4096^2 FP32).
__host__ __device__ constexpr int march_per_sm(int nl) { return nl == 2 ? 16 : 12; }
constexpr int kMarchChunks = 17;              // chunks of four elements per staged plane-row
constexpr int kMarchStage = 9 * kMarchChunks; // chunks per ring slot
constexpr int kMarchRow = 4 * kMarchChunks;   // elements per staged plane-row
constexpr int kMarchSlots = 3;                // ring slots: two rows ahead of the walk (4096^2 FP32
                                              // on the prototype: 2 slots 180 GLUPS, 3 209, 4 206, 5 145)
constexpr int kMarchMaxSeg = 64;              // rows of a segment at most

// How a launch is cut (march_rectangle, march_cut): columns [s0, s1) of strips and rows
// [y0, y1) are the rectangle without checks.
struct MarchGrid {
    int strips, s0, s1, y0, y1;
    int seg, seg_gen;      // rows per segment, in the rectangle and outside it
    int n_side, n_middle;  // blocks of the side strips, and of the rows above and below
    int n_top;             // segments above the rectangle
    int blocks;
};

// The strips of a lattice and its rectangle without checks for launches of nl levels.
inline MarchGrid march_rectangle(const Geometry& g, const StepConst<F2>& k, int variant, int nl) {
    MarchGrid m{};
    const int width = march_width(nl), halo = march_halo(nl);
    m.strips = (g.nx + width - 1) / width;
    // strips whose staged columns lie in the lattice and whose cells lie in the bulk
    const bool layer = variant != kNone;
    auto fast = [&](int s) {
        const int x = s * width;
        return x - 4 >= 0 && x - 4 + kMarchRow <= g.nx &&
               (!layer || (x - halo >= k.bulk_x0 && x - halo + 64 <= k.bulk_x1));
    };
    m.s0 = 0;
    while (m.s0 < m.strips && !fast(m.s0)) ++m.s0;
    m.s1 = m.s0;
    while (m.s1 < m.strips && fast(m.s1)) ++m.s1;
    // rows whose segments pull rows of the lattice and collide rows of the bulk
    m.y0 = layer && k.bulk_y0 - 1 > 0 ? k.bulk_y0 - 1 + nl : nl;
    m.y1 = (layer && k.bulk_y1 + 1 < g.ny ? k.bulk_y1 + 1 : g.ny) - nl;
    if (m.y1 <= m.y0 || m.s1 == m.s0) {
        m.s0 = m.s1 = m.strips;
        m.y0 = m.y1 = g.ny;
    }
    return m;
}

// Cells of its strips (whole ones, so the last strip's idle lanes count), and of the rectangle.
inline long long march_cells(const MarchGrid& m, int ny, int nl) {
    return static_cast<long long>(m.strips) * march_width(nl) * ny;
}
inline long long march_fast_cells(const MarchGrid& m, int nl) {
    return static_cast<long long>(m.s1 - m.s0) * march_width(nl) * (m.y1 - m.y0);
}

// Cut it into segments of seg rows, 5/8 as long outside the rectangle, where a row
// costs about 1.5 times as much.  Returns the blocks.
inline int march_cut(MarchGrid& m, int ny, int seg) {
    const long long ns = m.s0 + m.strips - m.s1, nm = m.s1 - m.s0;
    const auto segs = [](int n, int s) { return (n + s - 1) / s; };
    m.seg = seg;
    m.seg_gen = seg * 5 / 8;
    m.n_side = static_cast<int>(ns * segs(ny, m.seg_gen));
    m.n_top = nm ? segs(m.y0, m.seg_gen) : 0;
    m.n_middle = nm ? static_cast<int>(nm * (m.n_top + segs(ny - m.y1, m.seg_gen))) : 0;
    m.blocks = static_cast<int>(m.n_side + m.n_middle + nm * segs(m.y1 - m.y0, seg));
    return m.blocks;
}

// The shortest segments whose blocks (blocks(seg) of them) fit the device's slots k
// times, for the smallest k that keeps them within kMarchMaxSeg rows: the last wave is
// then nearly full, and few rows are computed twice.  2048^2 FP32, three levels: 189 GLUPS
// with segments of 16 rows, 219 fitted (the two-step tiles: 129).
template <typename F>
inline int march_segment(int nl, int sms, F blocks) {
    const long long slots = static_cast<long long>(sms) * march_per_sm(nl);
    for (long long waves = 1;; ++waves)
        for (int seg = 4; seg <= kMarchMaxSeg; ++seg)
            if (blocks(seg) <= waves * slots) return seg;
}

// Many lattices in one launch (lbm_march_batch.cuh): an instance, and the launch.
struct MarchItem {
    StepConst<F2> k;
    const void* src;
    void* dst;
    const AxisCoef<float>*tx, *ty;
    int nx, ny, pitch;
    unsigned plane;
    int block0;  // its first block
    MarchGrid grid;
};
constexpr int kMarchItems = 32;
struct MarchBatch {
    int count, blocks, sms;
    MarchItem item[kMarchItems];
};
static_assert(sizeof(MarchBatch) <= 32764, "the parameters of one launch");
cudaError_t launch_march_batch_f32(const MarchBatch& p, int variant, cudaStream_t st, int pdl);
cudaError_t launch_march_batch_f16(const MarchBatch& p, int variant, cudaStream_t st, int pdl);
cudaError_t launch_march_batch_bf16(const MarchBatch& p, int variant, cudaStream_t st, int pdl);

}  // namespace lbm
