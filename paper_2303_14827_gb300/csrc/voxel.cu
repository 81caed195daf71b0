// voxel.cu -- voxel occupancy grid (Fig. voxels, the paper's voxel prototype):
// every cell of a g x g x g grid over the march box is classified at its centre
// like a ray sample (slice map, then the escape-time iteration), giving an
// occupancy byte (1 = no escape by max_iter) and the escape count.
//
// Fine grids (FP32) are taken in bricks of 16 x 8 x 4 cells, eight sub-bricks of 8 x
// 4 x 2 each.  Far from the set the escape count is constant over whole bricks, and a
// bound proves it (settle_box): those are filled, as are the settled sub-bricks
// of the others; only what is left is classified, a sub-brick at a time (lane =
// column, its two z cells in the float2 halves of the paired march
// classification).  Coarse grids classify every cell, in 32 x 2 row segments.
// Warps claim their work through an atomic counter (persistent grid).
// FP64 runs one cell per lane; FP32 + recheck queues cells whose modulus came
// within the margin of R^2 and re-classifies them in FP64 afterwards (a queue
// overflow re-runs the whole grid in FP64).
#include <algorithm>
#include <cmath>

#include "render_common.cuh"
#include "runtime.h"

namespace dqj {

namespace {

struct VoxelArgs {
    int32_t g;
    uint32_t segs_per_row;                 // FP32, row segments
    uint64_t nsegs;
    uint32_t bricks_x, bricks_y, nbricks;  // FP32, bricks along x, along y, in all
    float radius;                          // |slice origin| + largest |corner| of the box
    int32_t wide;                          // rows of 16 cells are 16-byte aligned in occ and counts
    uint8_t *occ;       // g^3 or NULL
    uint16_t *count;    // g^3 or NULL
    Counters *ctr;      // stats in DQJ_STAT_* order, tile_next = segment claim, queue_count
    uint32_t *queue;    // FP32 + recheck: cells to re-classify in FP64
    uint32_t queue_cap;
};

// Scene-space step of the grid along each axis.
template <typename T>
__device__ __forceinline__ void grid_step(const FrameT<T> &F, int g, T (&step)[3])
{
#pragma unroll
    for (int a = 0; a < 3; ++a) step[a] = (F.bmax[a] - F.bmin[a]) / T(g);
}

// Slice image of the cell centre (x, y, z) = (p0, row's y, row's z): the row
// part O + y E_1 + z E_2 is shared by the whole row.
template <typename T>
__device__ __forceinline__ void row_base(const FrameT<T> &F, const T (&step)[3], int j, int k, T (&base)[8])
{
    const T y = dfma(T(j) + T(0.5), step[1], F.bmin[1]);
    const T z = dfma(T(k) + T(0.5), step[2], F.bmin[2]);
#pragma unroll
    for (int i = 0; i < 8; ++i) base[i] = dfma(z, F.E[2][i], dfma(y, F.E[1][i], F.O[i]));
}

__device__ __forceinline__ void write_cell(const VoxelArgs &va, uint64_t lin, bool inside, int esc)
{
    if (va.occ) va.occ[lin] = inside ? 1 : 0;
    if (va.count) va.count[lin] = (uint16_t)(inside ? 0 : esc);
}

// Re-classify cell lin in FP64 (n = its FP64 escape count) and overwrite it
// where the result differs; returns the change of the inside count.
__device__ __forceinline__ long long fix_cell(const VoxelArgs &va, uint64_t lin, int n, unsigned long long &fixed)
{
    const bool inside = n == 0;
    const bool was = va.occ ? va.occ[lin] != 0 : va.count[lin] == 0;
    const bool changed = was != inside || (va.count && va.count[lin] != (uint16_t)n);
    if (!changed) return 0;
    write_cell(va, lin, inside, n);
    fixed += 1;
    return (inside ? 1 : 0) - (was ? 1 : 0);
}

// Segments are claimed kBatch at a time; inside a batch the row coordinates
// advance incrementally (no division per segment).
constexpr uint32_t kBatch = 16;

// Grids of fewer than kBrickGrid cells a side: paired FP32 classification of two
// cells per lane, every cell.  A segment is 32 x 2
// cells: 32 along x in the row pair (2 jp, 2 jp + 1) of one z slice; lane l
// takes column x0 + l of both rows, so its two cells share px and differ only
// in the rows' (warp-uniform) slice bases, and each warp store covers 32
// consecutive cells of a row.  32 x 2 segments keep the warp's cells closer
// together than 64 x 1 rows, so its lockstep rounds wait less for the slowest
// cell (escape counts of the default grid at 1024^3: 0.945 of the steps are
// useful against 0.904).  Cell indices fit in 32 bits (g <= 1024); per-lane
// counts are 32-bit within a batch.
template <int SQ, int MOD, bool RECHECK, bool AXIS>
__global__ void __launch_bounds__(kBlock, 5) voxel2_kernel(const __grid_constant__ FrameDesc fd, const VoxelArgs va)
{
    const FrameT<float> &F = fd.f;
    const int lane = threadIdx.x & 31;
    const int g = va.g;
    const uint32_t gu = (uint32_t)g;
    const uint32_t spr = va.segs_per_row, nsegs = (uint32_t)va.nsegs;
    const uint32_t npairs = (gu + 1u) / 2u;
    const uint32_t max_iter = (uint32_t)fd.max_iter;
    float step[3];
    grid_step<float>(F, g, step);
    unsigned long long iters = 0, inside_n = 0, rechecks = 0, cells = 0;
    for (;;) {
        uint32_t first = 0;
        if (lane == 0) first = atomicAdd(&va.ctr->tile_next, kBatch);
        first = __shfl_sync(kFull, first, 0);
        if (first >= nsegs) break;
        const uint32_t last = min(first + kBatch, nsegs);
        uint32_t rp = first / spr;
        int x0 = (int)(first - rp * spr) * 32;
        int jp = (int)(rp % npairs), k = (int)(rp / npairs);
        float ba[8], bb[8];  // slice bases of the two rows (row 2 jp + 1 = g of an odd grid is unused)
        row_base<float>(F, step, 2 * jp, k, ba);
        row_base<float>(F, step, 2 * jp + 1, k, bb);
        uint32_t it32 = 0, in32 = 0, cl32 = 0, re32 = 0;
        for (uint32_t seg = first; seg < last; ++seg) {
            const int x = x0 + lane, j0 = 2 * jp;
            const bool two = j0 + 1 < g;
            bool aa = x < g, ab = aa && two;
            const float p = fmaf((float)x + 0.5f, step[0], F.bmin[0]);
            const float2 px = make_float2(p, p);
            float2 z[8];
#pragma unroll
            for (int i = 0; i < (AXIS ? 3 : 8); ++i)  // AXIS: components 3..7 are zero
                z[i] = f2fma(px, make_float2(F.E[0][i], F.E[0][i]), make_float2(ba[i], bb[i]));
            int ca, cb;
            bool live;
            float2 dm;
            const bool va_ = aa, vb_ = ab;
            classify_lockstep2<SQ, MOD, RECHECK, AXIS>(z, fd.p2, F.R2, fd.max_iter, aa, ab, ca, cb, dm, live);
            const bool mga = dm.x <= fd.p2.margin_t, mgb = dm.y <= fd.p2.margin_t;
            const uint32_t la = ((uint32_t)k * gu + (uint32_t)j0) * gu + (uint32_t)x, lb = la + gu;
            if (lane == 0) cl32 += (uint32_t)min(32, g - x0) * (two ? 2u : 1u);
            if (va_) {
                write_cell(va, la, aa, ca + 1);
                it32 += aa ? max_iter : (uint32_t)(ca + 1);
                in32 += aa ? 1u : 0u;
            }
            if (vb_) {
                write_cell(va, lb, ab, cb + 1);
                it32 += ab ? max_iter : (uint32_t)(cb + 1);
                in32 += ab ? 1u : 0u;
            }
            if (RECHECK) {
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const bool push = h == 0 ? (va_ && mga) : (vb_ && mgb);
                    const unsigned m = __ballot_sync(kFull, push);
                    if (m == 0) continue;
                    const int leader = __ffs(m) - 1;
                    unsigned b = 0;
                    if (lane == leader) b = atomicAdd(&va.ctr->queue_count, (unsigned)__popc(m));
                    b = __shfl_sync(kFull, b, leader);
                    if (push) {
                        const unsigned slot = b + __popc(m & ((1u << lane) - 1u));
                        if (slot < va.queue_cap)
                            va.queue[slot] = h == 0 ? la : lb;
                        else
                            atomicAdd(&va.ctr->stats[7], 1ull);  // overflow: the FP64 pass re-runs the grid
                        re32 += 1;
                    }
                }
            }
            x0 += 32;  // next segment: same row pair, or the start of the next one
            if (x0 >= g) {
                x0 = 0;
                if (++jp == (int)npairs) {
                    jp = 0;
                    ++k;
                }
                if (seg + 1 < last) {
                    row_base<float>(F, step, 2 * jp, k, ba);
                    row_base<float>(F, step, 2 * jp + 1, k, bb);
                }
            }
        }
        iters += it32;
        inside_n += in32;
        cells += cl32;
        rechecks += re32;
    }
    flush_stat(&va.ctr->stats[0], iters);
    flush_stat(&va.ctr->stats[2], cells);
    flush_stat(&va.ctr->stats[3], inside_n);
    if (RECHECK) flush_stat(&va.ctr->stats[4], rechecks);
}

// Bricks against 32 x 2 row segments, FP32, axis / random slice (ms): 256^3 0.105 /
// 0.143 against 0.092 / 0.135, 300^3 0.141 / 0.192 against 0.130 / 0.199, 333^3 0.166 /
// 0.225 against 0.166 / 0.253, 400^3 0.16 / 0.27 against 0.25 / 0.40, 1024^3 1.67 /
// 2.83 against 3.42 / 5.73: coarse bricks settle too seldom to pay for the bound.
constexpr int kBrickGrid = 336;
constexpr int kBrickX = 16, kBrickY = 8, kBrickZ = 4;  // a brick; its eight sub-bricks are half as long each way
constexpr uint32_t kBrickClaim = 4;                     // bricks a warp claims: a sub-brick per lane

// The count (15: inside) shared by the cells of the sub-brick at (x, y, z) (clipped
// to the grid), or 0 when the bound does not prove one.
template <int SQ, int MOD, bool AXIS>
__device__ __forceinline__ int settle_cells(const FrameDesc &fd, const VoxelArgs &va, const float (&step)[3], int x,
                                            int y, int z)
{
    const int lo[3] = {x, y, z};
    const int n[3] = {min(kBrickX / 2, va.g - x), min(kBrickY / 2, va.g - y), min(kBrickZ / 2, va.g - z)};
    const float rho = 4e-6f * va.radius, e1 = 8e-6f * va.radius * va.radius;
    float p[3], h[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        p[a] = fmaf((float)lo[a] + 0.5f * (float)n[a], step[a], fd.f.bmin[a]);
        h[a] = fmaf(0.5f * (float)(n[a] - 1), step[a], rho);
    }
    return settle_box<SQ, MOD, AXIS, true>(fd, p, h, rho, e1);
}

// A row of 16 settled cells starting at lin.
__device__ __forceinline__ void fill_row16(const VoxelArgs &va, uint32_t lin, int n)
{
    const bool in = n == kSettleInside;
    const unsigned o = in ? 0x01010101u : 0u, v = in ? 0u : (unsigned)n * 0x10001u;
    if (va.occ) *reinterpret_cast<uint4 *>(va.occ + lin) = make_uint4(o, o, o, o);
    if (va.count) {
        uint4 *c = reinterpret_cast<uint4 *>(va.count + lin);
        c[0] = make_uint4(v, v, v, v);
        c[1] = make_uint4(v, v, v, v);
    }
}

// Grids of kBrickGrid cells a side or more (see the head of this file).  A claim is
// four bricks, whose 32 sub-bricks are settled one per lane.  Larger claims, whole
// bricks tried first, bounded fewer boxes but left the warps unequal shares; they
// were slower at every size (default c / random slice / random c, ms): 512^3 0.275 /
// 0.473 / 0.189 with four bricks, 0.334 / 0.585 / 0.262 with 16, 0.404 / 0.714 / 0.280
// with 32; 1024^3 1.68 / 2.80 / 1.33, 1.89 / 2.94 / 1.75, 1.95 / 2.93 / 1.87.
// 1024^3 (default constant): nine in ten sub-bricks settle (inside ones too), 3.42 ->
// 1.67 ms; the 3.2 GB written take 0.47 ms at the measured copy rate.  What is left
// is the classification of the others, whose cells run 8 to max_iter steps.
template <int SQ, int MOD, bool RECHECK, bool AXIS>
__global__ void __launch_bounds__(kBlock, 5) voxel_brick_kernel(const __grid_constant__ FrameDesc fd, const VoxelArgs va)
{
    const FrameT<float> &F = fd.f;
    const int lane = threadIdx.x & 31;
    const int g = va.g;
    const uint32_t gu = (uint32_t)g;
    const uint32_t max_iter = (uint32_t)fd.max_iter;
    float step[3];
    grid_step<float>(F, g, step);
    const int lx = lane & 7, ly = lane >> 3;  // column of a sub-brick
    unsigned long long iters = 0, inside_n = 0, rechecks = 0, cells = 0;
    for (;;) {
        uint32_t first = 0;
        if (lane == 0) first = atomicAdd(&va.ctr->tile_next, kBrickClaim);
        first = __shfl_sync(kFull, first, 0);
        if (first >= va.nbricks) break;
        const int nb = (int)min(kBrickClaim, va.nbricks - first);
        // lane 8 b + s: sub-brick s of brick first + b; w: the counts of the lane's
        // brick, four bits a sub-brick
        int bx, by, bz;
        unsigned w;
        {
            const uint32_t id = first + (uint32_t)min(lane >> 3, nb - 1), row = id / va.bricks_x;
            bx = (int)(id - row * va.bricks_x) * kBrickX;
            bz = (int)(row / va.bricks_y);
            by = (int)(row - (uint32_t)bz * va.bricks_y) * kBrickY;
            bz *= kBrickZ;
            const int sb = lane & 7;
            const int x = bx + (sb & 1) * (kBrickX / 2), y = by + (sb >> 1 & 1) * (kBrickY / 2),
                      z = bz + (sb >> 2) * (kBrickZ / 2);
            int n = 0;
            if ((lane >> 3) < nb && x < g && y < g && z < g) n = settle_cells<SQ, MOD, AXIS>(fd, va, step, x, y, z);
            __syncwarp();
            w = (unsigned)n << (4 * sb);
            w |= __shfl_xor_sync(kFull, w, 1);
            w |= __shfl_xor_sync(kFull, w, 2);
            w |= __shfl_xor_sync(kFull, w, 4);
        }
        uint32_t it32 = 0, in32 = 0, cl32 = 0, re32 = 0;
        for (int b = 0; b < nb; ++b) {
            const unsigned word = __shfl_sync(kFull, w, 8 * b);
            const int x0 = __shfl_sync(kFull, bx, 8 * b), y0 = __shfl_sync(kFull, by, 8 * b),
                      z0 = __shfl_sync(kFull, bz, 8 * b);
            const int n0 = (int)(word & 15u);
            if (va.wide && n0 && word == (unsigned)n0 * 0x11111111u && x0 + kBrickX <= g) {
                // a settled brick: 32 rows of 16 cells, one per lane
                const int y = y0 + (lane & 7), z = z0 + (lane >> 3);
                if (y < g && z < g) {
                    fill_row16(va, ((uint32_t)z * gu + (uint32_t)y) * gu + (uint32_t)x0, n0);
                    it32 += 16u * (n0 == kSettleInside ? max_iter : (uint32_t)n0);
                    in32 += n0 == kSettleInside ? 16u : 0u;
                    cl32 += 16u;
                }
                continue;
            }
            // the lane's column in the brick's first sub-brick, its coordinates in
            // cells (exact: no conversion per sub-brick) and linear index
            const int xb = x0 + lx, yb = y0 + ly;
            const float xf = (float)xb + 0.5f, yf = (float)yb + 0.5f, zf = (float)z0 + 0.5f;
            const uint32_t lin = ((uint32_t)z0 * gu + (uint32_t)yb) * gu + (uint32_t)xb;
#pragma unroll 1
            for (int sb = 0; sb < 8; ++sb) {
                const int dx = (sb & 1) * (kBrickX / 2), dy = (sb >> 1 & 1) * (kBrickY / 2), dz = (sb >> 2) * (kBrickZ / 2);
                const int z = z0 + dz;
                if (x0 + dx >= g || y0 + dy >= g || z >= g) continue;  // warp-uniform
                const int n = (int)((word >> (4 * sb)) & 15u);
                const bool va_ = xb + dx < g && yb + dy < g, vb_ = va_ && z + 1 < g;
                const uint32_t la = lin + ((uint32_t)dz * gu + (uint32_t)dy) * gu + (uint32_t)dx, lb = la + gu * gu;
                cl32 += (va_ ? 1u : 0u) + (vb_ ? 1u : 0u);
                if (n) {  // a settled sub-brick
                    const bool in = n == kSettleInside;
                    const uint32_t c = (va_ ? 1u : 0u) + (vb_ ? 1u : 0u);
                    if (va_) write_cell(va, la, in, n);
                    if (vb_) write_cell(va, lb, in, n);
                    it32 += (in ? max_iter : (uint32_t)n) * c;
                    in32 += in ? c : 0u;
                    continue;
                }
                bool aa = va_, ab = vb_;
                const float px = fmaf(xf + (sb & 1 ? (float)(kBrickX / 2) : 0.f), step[0], F.bmin[0]);
                const float py = fmaf(yf + (sb & 2 ? (float)(kBrickY / 2) : 0.f), step[1], F.bmin[1]);
                const float zc = zf + (sb & 4 ? (float)(kBrickZ / 2) : 0.f);
                const float pz = fmaf(zc, step[2], F.bmin[2]), pz1 = fmaf(zc + 1.f, step[2], F.bmin[2]);
                float2 q[8];
#pragma unroll
                for (int i = 0; i < (AXIS ? 3 : 8); ++i) {  // AXIS: components 3..7 are zero
                    const float r = fmaf(py, F.E[1][i], F.O[i]);
                    q[i] = f2fma(make_float2(px, px), make_float2(F.E[0][i], F.E[0][i]),
                                 make_float2(fmaf(pz, F.E[2][i], r), fmaf(pz1, F.E[2][i], r)));
                }
                int ca, cb;
                bool live;
                float2 dm;
                classify_lockstep2<SQ, MOD, RECHECK, AXIS>(q, fd.p2, F.R2, fd.max_iter, aa, ab, ca, cb, dm, live);
                const bool mga = dm.x <= fd.p2.margin_t, mgb = dm.y <= fd.p2.margin_t;
                if (va_) {
                    write_cell(va, la, aa, ca + 1);
                    it32 += aa ? max_iter : (uint32_t)(ca + 1);
                    in32 += aa ? 1u : 0u;
                }
                if (vb_) {
                    write_cell(va, lb, ab, cb + 1);
                    it32 += ab ? max_iter : (uint32_t)(cb + 1);
                    in32 += ab ? 1u : 0u;
                }
                if (RECHECK) {
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const bool push = h == 0 ? (va_ && mga) : (vb_ && mgb);
                        const unsigned m = __ballot_sync(kFull, push);
                        if (m == 0) continue;
                        const int leader = __ffs(m) - 1;
                        unsigned at = 0;
                        if (lane == leader) at = atomicAdd(&va.ctr->queue_count, (unsigned)__popc(m));
                        at = __shfl_sync(kFull, at, leader);
                        if (push) {
                            const unsigned slot = at + __popc(m & ((1u << lane) - 1u));
                            if (slot < va.queue_cap)
                                va.queue[slot] = h == 0 ? la : lb;
                            else
                                atomicAdd(&va.ctr->stats[7], 1ull);  // overflow: the FP64 pass re-runs the grid
                            re32 += 1;
                        }
                    }
                }
            }
        }
        iters += it32;
        inside_n += in32;
        cells += cl32;
        rechecks += re32;
    }
    flush_stat(&va.ctr->stats[0], iters);
    flush_stat(&va.ctr->stats[2], cells);
    flush_stat(&va.ctr->stats[3], inside_n);
    if (RECHECK) flush_stat(&va.ctr->stats[4], rechecks);
}

// FP64 classification, one cell per lane (32-cell row segments).
template <int SQ, int MOD>
__global__ void __launch_bounds__(kBlock) voxel64_kernel(const __grid_constant__ FrameDesc fd, const VoxelArgs va)
{
    const FrameT<double> &F = fd.d;
    const int lane = threadIdx.x & 31;
    const int g = va.g;
    const uint32_t spr = (uint32_t)((g + 31) / 32);
    const uint32_t nsegs = (uint32_t)g * (uint32_t)g * spr;
    double step[3];
    grid_step<double>(F, g, step);
    unsigned long long iters = 0, inside_n = 0, cells = 0;
    for (;;) {
        uint32_t first = 0;
        if (lane == 0) first = atomicAdd(&va.ctr->tile_next, kBatch);
        first = __shfl_sync(kFull, first, 0);
        if (first >= nsegs) break;
        const uint32_t last = min(first + kBatch, nsegs);
        for (uint32_t seg = first; seg < last; ++seg) {
            const uint32_t row = seg / spr;
            const int x = (int)(seg - row * spr) * 32 + lane;
            const int j = (int)(row % (uint32_t)g), k = (int)(row / (uint32_t)g);
            double base[8], z[8];
            row_base<double>(F, step, j, k, base);
            const double p0 = fma((double)x + 0.5, step[0], F.bmin[0]);
#pragma unroll
            for (int i = 0; i < 8; ++i) z[i] = fma(p0, F.E[0][i], base[i]);
            bool mg;
            const bool part = x < g;
            const int n = classify_sample<double, SQ, MOD, false>(fd, z, part, mg);
            if (part) {
                write_cell(va, (uint64_t)row * (uint64_t)g + x, n == 0, n);
                iters += n ? (unsigned)n : (unsigned)fd.max_iter;
                inside_n += n == 0 ? 1 : 0;
                cells += 1;
            }
        }
    }
    flush_stat(&va.ctr->stats[0], iters);
    flush_stat(&va.ctr->stats[2], cells);
    flush_stat(&va.ctr->stats[3], inside_n);
}

// FP64 re-classification of one cell (recheck and overflow passes).
template <int SQ, int MOD>
__device__ __forceinline__ int cell_fp64(const FrameDesc &fd, int g, uint64_t lin, unsigned long long &it)
{
    const FrameT<double> &F = fd.d;
    double step[3], base[8], z[8];
    grid_step<double>(F, g, step);
    const int x = (int)(lin % (uint64_t)g);
    const uint64_t row = lin / (uint64_t)g;
    row_base<double>(F, step, (int)(row % (uint64_t)g), (int)(row / (uint64_t)g), base);
    const double p0 = fma((double)x + 0.5, step[0], F.bmin[0]);
#pragma unroll
    for (int i = 0; i < 8; ++i) z[i] = fma(p0, F.E[0][i], base[i]);
    bool certain;
    int n = count_bound64<SQ, MOD>(fd, z, certain);
    if (!certain) n = count64<SQ, MOD>(fd, z);
    it += n ? (unsigned)n : (unsigned)fd.max_iter;
    return n;
}

template <int SQ, int MOD>
__global__ void __launch_bounds__(kBlock) voxel_recheck_kernel(const __grid_constant__ FrameDesc fd, const VoxelArgs va)
{
    const unsigned nq = min(*(volatile unsigned *)&va.ctr->queue_count, va.queue_cap);
    unsigned long long fixed = 0, it = 0;
    long long delta = 0;
    for (unsigned q = blockIdx.x * blockDim.x + threadIdx.x; q < nq; q += gridDim.x * blockDim.x) {
        const uint64_t lin = va.queue[q];
        delta += fix_cell(va, lin, cell_fp64<SQ, MOD>(fd, va.g, lin, it), fixed);
    }
    flush_stat(&va.ctr->stats[5], fixed);
    flush_stat(&va.ctr->stats[6], it);
    flush_stat(&va.ctr->stats[3], (unsigned long long)delta);
}

// After a queue overflow: every cell again in FP64 (and the inside count with it).
template <int SQ, int MOD>
__global__ void __launch_bounds__(kBlock) voxel_overflow_kernel(const __grid_constant__ FrameDesc fd, const VoxelArgs va)
{
    if (*(volatile unsigned long long *)&va.ctr->stats[7] == 0) return;
    const uint64_t n = (uint64_t)va.g * (uint64_t)va.g * (uint64_t)va.g;
    unsigned long long fixed = 0, it = 0;
    long long delta = 0;
    for (uint64_t lin = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; lin < n;
         lin += (uint64_t)gridDim.x * blockDim.x)
        delta += fix_cell(va, lin, cell_fp64<SQ, MOD>(fd, va.g, lin, it), fixed);
    flush_stat(&va.ctr->stats[5], fixed);
    flush_stat(&va.ctr->stats[6], it);
    flush_stat(&va.ctr->stats[3], (unsigned long long)delta);
}

template <int SQ, int MOD>
cudaError_t launch_voxels_t(const FrameDesc &fd, const VoxelArgs &args, cudaStream_t st, int num_sms)
{
    static std::atomic<int> g64{0}, g2{0}, gb{0}, gre{0}, gov{0};
    if (fd.precision == DQJ_FP64) {
        voxel64_kernel<SQ, MOD><<<num_sms * resident_per_sm(g64, voxel64_kernel<SQ, MOD>), kBlock, 0, st>>>(fd, args);
        return cudaGetLastError();
    }
    const bool re = fd.precision == DQJ_FP32_RECHECK;
    const int axis = fd.axis_slice ? 1 : 0;
    if (args.g >= kBrickGrid && fd.blocks) {
        const uint32_t cap =
            (uint32_t)num_sms * (uint32_t)resident_per_sm(gb, voxel_brick_kernel<SQ, MOD, false, false>);
        const uint32_t claims = (args.nbricks + kBrickClaim - 1u) / kBrickClaim;
        const int gg = (int)std::min(cap, (claims + 3u) / 4u);
        if (re)
            axis ? voxel_brick_kernel<SQ, MOD, true, true><<<gg, kBlock, 0, st>>>(fd, args)
                 : voxel_brick_kernel<SQ, MOD, true, false><<<gg, kBlock, 0, st>>>(fd, args);
        else
            axis ? voxel_brick_kernel<SQ, MOD, false, true><<<gg, kBlock, 0, st>>>(fd, args)
                 : voxel_brick_kernel<SQ, MOD, false, false><<<gg, kBlock, 0, st>>>(fd, args);
    } else {
        const int gm = (int)min((uint64_t)num_sms * resident_per_sm(g2, voxel2_kernel<SQ, MOD, false, false>),
                                (args.nsegs + 4 * kBatch - 1) / (4 * kBatch));
        const int gg = gm > 0 ? gm : 1;
        if (re)
            axis ? voxel2_kernel<SQ, MOD, true, true><<<gg, kBlock, 0, st>>>(fd, args)
                 : voxel2_kernel<SQ, MOD, true, false><<<gg, kBlock, 0, st>>>(fd, args);
        else
            axis ? voxel2_kernel<SQ, MOD, false, true><<<gg, kBlock, 0, st>>>(fd, args)
                 : voxel2_kernel<SQ, MOD, false, false><<<gg, kBlock, 0, st>>>(fd, args);
    }
    if (re) {
        voxel_recheck_kernel<SQ, MOD><<<num_sms * resident_per_sm(gre, voxel_recheck_kernel<SQ, MOD>), kBlock, 0, st>>>(fd, args);
        voxel_overflow_kernel<SQ, MOD><<<num_sms * resident_per_sm(gov, voxel_overflow_kernel<SQ, MOD>), kBlock, 0, st>>>(fd, args);
    }
    return cudaGetLastError();
}

cudaError_t launch_voxels(const FrameDesc &fd, const VoxelArgs &va, cudaStream_t st, int num_sms)
{
    if (fd.square_mode == 0)
        return fd.modulus_mode == 0 ? launch_voxels_t<0, 0>(fd, va, st, num_sms)
                                    : launch_voxels_t<0, 1>(fd, va, st, num_sms);
    return fd.modulus_mode == 0 ? launch_voxels_t<1, 0>(fd, va, st, num_sms) : launch_voxels_t<1, 1>(fd, va, st, num_sms);
}

}  // namespace

}  // namespace dqj

using namespace dqj;

extern "C" dqj_status dqj_voxelize(dqj_ctx *ctx, const dqj_params *p, int32_t grid_n, uint8_t *occupancy,
                                   uint16_t *counts, int64_t *stats, void *cuda_stream)
{
    return dqj::guarded([&]() -> dqj_status {
        if (!ctx) return fail(DQJ_ERR_INVALID, "ctx is NULL");
        dqj_status s = validate(p);
        if (s != DQJ_OK) return s;
        if (grid_n < 1 || grid_n > DQJ_VOXEL_MAX_GRID)
            return fail(DQJ_ERR_INVALID, "grid_n must be in 1.." + std::to_string(DQJ_VOXEL_MAX_GRID));
        if (counts && (reinterpret_cast<uintptr_t>(counts) & 1u)) return fail(DQJ_ERR_INVALID, "counts must be 2-byte aligned");
        if (stats && (reinterpret_cast<uintptr_t>(stats) & 7u)) return fail(DQJ_ERR_INVALID, "stats must be 8-byte aligned");
        if (!occupancy && !counts) return fail(DQJ_ERR_INVALID, "occupancy and counts are both NULL");
        if (ctx->device == DQJ_DEVICE_MOCK) return fail(DQJ_ERR_INVALID, "a mock context cannot voxelize");
        std::lock_guard<std::mutex> lk(ctx->mu);
        cudaError_t e = cudaSetDevice(ctx->device);
        if (e != cudaSuccess) return cuda_fail(e, "voxelize: cudaSetDevice");
        const uint64_t cells = (uint64_t)grid_n * (uint64_t)grid_n * (uint64_t)grid_n;
        const bool re = p->precision == DQJ_FP32_RECHECK;
        const uint64_t qcap = re ? std::min<uint64_t>(cells, 1ull << 24) : 0;
        const size_t need = 256 + qcap * sizeof(uint32_t);
        if (ctx->vox_bytes < need) {
            e = cudaDeviceSynchronize();
            if (e != cudaSuccess) return cuda_fail(e, "voxelize: synchronize");
            if (ctx->vox_scratch) cudaFree(ctx->vox_scratch);
            ctx->vox_scratch = nullptr;
            ctx->vox_bytes = 0;
            e = cudaMalloc(&ctx->vox_scratch, need);
            if (e != cudaSuccess) return cuda_fail(e, "voxelize: cudaMalloc");
            ctx->vox_bytes = need;
        }
        FrameDesc fd;
        derive_frame(*p, fd, 8, 8);
        VoxelArgs va{};
        va.g = grid_n;
        va.segs_per_row = (uint32_t)((grid_n + 31) / 32);  // 32 x 2 segments
        va.nsegs = (uint64_t)grid_n * (uint64_t)((grid_n + 1) / 2) * va.segs_per_row;
        va.bricks_x = (uint32_t)((grid_n + kBrickX - 1) / kBrickX);
        va.bricks_y = (uint32_t)((grid_n + kBrickY - 1) / kBrickY);
        va.nbricks = va.bricks_x * va.bricks_y * (uint32_t)((grid_n + kBrickZ - 1) / kBrickZ);
        double corner = 0.0;
        for (int a = 0; a < 3; ++a) {
            const double m = std::max(std::fabs(p->box_min[a]), std::fabs(p->box_max[a]));
            corner += m * m;
        }
        double origin = 0.0;
        for (int i = 0; i < 8; ++i) origin += p->slice_origin[i] * p->slice_origin[i];
        va.radius = (float)(std::sqrt(corner) + std::sqrt(origin));
        va.wide = grid_n % 16 == 0 && (reinterpret_cast<uintptr_t>(occupancy) & 15u) == 0 &&
                  (reinterpret_cast<uintptr_t>(counts) & 15u) == 0;
        va.occ = occupancy;
        va.count = counts;
        va.ctr = static_cast<Counters *>(ctx->vox_scratch);
        va.queue = reinterpret_cast<uint32_t *>(static_cast<char *>(ctx->vox_scratch) + 256);
        va.queue_cap = (uint32_t)qcap;
        cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
        e = cudaStreamWaitEvent(st, ctx->done_ev, 0);
        if (e == cudaSuccess) e = cudaMemsetAsync(va.ctr, 0, sizeof(Counters), st);
        if (e == cudaSuccess) e = launch_voxels(fd, va, st, ctx->num_sms);
        if (e == cudaSuccess && stats)
            e = cudaMemcpyAsync(stats, va.ctr->stats, DQJ_NSTATS * sizeof(int64_t), cudaMemcpyDeviceToDevice, st);
        if (e == cudaSuccess) e = cudaEventRecord(ctx->done_ev, st);
        if (e != cudaSuccess) return cuda_fail(e, "voxelize: launch");
        return DQJ_OK;
    });
}
