// render_passes.cuh -- sm_103a kernels of the dual-quaternion Julia isosurface renderer.
//
// One frame runs as up to four stream-ordered passes:
//   march   : one ray per lane, 32 rays of a screen tile per warp.  The lanes
//             march in step: every trip of the warp classifies sample k of each
//             lane's ray (Method, "Ray-Marching": fixed steps over the box), so
//             neighbouring rays - which see almost the same escape counts - share
//             trips and no lane diverges.  Runs of samples whose count a bound
//             proves for the whole tile are not iterated (settle.cuh).  Misses write their final outputs;
//             hits are appended to a compacted hit list.
//   bisect  : one hit per lane: B bisection steps of the first outside->inside
//             bracket, then the six central-difference evaluations of the normal
//             field (Method, "Lighting/Illumination") and Eq. phong shading
//             (ambient + diffuse).  Splitting hits from the march keeps the long
//             near-surface classifications together instead of stalling warps
//             that are still marching.
//   recheck : (FP32_RECHECK) samples whose modulus came within the margin of R^2
//             and whose count the FP32 orbit's rounding bound leaves open are
//             decided from FP64 ray parameters, by a two-float orbit and its
//             bound, else in FP64, gathered; a pixel whose count differs goes to
//   fixup   : a re-render of that pixel at FP64 accuracy, five pixels per warp.
// Iteration counts are the algorithmic ones (escape count, or max_iter for an
// inside sample), accumulated per lane and added once per warp.
#pragma once

#include <algorithm>
#include <cstdlib>

#include "render_common.cuh"
#include "../../include/dqj.h"

namespace dqj {

namespace {

// ---------------------------------------------------------------------------
// march
// ---------------------------------------------------------------------------
// AXIS: an axis-aligned slice, for the settled blocks (the samples themselves
// take the general step, whose products with zero components change nothing).
template <typename T, int SQ, int MOD, bool RECHECK, bool AXIS>
__global__ void __launch_bounds__(kBlock) march_kernel(const __grid_constant__ FrameDesc fd, const Scratch sc)
{
    __shared__ TileBox s_box[kBlock / 32];
    TileBox &box = s_box[threadIdx.x >> 5];
    const FrameT<T> &F = frame<T>(fd);
    const int lane = threadIdx.x & 31;
    const unsigned ntiles = subset_tiles(fd, (unsigned)fd.tiles_x * (unsigned)fd.tiles_y);
    unsigned long long s_iters = 0, s_samples = 0, s_hits = 0, s_rechecks = 0;
    for (;;) {
        unsigned tile = 0;
        if (lane == 0) tile = atomicAdd(&sc.ctr->tile_next, 1u);
        tile = __shfl_sync(kFull, tile, 0);
        if (tile >= ntiles) break;
        tile = subset_tile(fd, tile);
        const int tx = (int)(tile % (unsigned)fd.tiles_x), ty = (int)(tile / (unsigned)fd.tiles_x);
        const int x = tx * fd.tile_w + lane % fd.tile_w;
        const int y = ty * fd.tile_h + lane / fd.tile_w;
        const bool valid = x < fd.W && y < fd.H;
        T d[3] = {T(0), T(0), T(1)};
        T t_in = T(0), t_out = T(0);
        bool active = valid && camera_clip<T>(F, fd.W, fd.H, x, y, d, t_in, t_out);
        if (!active) t_in = t_out = T(0);
        if (fd.settle) {
            const float df[3] = {(float)d[0], (float)d[1], (float)d[2]};
            tile_box(fd, active, df, (float)t_in, (float)t_out, false, df, 0.f, 0.f, box);
        }
        T D[8];
        slice_dir<T>(F, d, D);
        const T delta = (t_out - t_in) / T(fd.N);
        // FP32 general slice: the first-iterate form of the paired kernel, same
        // operations per ray
        constexpr bool it1 = sizeof(T) == 4 && !AXIS;
        T Q0[8], Q1[8], Q2[8], dot = T(0);
        if constexpr (it1) first_iterate_coeffs<float, SQ>(F.A, D, F.c, dot, Q0, Q1, Q2);
        const T s_in = it1 ? (T)vadd((float)t_in, (float)dot) : t_in;
        int esc_max = 0, k_first = -1;
        unsigned iters = 0, samples = 0;
        bool more = __any_sync(kFull, active);
        auto sample = [&](int k, auto finished) {
            T z[8];
            bool mg;
            int n;
            if constexpr (it1) {
                first_iterate<float, 8>(vfma((float)k, delta, s_in), Q0, Q1, Q2, z);
                n = classify_lockstep_it1<T, SQ, MOD, RECHECK>(z, F, fd.max_iter, active, mg);
            } else {
                const T t = dfma(T(k), delta, t_in);
#pragma unroll
                for (int i = 0; i < 8; ++i) z[i] = dfma(t, D[i], F.A[i]);
                n = classify_sample<T, SQ, MOD, RECHECK>(fd, z, active, mg);
            }
            if (RECHECK) {
                const bool push = active && mg;
                if (warp_push(push, make_int4(y * fd.W + x, k | (kMarchSample << 16), x | (y << 16), n), sc.queue,
                              sc.queue_cap, &sc.ctr->queue_count)) {
                    atomicAdd(&sc.ctr->stats[7], 1ull);
                    mark_dirty(fd, sc, y * fd.W + x);
                }
                s_rechecks += push ? 1 : 0;
            }
            if (active) {
                iters += n ? (unsigned)n : (unsigned)fd.max_iter;
                samples += 1;
                if (n) esc_max = n > esc_max ? n : esc_max;
            }
            const bool ends = active && n == 0;
            if (__any_sync(kFull, ends)) {
                finished(ends);
                if (ends) {
                    k_first = k;
                    active = false;
                }
                more = __any_sync(kFull, active);
            }
        };
        // the settled samples add to the counts of the rays that pass them
        // (sums and maxima of count - 1, over cnt samples)
        auto add = [&](bool f, int s, int cnt, int m) {
            if (f && cnt) {
                iters += (unsigned)(s + cnt);
                samples += (unsigned)cnt;
                esc_max = max(esc_max, m + 1);
            }
        };
        for (int kc = 0; kc <= fd.N && more; kc += kSettleChunk) {
            const int ke = min(kc + kSettleChunk, fd.N + 1), pairs = settle_pairs(ke - kc);
            unsigned w = 0;
            if (fd.settle && ke - kc > kSettleMin) w = settle_chunk<SQ, MOD, AXIS>(fd, box, kc, ke, pairs);
            const unsigned open = open_pairs(w, kc, ke, pairs);
            unsigned blocks = __ballot_sync(kFull, open != 0);
            int marched = 0;  // samples of the chunk marched so far
            while (blocks && more) {
                const int b = __ffs(blocks) - 1;
                blocks &= blocks - 1;
                unsigned ob = __shfl_sync(kFull, open, b);
                while (ob && more) {
                    const int p = (__ffs(ob) - 1) >> 2;
                    ob &= ob - 1;
                    const int k = kc + 2 * (pairs * b + p);
                    for (int j = 0; j < 2 && k + j < ke && more; ++j) {
                        sample(k + j, [&](bool ends) {
                            int s, m;
                            settled_before(w, kc, ke, pairs, b, p, s, m);
                            add(ends, s, k + j - kc - marched, m);
                        });
                        ++marched;
                    }
                }
            }
            if (more) {
                int s, m;
                settled_before(w, kc, ke, pairs, 32, 0, s, m);
                add(active, s, ke - kc - marched, m);
            }
        }
        s_iters += iters;
        s_samples += samples;
        const bool hit = valid && k_first >= 0;
        if (valid && !hit) write_miss<T>(fd, x, y, esc_max);
        s_hits += hit ? 1 : 0;
        warp_push(hit, make_int4(y * fd.W + x, k_first, 0, 0), sc.hits, sc.hit_cap, &sc.ctr->hit_count);
    }
    flush_stat(&sc.ctr->stats[0], s_iters);
    flush_stat(&sc.ctr->stats[8], s_iters);
    flush_stat(&sc.ctr->stats[2], s_samples);
    flush_stat(&sc.ctr->stats[3], s_hits);
    if (RECHECK) flush_stat(&sc.ctr->stats[4], s_rechecks);
}

// ---------------------------------------------------------------------------
// march, paired: two rays per lane, tile slots `lane` and `lane + 32` of a
// 64-ray tile, advanced together in the two halves of float2 registers by the
// paired FP32 instructions.  Same per-ray arithmetic as march_kernel<float>.
// Per ray it keeps only running sums: sum_* (steps stayed bounded, summed over
// samples), max_* (largest escape count - 1) and the first inside sample kf_*;
// the iteration and sample counts follow from them once the ray is done.  The
// escape count of the sample before a hit is classified again by the
// bisection pass, which needs it only for hits.
// ---------------------------------------------------------------------------
template <int SQ, int MOD, bool RECHECK, bool AXIS>
__global__ void __launch_bounds__(kBlock, AXIS ? 5 : 4)  // the general form keeps 24 coefficients per ray pair
    march2_kernel(const __grid_constant__ FrameDesc fd, const Scratch sc)
{
    __shared__ int4 stage[RECHECK ? kBlock / 32 : 1][RECHECK ? kQStage : 1];  // recheck entries, per warp
    int4 *qs = stage[RECHECK ? threadIdx.x >> 5 : 0];
    int left = 0;  // entries staged by the warp's earlier tiles
    const int lane = threadIdx.x & 31;
    const unsigned ntiles = subset_tiles(fd, (unsigned)fd.tiles_x * (unsigned)fd.tiles_y);
    for (;;) {
        unsigned tile = 0;
        if (lane == 0) tile = atomicAdd(&sc.ctr->tile_next, 1u);
        tile = __shfl_sync(kFull, tile, 0);
        if (tile >= ntiles) break;
        tile = subset_tile(fd, tile);
        // counters are added per tile, so none stays live across the march loop
        LaneStats st;
        march2_tile<SQ, MOD, RECHECK, AXIS>(fd, fd.p2, sc, tile, st, qs, &left);
        flush_lane_stats<false>(sc, st, true);
    }
    if (RECHECK) flush_rest(fd, sc, qs, left);
}

// march2_kernel with two samples of each ray per round (march4_tile).  Its
// four sets of iterates take more registers: four CTAs per SM on an axis
// slice, three with the general form's first-iterate coefficients.  The recheck
// form with settled blocks takes three too: at four it spilled, and 16 warps at
// as many places of its longer code stalled on instruction fetch (recheck march
// at 1080p 0.562 / 0.525 ms at four / three).
template <int SQ, int MOD, bool RECHECK, bool AXIS, bool SETTLE>
__global__ void __launch_bounds__(kBlock, AXIS && !(RECHECK && SETTLE) ? 4 : 3) march4_kernel(const __grid_constant__ FrameDesc fd,
                                                                      const Scratch sc)
{
    __shared__ int4 stage[RECHECK ? kBlock / 32 : 1][RECHECK ? kQStage : 1];  // recheck entries, per warp
    int4 *qs = stage[RECHECK ? threadIdx.x >> 5 : 0];
    int left = 0;  // entries staged by the warp's earlier tiles
    __shared__ TileBox box[kBlock / 32];
    const int lane = threadIdx.x & 31;
    const unsigned ntiles = subset_tiles(fd, (unsigned)fd.tiles_x * (unsigned)fd.tiles_y);
    for (;;) {
        unsigned tile = 0;
        if (lane == 0) tile = atomicAdd(&sc.ctr->tile_next, 1u);
        tile = __shfl_sync(kFull, tile, 0);
        if (tile >= ntiles) break;
        tile = subset_tile(fd, tile);
        LaneStats st;
        march4_tile<SQ, MOD, RECHECK, AXIS, false, SETTLE>(fd, fd.p2, sc, tile, st, box[threadIdx.x >> 5], qs, &left);
        flush_lane_stats<false>(sc, st, true);
    }
    if (RECHECK) flush_rest(fd, sc, qs, left);
}

// A small frame's three kernels follow one another within 90 us, of which the
// gaps between them are several (256x256: 88.4 -> 85.3 us).  The two later ones are launched as programmatic
// dependents (launch_after): they are put on the SMs while the one before still
// runs, once all its CTAs have started (start_next), and wait for its end and its
// writes before they read anything (wait_previous).  Neither does anything in a
// kernel launched the usual way.
__device__ __forceinline__ void start_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void wait_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// ---------------------------------------------------------------------------
// split march, for frames with fewer tiles than the GPU has resident warps: a
// work item is one 64-ray tile and one of fd.k_split contiguous ranges of the
// samples, so that more warps share a small frame.  Ranges past a ray's first
// inside sample do work the march would not do (less when an earlier range
// has already recorded its hit: the ray is skipped); march_merge_kernel keeps
// only the ranges up to the first inside sample, so outputs and iteration
// counts are the march's.
// ---------------------------------------------------------------------------
template <int SQ, int MOD, bool AXIS>
__global__ void __launch_bounds__(kBlock, AXIS ? 5 : 4) march2_split_kernel(const __grid_constant__ FrameDesc fd, const Scratch sc)
{
    start_next();
    const int lane = threadIdx.x & 31;
    const unsigned ntiles = subset_tiles(fd, (unsigned)fd.tiles_x * (unsigned)fd.tiles_y);
    const unsigned items = ntiles * (unsigned)fd.k_split;
    for (;;) {
        unsigned item = 0;
        if (lane == 0) item = atomicAdd(&sc.ctr->tile_next, 1u);
        item = __shfl_sync(kFull, item, 0);
        if (item >= items) break;
        // lower ranges first, so that later ones find the rays they can skip
        const unsigned r = item / ntiles, tile = subset_tile(fd, item % ntiles);
        const int kb = (int)r * fd.k_chunk, ke = min(kb + fd.k_chunk, fd.N + 1);
        LaneStats st;
        march2_tile<SQ, MOD, false, AXIS, true>(fd, fd.p2, sc, tile, st, nullptr, nullptr, kb, ke);
    }
}

// march2_split_kernel with two samples of each ray per round (march4_tile).
template <int SQ, int MOD, bool AXIS>
__global__ void __launch_bounds__(kBlock, AXIS ? 4 : 3) march4_split_kernel(const __grid_constant__ FrameDesc fd,
                                                                            const Scratch sc)
{
    __shared__ TileBox box[kBlock / 32];
    start_next();
    const int lane = threadIdx.x & 31;
    const unsigned ntiles = subset_tiles(fd, (unsigned)fd.tiles_x * (unsigned)fd.tiles_y);
    const unsigned items = ntiles * (unsigned)fd.k_split;
    for (;;) {
        unsigned item = 0;
        if (lane == 0) item = atomicAdd(&sc.ctr->tile_next, 1u);
        item = __shfl_sync(kFull, item, 0);
        if (item >= items) break;
        const unsigned r = item / ntiles, tile = subset_tile(fd, item % ntiles);
        const int kb = (int)r * fd.k_chunk, ke = min(kb + fd.k_chunk, fd.N + 1);
        LaneStats st;
        march4_tile<SQ, MOD, false, AXIS, true, false>(fd, fd.p2, sc, tile, st, box[threadIdx.x >> 5], nullptr, nullptr, kb, ke);
    }
}

// Per pixel: the ranges of the split march in sample order up to the first
// with an inside sample give the pixel's result (a miss's largest escape count,
// or the hit's first inside sample for the bisection pass) and its iterations
// and samples.
__global__ void __launch_bounds__(kBlock) march_merge_kernel(const __grid_constant__ FrameDesc fd, const Scratch sc)
{
    start_next();
    wait_previous();
    const int64_t npx = (int64_t)fd.W * fd.H;
    LaneStats st;
    for (int64_t base = (int64_t)blockIdx.x * blockDim.x; base < npx; base += (int64_t)gridDim.x * blockDim.x) {
        const int64_t pixel = base + threadIdx.x;
        const int x = (int)(pixel % fd.W), y = (int)(pixel / fd.W);
        // only the pixels of the frame's tile subset (dqj_render_tiles)
        const unsigned tile = (unsigned)(y / fd.tile_h) * (unsigned)fd.tiles_x + (unsigned)(x / fd.tile_w);
        const bool part = pixel < npx && tile % (unsigned)fd.tile_parts == (unsigned)fd.tile_part;
        int kf = -1, m = 0;
        unsigned iters = 0, samples = 0;
        // the first range with an inside sample is part_hit (the smallest range
        // that recorded one), so the ranges to read are known up front and
        // their loads need not wait on one another
        const unsigned rh = part ? __ldcg(sc.part_hit + pixel) : 0u;
        const int nr = part ? (rh < (unsigned)fd.k_split ? (int)rh + 1 : fd.k_split) : 0;
#pragma unroll 4
        for (int r = 0; r < nr; ++r) {
            const int4 e = __ldcg(sc.part + (int64_t)r * npx + pixel);
            iters += (unsigned)e.y;
            samples += (unsigned)e.w;
            if (r == (int)rh) kf = e.x;
            else m = max(m, e.z);
        }
        const bool hit = kf >= 0;
        st.iters += iters;
        st.samples += samples;
        st.hits += hit ? 1 : 0;
        if (part && !hit) write_miss<float>(fd, x, y, m);
        warp_push(hit, make_int4((int)pixel, kf, 0, 0), sc.hits, sc.hit_cap, &sc.ctr->hit_count);
    }
    flush_lane_stats<false>(sc, st, true);
}

// ---------------------------------------------------------------------------
// bisect + normal + shade over the hit list
// ---------------------------------------------------------------------------
// Hit lists shorter than group_below take group_lanes (4) lanes per hit
// (bisect_group): one lane per hit would give the launch's warps too few hits
// to hide the bisection's dependent chain.  Longer lists take one lane per hit
// (the least work per hit).  Both forms give the same results.
template <typename T, int SQ, int MOD, bool RECHECK>
__global__ void __launch_bounds__(kBlock) bisect_kernel(const __grid_constant__ FrameDesc fd, const Scratch sc,
                                                        unsigned group_below, int group_lanes)
{
    wait_previous();
    const int lane = threadIdx.x & 31;
    const unsigned nhits = min(*(volatile unsigned *)&sc.ctr->hit_count, sc.hit_cap);
    const int lanes = nhits < group_below ? group_lanes : 1;
    constexpr bool kLate = RECHECK && sizeof(T) == 4;
    __shared__ int4 s_late[kLate ? kBlock / 32 : 1][kLate ? kLateGroup + 32 : 1];  // late hits, per warp
    int4 *late = s_late[kLate ? threadIdx.x >> 5 : 0];
    int nlate = 0;
    const unsigned per = 32u / (unsigned)lanes;
    LaneStats st;
    for (;;) {
        unsigned base = 0;
        if (lane == 0) base = atomicAdd(&sc.ctr->hit_next, per);
        base = __shfl_sync(kFull, base, 0);
        if (base >= nhits) break;
        if (lanes == 4)
            bisect_group<T, SQ, MOD, RECHECK, 4>(fd, sc, base, nhits, st, late, nlate);
        else
            bisect_chunk<T, SQ, MOD, RECHECK>(fd, sc, base, nhits, st, late, nlate);
    }
    if constexpr (kLate)
        if (nlate > 0) late_normals<SQ, MOD, false>(fd, late, nlate, st.niters);
    flush_lane_stats<RECHECK>(sc, st, false);
}

// ---------------------------------------------------------------------------
// FP64 recheck of queued samples and FP64 re-render of disagreeing pixels
// ---------------------------------------------------------------------------
// A queued sample is a march sample its warp's bound left over, or a flagged
// bisection sample.  Most of the latter are bounded or late orbits (every
// sample past late_step is flagged), whose 20 to 30 FP64 steps bound this pass
// until the FP32 bound took the four in five it can prove: 512 x 512, max_iter
// 24, 747k entries: 0.85 -> 0.38 ms.
template <int SQ, int MOD>
__global__ void __launch_bounds__(kBlock) recheck_kernel(const __grid_constant__ FrameDesc fd, const Scratch sc)
{
    __shared__ int4 stage[kBlock / 32][64];
    int4 *qs = stage[threadIdx.x >> 5];
    const int lane = threadIdx.x & 31;
    const unsigned total = *(volatile unsigned *)&sc.ctr->queue_count;
    const unsigned nq = min(total, sc.queue_cap);
    const unsigned warp = (threadIdx.x >> 5) * gridDim.x + blockIdx.x, nwarps = gridDim.x * (blockDim.x >> 5);
    int left = 0;
    for (unsigned base = warp * 32; base < nq; base += nwarps * 32)
        left = recheck_batch<SQ, MOD>(fd, sc, base, nq, qs, left);
    if (lane < left) recheck_entry<SQ, MOD>(fd, sc, qs[lane]);
    // a full queue: pixels whose samples did not fit were flagged by the pushers
}

// FP64 re-render of the pixels queued by the recheck (fixup_pixels), up to five
// per warp at a time, one while there are fewer pixels than warps.  Pixels go to
// warps of different blocks first, so a short list spreads over the SMs.
template <int SQ, int MOD>
__global__ void __launch_bounds__(kBlock) fixup_kernel(const __grid_constant__ FrameDesc fd, const Scratch sc)
{
    __shared__ TileBox box[kBlock / 32];
    __shared__ int4 list[kBlock / 32][kLateGroup];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const unsigned nd = min(*(volatile unsigned *)&sc.ctr->dirty_count, sc.dirty_cap);
    const unsigned warp = wib * gridDim.x + blockIdx.x, nwarps = gridDim.x * (blockDim.x >> 5);
    const unsigned per = min((unsigned)kLateGroup, max(1u, (nd + nwarps - 1u) / nwarps));
    unsigned long long its = 0, npx = 0;
    for (unsigned i = warp * per; i < nd; i += nwarps * per)
        fixup_pixels<SQ, MOD>(fd, sc, i, (int)min(per, nd - i), box[wib], list[wib], its, npx);
    const unsigned long long v = warp_sum(its), p = warp_sum(npx);
    if (lane == 0) {
        if (v) atomicAdd(&sc.ctr->stats[6], v);
        if (p) atomicAdd(&sc.ctr->stats[5], p);
    }
}

// Lanes per hit of a short hit list, and the hit-list length below which a
// list counts as short: fewer hits than 32 per resident warp of the bisection
// launch (capb CTAs of four warps).  DQJ_BISECT_GROUP = 1 or 4 forces that
// many lanes per hit for every list.  (Eight lanes per hit, three tree levels
// per round, measured slower than four at every list length.)
int bisect_forced_lanes()
{
    static const int forced = [] {
        const char *e = std::getenv("DQJ_BISECT_GROUP");
        const long v = e ? std::strtol(e, nullptr, 10) : 0L;
        return v == 1 || v == 4 ? (int)v : 0;
    }();
    return forced;
}
int bisect_group_lanes() { return 4; }
unsigned bisect_group_below(int capb)
{
    if (bisect_forced_lanes() == 1) return 0u;
    if (bisect_forced_lanes() > 1) return 0xffffffffu;
    return (unsigned)capb * 4u * 32u;
}

// Launch on st; `dependent`: as a programmatic dependent of the kernel before it.
template <typename... P, typename... A>
void launch_after(bool dependent, void (*kernel)(P...), int grid, cudaStream_t st, A... args)
{
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3(kBlock);
    cfg.stream = st;
    cfg.attrs = &attr;
    cfg.numAttrs = dependent ? 1 : 0;
    cudaLaunchKernelEx(&cfg, kernel, P(args)...);  // the error stays for cudaGetLastError
}

template <int SQ, int MOD, bool RECHECK, bool AXIS, bool SETTLE>
void launch_march4(const FrameDesc &fd, const Scratch &sc, cudaStream_t st, int num_sms, unsigned ntiles)
{
    static std::atomic<int> g{0};
    const int cap = num_sms * resident_per_sm(g, march4_kernel<SQ, MOD, RECHECK, AXIS, SETTLE>);
    const int gm = (int)min((unsigned)cap, (ntiles + 3u) / 4u);
    march4_kernel<SQ, MOD, RECHECK, AXIS, SETTLE><<<gm > 0 ? gm : 1, kBlock, 0, st>>>(fd, sc);
}

template <typename T, int SQ, int MOD, bool RECHECK>
cudaError_t launch_passes(const FrameDesc &fd, const Scratch &sc, cudaStream_t st, int num_sms, cudaEvent_t *ev)
{
    static std::atomic<int> g_march{0}, g_marchg{0}, g_march2a{0}, g_march2g{0}, g_bisect{0};
    const unsigned ntiles = subset_tiles(fd, (unsigned)fd.tiles_x * (unsigned)fd.tiles_y);
    // split frames: not under capture (a captured graph keeps plain edges), nor
    // with an event between the kernels
    bool dependent = false;
    if (ev) cudaEventRecord(ev[0], st);
    if constexpr (sizeof(T) == 4 && !RECHECK) {
        if (fd.march_variant == 1 && fd.k_split > 1) {
            cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
            dependent = !ev && cudaStreamIsCapturing(st, &cap) == cudaSuccess && cap == cudaStreamCaptureStatusNone;
            static std::atomic<int> g_sa{0}, g_sg{0}, g_mg{0};
            const unsigned items = ntiles * (unsigned)fd.k_split;
            if (fd.march_samples == 2) {
                static std::atomic<int> g_s4a{0}, g_s4g{0};
                if (fd.axis_slice) {
                    const int cap = num_sms * resident_per_sm(g_s4a, march4_split_kernel<SQ, MOD, true>);
                    march4_split_kernel<SQ, MOD, true>
                        <<<(int)min((unsigned)cap, (items + 3u) / 4u), kBlock, 0, st>>>(fd, sc);
                } else {
                    const int cap = num_sms * resident_per_sm(g_s4g, march4_split_kernel<SQ, MOD, false>);
                    march4_split_kernel<SQ, MOD, false>
                        <<<(int)min((unsigned)cap, (items + 3u) / 4u), kBlock, 0, st>>>(fd, sc);
                }
            } else if (fd.axis_slice) {
                const int cap = num_sms * resident_per_sm(g_sa, march2_split_kernel<SQ, MOD, true>);
                march2_split_kernel<SQ, MOD, true><<<(int)min((unsigned)cap, (items + 3u) / 4u), kBlock, 0, st>>>(fd, sc);
            } else {
                const int cap = num_sms * resident_per_sm(g_sg, march2_split_kernel<SQ, MOD, false>);
                march2_split_kernel<SQ, MOD, false><<<(int)min((unsigned)cap, (items + 3u) / 4u), kBlock, 0, st>>>(fd, sc);
            }
            const unsigned npx = (unsigned)fd.W * (unsigned)fd.H;
            const int capm = num_sms * resident_per_sm(g_mg, march_merge_kernel);
            launch_after(dependent, march_merge_kernel, (int)min((unsigned)capm, (npx + kBlock - 1) / kBlock), st, fd, sc);
        }
    }
    if constexpr (sizeof(T) == 4) {
        if (fd.march_variant == 1 && !(fd.k_split > 1 && !RECHECK)) {
            // a persistent grid per instantiation: the axis and general forms
            // have different register counts and resident CTAs per SM
            if (fd.march_samples == 2) {
                if (fd.axis_slice)
                    fd.settle ? launch_march4<SQ, MOD, RECHECK, true, true>(fd, sc, st, num_sms, ntiles)
                              : launch_march4<SQ, MOD, RECHECK, true, false>(fd, sc, st, num_sms, ntiles);
                else
                    fd.settle ? launch_march4<SQ, MOD, RECHECK, false, true>(fd, sc, st, num_sms, ntiles)
                              : launch_march4<SQ, MOD, RECHECK, false, false>(fd, sc, st, num_sms, ntiles);
            } else if (fd.axis_slice) {
                const int cap = num_sms * resident_per_sm(g_march2a, march2_kernel<SQ, MOD, RECHECK, true>);
                const int gm = (int)min((unsigned)cap, (ntiles + 3u) / 4u);
                march2_kernel<SQ, MOD, RECHECK, true><<<gm > 0 ? gm : 1, kBlock, 0, st>>>(fd, sc);
            } else {
                const int cap = num_sms * resident_per_sm(g_march2g, march2_kernel<SQ, MOD, RECHECK, false>);
                const int gm = (int)min((unsigned)cap, (ntiles + 3u) / 4u);
                march2_kernel<SQ, MOD, RECHECK, false><<<gm > 0 ? gm : 1, kBlock, 0, st>>>(fd, sc);
            }
        }
    }
    if (sizeof(T) != 4 || fd.march_variant != 1) {
        if (fd.axis_slice) {
            const int cap = num_sms * resident_per_sm(g_march, march_kernel<T, SQ, MOD, RECHECK, true>);
            const int gm = (int)min((unsigned)cap, (ntiles + 3u) / 4u);
            march_kernel<T, SQ, MOD, RECHECK, true><<<gm > 0 ? gm : 1, kBlock, 0, st>>>(fd, sc);
        } else {
            const int cap = num_sms * resident_per_sm(g_marchg, march_kernel<T, SQ, MOD, RECHECK, false>);
            const int gm = (int)min((unsigned)cap, (ntiles + 3u) / 4u);
            march_kernel<T, SQ, MOD, RECHECK, false><<<gm > 0 ? gm : 1, kBlock, 0, st>>>(fd, sc);
        }
    }
    if (ev) cudaEventRecord(ev[1], st);
    const int capb = num_sms * resident_per_sm(g_bisect, bisect_kernel<T, SQ, MOD, RECHECK>);
    const unsigned maxw = ((unsigned)fd.W * (unsigned)fd.H + 31u) / 32u;
    const int gb = (int)min((unsigned)capb, (maxw + 3u) / 4u);
    launch_after(dependent, bisect_kernel<T, SQ, MOD, RECHECK>, gb > 0 ? gb : 1, st, fd, sc, bisect_group_below(capb),
                 bisect_group_lanes());
    if (ev) cudaEventRecord(ev[2], st);
    if (RECHECK) {
        static std::atomic<int> g_re{0}, g_fx{0};
        recheck_kernel<SQ, MOD><<<num_sms * resident_per_sm(g_re, recheck_kernel<SQ, MOD>), kBlock, 0, st>>>(fd, sc);
        if (ev) cudaEventRecord(ev[3], st);
        fixup_kernel<SQ, MOD><<<num_sms * resident_per_sm(g_fx, fixup_kernel<SQ, MOD>), kBlock, 0, st>>>(fd, sc);
        if (ev) cudaEventRecord(ev[4], st);
    } else if (ev) {
        cudaEventRecord(ev[3], st);
        cudaEventRecord(ev[4], st);
    }
    return cudaGetLastError();
}

template <int SQ, int MOD>
cudaError_t launch_mode(const FrameDesc &fd, const Scratch &sc, cudaStream_t st, int num_sms, cudaEvent_t *ev)
{
    switch (fd.precision) {
    case 0: return launch_passes<float, SQ, MOD, false>(fd, sc, st, num_sms, ev);
    case 1: return launch_passes<float, SQ, MOD, true>(fd, sc, st, num_sms, ev);
    default: return launch_passes<double, SQ, MOD, false>(fd, sc, st, num_sms, ev);
    }
}

}  // namespace

}  // namespace dqj
