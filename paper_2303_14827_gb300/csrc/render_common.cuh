// render_common.cuh -- device helpers shared by the render kernels and the
// persistent serving kernel: camera ray and box clip, slice map, warp-aggregated
// queue pushes, output writes and shading, and the per-tile bodies of the march
// and bisection passes.
#pragma once

#include <atomic>

#include "dq_math.cuh"
#include "settle.cuh"

namespace dqj {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kBlock = 128;  // 4 warps per CTA

// Resident CTAs of `kernel` per SM at `block` threads, cached in `slot` (one slot
// per kernel instantiation).  The count depends on the kernel's registers and
// shared memory only, so it holds for every device of this single-architecture
// build; callers multiply it by the launching device's SM count.  Threads that
// race on an empty slot compute and store the same value.
template <typename K>
inline int resident_per_sm(std::atomic<int> &slot, K kernel, int block = kBlock)
{
    int v = slot.load(std::memory_order_relaxed);
    if (v > 0) return v;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&v, kernel, block, 0) != cudaSuccess || v < 1) {
        cudaGetLastError();
        return 1;
    }
    slot.store(v, std::memory_order_relaxed);
    return v;
}

// The frame's tile subset (dqj_render_tiles): the number of its tiles out of
// ntiles, and the tile index of the subset's i-th tile.
__host__ __device__ __forceinline__ unsigned subset_tiles(const FrameDesc &fd, unsigned ntiles)
{
    const unsigned part = (unsigned)fd.tile_part, parts = (unsigned)fd.tile_parts;
    return part < ntiles ? (ntiles - part + parts - 1) / parts : 0u;
}
__device__ __forceinline__ unsigned subset_tile(const FrameDesc &fd, unsigned i)
{
    return i * (unsigned)fd.tile_parts + (unsigned)fd.tile_part;
}

// Per-lane counters, added to the frame's stats once per warp (DQJ_STAT_*).
struct LaneStats {
    unsigned long long iters = 0, samples = 0, hits = 0, rechecks = 0, niters = 0;
};


template <typename T>
__device__ __forceinline__ const FrameT<T> &frame(const FrameDesc &fd);
template <>
__device__ __forceinline__ const FrameT<float> &frame<float>(const FrameDesc &fd) { return fd.f; }
template <>
__device__ __forceinline__ const FrameT<double> &frame<double>(const FrameDesc &fd) { return fd.d; }

template <typename T>
__device__ __forceinline__ T tinf();
template <>
__device__ __forceinline__ float tinf<float>() { return __int_as_float(0x7f800000); }
template <>
__device__ __forceinline__ double tinf<double>() { return __longlong_as_double(0x7ff0000000000000ll); }

// Pinhole camera ray through pixel centre (x + 0.5, y + 0.5), row 0 at the top,
// and its slab clip against the box, t >= 0.  Returns false when the ray misses
// the box (t_in >= t_out).  The FP64 form follows the reference formula term by
// term; the FP32 form folds the pixel-to-screen map into one FMA per axis.
template <typename T>
__device__ __forceinline__ bool camera_clip(const FrameT<T> &F, int W, int H, int x, int y, T (&d)[3], T &t_in,
                                            T &t_out)
{
    T sx, sy;
    if constexpr (sizeof(T) == 4) {
        sx = dfma(T(x) + T(0.5), F.sxa, F.sxb);
        sy = dfma(T(y) + T(0.5), F.sya, F.syb);
    } else {
        sx = (T(2) * (T(x) + T(0.5)) / T(W) - T(1)) * F.th * F.aspect;
        sy = (T(1) - T(2) * (T(y) + T(0.5)) / T(H)) * F.th;
    }
#pragma unroll
    for (int a = 0; a < 3; ++a) d[a] = F.fwd[a] + sx * F.right[a] + sy * F.upv[a];
    const T len = sqrt(d[0] * d[0] + d[1] * d[1] + d[2] * d[2]);
#pragma unroll
    for (int a = 0; a < 3; ++a) d[a] = d[a] / len;
    T t0 = -tinf<T>(), t1 = tinf<T>();
    bool ok = true;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        if (d[a] == T(0)) {
            if (F.eye[a] < F.bmin[a] || F.eye[a] > F.bmax[a]) ok = false;
        } else {
            T ta = (F.bmin[a] - F.eye[a]) / d[a];
            T tb = (F.bmax[a] - F.eye[a]) / d[a];
            if (ta > tb) {
                const T tmp = ta;
                ta = tb;
                tb = tmp;
            }
            t0 = ta > t0 ? ta : t0;
            t1 = tb < t1 ? tb : t1;
        }
    }
    if (t0 < T(0)) t0 = T(0);
    t_in = t0;
    t_out = t1;
    return ok && (t0 < t1);
}

// D = E d: direction of the ray in the 8-D slice.
template <typename T>
__device__ __forceinline__ void slice_dir(const FrameT<T> &F, const T (&d)[3], T (&D)[8])
{
#pragma unroll
    for (int i = 0; i < 8; ++i) D[i] = dfma(d[0], F.E[0][i], dfma(d[1], F.E[1][i], d[2] * F.E[2][i]));
}

// Warp-aggregated append of one int4 per flagged lane.  All lanes must call.
// Returns true on the lanes whose entry did not fit (the caller falls back).
__device__ __forceinline__ bool warp_push(bool flag, int4 v, int4 *buf, unsigned cap, unsigned *count)
{
    const unsigned m = __ballot_sync(kFull, flag);
    if (m == 0) return false;
    const int lane = threadIdx.x & 31;
    const int leader = __ffs(m) - 1;
    unsigned base = 0;
    if (lane == leader) base = atomicAdd(count, (unsigned)__popc(m));
    base = __shfl_sync(kFull, base, leader);
    if (!flag) return false;
    const unsigned slot = base + __popc(m & ((1u << lane) - 1u));
    if (slot < cap) {
        buf[slot] = v;
        return false;
    }
    return true;
}

// Queue a pixel for an FP64 re-render once per frame.
__device__ __forceinline__ void mark_dirty(const FrameDesc &fd, const Scratch &sc, int pixel)
{
    const uint32_t old = atomicExch(&sc.dirty_flag[pixel], fd.epoch);
    if (old != fd.epoch) {
        const unsigned slot = atomicAdd(&sc.ctr->dirty_count, 1u);
        if (slot < sc.dirty_cap) sc.dirty_list[slot] = pixel;
    }
}

__device__ __forceinline__ unsigned long long warp_sum(unsigned long long v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
    return v;
}

__device__ __forceinline__ void flush_stat(unsigned long long *dst, unsigned long long v)
{
    v = warp_sum(v);
    if ((threadIdx.x & 31) == 0 && v) atomicAdd(dst, v);
}

// flush_stat of a count below 2^51: two warp reductions of 32-bit parts (24 low
// bits, and the rest) instead of ten 64-bit shuffles and additions.
__device__ __forceinline__ void flush_count(unsigned long long *dst, unsigned long long v)
{
    const unsigned lo = __reduce_add_sync(kFull, (unsigned)v & 0xffffffu);
    const unsigned hi = __reduce_add_sync(kFull, (unsigned)(v >> 24));
    if ((threadIdx.x & 31) == 0 && (lo | hi)) atomicAdd(dst, ((unsigned long long)hi << 24) + lo);
}

template <typename T>
__device__ __forceinline__ void write_miss(const FrameDesc &fd, int x, int y, int iter)
{
    const int64_t o = (int64_t)y * fd.pitch + x;
    if (fd.iter) fd.iter[o] = iter;
    if (fd.depth) fd.depth[o] = tinf<float>();
    if (fd.normal) {
        fd.normal[3 * o + 0] = 0.f;
        fd.normal[3 * o + 1] = 0.f;
        fd.normal[3 * o + 2] = 0.f;
    }
    if (fd.rgba) *reinterpret_cast<uchar4 *>(fd.rgba + 4 * o) = make_uchar4(0, 0, 0, 0);
}

__device__ __forceinline__ unsigned char to_u8(double v)
{
    double x = floor(255.0 * v + 0.5);
    x = x < 0.0 ? 0.0 : (x > 255.0 ? 255.0 : x);
    return (unsigned char)x;
}
__device__ __forceinline__ unsigned char to_u8(float v)
{
    float x = floorf(255.f * v + 0.5f);
    x = x < 0.f ? 0.f : (x > 255.f ? 255.f : x);
    return (unsigned char)x;
}

// Largest normal-field value used for a gradient, 2^100 (exact in float and
// double): larger or non-finite field values select the fallback normal -d.
__device__ __forceinline__ float normal_fmax(float) { return 1.2676506002282294e30f; }
__device__ __forceinline__ double normal_fmax(double) { return 1.2676506002282294e30; }

// Normalise the central-difference gradient (fallback -d when guard is set or
// the gradient vanishes), shade with the ambient and diffuse terms of Eq. phong
// and write a hit pixel.  The gradient is scaled by its largest component first
// so that its squared length cannot overflow.
template <typename T>
__device__ __forceinline__ void shade_write(const FrameDesc &fd, const FrameT<T> &F, int x, int y, int iter,
                                            T depth, const T (&g)[3], bool guard, const T (&d)[3])
{
    T n[3];
    const T s = fmax(fabs(g[0]), fmax(fabs(g[1]), fabs(g[2])));
    if (guard || !(s > T(0))) {
        n[0] = -d[0];
        n[1] = -d[1];
        n[2] = -d[2];
    } else {
        const T g0 = g[0] / s, g1 = g[1] / s, g2 = g[2] / s;
        const T gl = sqrt(g0 * g0 + g1 * g1 + g2 * g2);
        n[0] = g0 / gl;
        n[1] = g1 / gl;
        n[2] = g2 / gl;
    }
    T ndl = n[0] * F.light[0] + n[1] * F.light[1] + n[2] * F.light[2];
    T spec = T(0);
    if (F.ks > T(0) && ndl > T(0)) {  // reflected light r = 2n(n.l) - l against v = -d
        const T rv = -((T(2) * ndl * n[0] - F.light[0]) * d[0] + (T(2) * ndl * n[1] - F.light[1]) * d[1] +
                       (T(2) * ndl * n[2] - F.light[2]) * d[2]);
        if (rv > T(0)) spec = F.ks * pow(rv, F.shin);
    }
    ndl = ndl > T(0) ? ndl : T(0);
    T v = F.ka + F.kd * ndl + spec;
    v = v < T(0) ? T(0) : (v > T(1) ? T(1) : v);
    const int64_t o = (int64_t)y * fd.pitch + x;
    if (fd.iter) fd.iter[o] = iter;
    if (fd.depth) fd.depth[o] = (float)depth;
    if (fd.normal) {
        fd.normal[3 * o + 0] = (float)n[0];
        fd.normal[3 * o + 1] = (float)n[1];
        fd.normal[3 * o + 2] = (float)n[2];
    }
    if (fd.rgba)
        *reinterpret_cast<uchar4 *>(fd.rgba + 4 * o) =
            make_uchar4(to_u8(v * F.albedo[0]), to_u8(v * F.albedo[1]), to_u8(v * F.albedo[2]), 255);
}

// A pixel's camera ray eye + tau w, not normalised (a sample's position depends
// only on its fraction of the ray's part inside the box).
template <typename T>
__device__ __forceinline__ void ray_w(const FrameT<T> &F, int x, int y, T (&w)[3])
{
    const T sx = dfma(T(x) + T(0.5), F.sxa, F.sxb), sy = dfma(T(y) + T(0.5), F.sya, F.syb);
#pragma unroll
    for (int a = 0; a < 3; ++a) w[a] = dfma(sy, F.upv[a], dfma(sx, F.right[a], F.fwd[a]));
}

// FP64 entry and exit (tau) of a ray that crosses the box.  Only the faces that
// can decide are intersected in FP64, one or two of three as a rule, and each
// needs one reciprocal, formed by two Newton steps on an FP32 one (relative error
// 1e-7, 1e-14, then rounding).  A face can decide unless its FP32 parameter lies
// behind another's by more than their rounding: 8 u of itself (the ray, its
// reciprocal, the product), and |1/w| times 3 u of the face's and the eye's
// coordinates, whose difference cancels where the eye is next to the face.  FP64
// runs at 1/64 of the FP32 rate here: with the normalised direction, three
// reciprocals and the whole clip a recheck took about 130 FP64 instructions, in
// this form about 85.
__device__ __forceinline__ void ray_clip64(const FrameDesc &fd, const double (&w)[3], double &t0, double &t1)
{
    const FrameT<float> &f = fd.f;
    const FrameT<double> &F = fd.d;
    constexpr float u = 5.9604645e-8f;
    // per axis, the latest the entry and the earliest the exit can be
    float rw[3], in_lo = 0.f, out_hi = tinf<float>(), entry[3], exit[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const float wf = (float)w[a];
        const bool flat = !(fabsf(wf) > 1e-30f);  // parallel to the slab, inside it
        rw[a] = 1.f / wf;
        const float p = (f.bmin[a] - f.eye[a]) * rw[a], q = (f.bmax[a] - f.eye[a]) * rw[a];
        const float near = fminf(p, q), far = fmaxf(p, q);
        const float abs_r = 3.f * u * fabsf(rw[a]) * (fabsf(f.eye[a]) + fmaxf(fabsf(f.bmin[a]), fabsf(f.bmax[a])));
        const float dn = fmaf(8.f * u, fabsf(near), abs_r), df = fmaf(8.f * u, fabsf(far), abs_r);
        entry[a] = flat ? -tinf<float>() : near + dn;
        exit[a] = flat ? tinf<float>() : far - df;
        if (!flat) {
            in_lo = fmaxf(in_lo, near - dn);
            out_hi = fminf(out_hi, far + df);
        }
    }
    t0 = 0.0;
    t1 = tinf<double>();
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const bool ci = !(entry[a] < in_lo), co = !(exit[a] > out_hi);  // an overflowed one is intersected
        if (ci || co) {
            double r = (double)rw[a];
            r = fma(r, fma(-w[a], r, 1.0), r);
            r = fma(r, fma(-w[a], r, 1.0), r);
            const bool up = rw[a] > 0.f;
            if (ci) t0 = fmax(t0, ((up ? F.bmin[a] : F.bmax[a]) - F.eye[a]) * r);
            if (co) t1 = fmin(t1, ((up ? F.bmax[a] : F.bmin[a]) - F.eye[a]) * r);
        }
    }
}

// FP64 slice point of one queued sample {pixel, k | b << 16, path, n32} on its
// FP64 ray: a march sample k (with x | y << 16 in place of the path), or
// bisection level b of the bracket (k - 1, k) replayed from the path bits.
// Positions may differ from the reference formula's in the last place, as the
// FP64 iteration's contracted FMAs already do.  Components 3..7 of an
// axis-aligned slice are set to zero.
__device__ __forceinline__ void entry_point64(const FrameDesc &fd, int4 e, double (&z)[8])
{
    const FrameT<double> &F = fd.d;
    const int pixel = e.x, k = e.y & 0xffff, b = e.y >> 16;
    const bool march = b == kMarchSample;
    const int x = march ? e.z & 0xffff : pixel % fd.W, y = march ? e.z >> 16 : pixel / fd.W;
    double w[3], t_in, t_out;
    ray_w<double>(F, x, y, w);
    ray_clip64(fd, w, t_in, t_out);
    const double delta = (t_out - t_in) * fd.inv_n;
    double t;
    if (march) {
        t = fma((double)k, delta, t_in);
    } else {
        double lo = fma((double)(k - 1), delta, t_in), hi = fma((double)k, delta, t_in);
        for (int l = 0; l < b; ++l) {
            const double mid = lo + 0.5 * (hi - lo);
            if ((unsigned)e.z >> l & 1u)
                lo = mid;
            else
                hi = mid;
        }
        t = lo + 0.5 * (hi - lo);
    }
    // the point in the scene first, then its slice image: eye + t w cancels to a
    // point of the box before its rounding is spread over the components (origin
    // + E eye + t E w took as many operations, and erred 1.2 times as far on
    // general slices)
    double p[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) p[a] = fma(t, w[a], F.eye[a]);
    auto comp = [&](int j) { z[j] = fma(p[2], F.E[2][j], fma(p[1], F.E[1][j], fma(p[0], F.E[0][j], F.O[j]))); };
#pragma unroll
    for (int j = 0; j < 3; ++j) comp(j);
#pragma unroll
    for (int j = 3; j < 8; ++j) z[j] = 0.0;
    if (!fd.axis_slice) {
#pragma unroll
        for (int j = 3; j < 8; ++j) comp(j);
    }
}

// One step of the bounds (er, ed) of an orbit's distance from the exact one, from
// the norms of its halves (see count_bound).  With the dual-number modulus
// (MOD 1) no test sees the dual half, and the real half does not depend on it.
template <int SQ, int MOD>
__device__ __forceinline__ void bound_step(float &er, float &ed, float ar, float ad, float round)
{
    const float ner = fmaf(er, fmaf(2.f, ar, er), round);
    if (MOD == 0) {
        if (SQ == 0)
            ed = fmaf(2.f, fmaf(ar, ed, fmaf(ad, er, er * ed)), round);
        else
            ed = fmaf(ed, fmaf(2.f, ad, ed), round);
    }
    er = ner;
}

// Escape count of a sample by its FP32 orbit beside a bound (er, ed) of that
// orbit's distance from the exact one on the real and dual halves: the given
// rounding of the starting point z, then per step
//     er <- 2 |z_r| er + er^2 + rounding,  ed <- 2 (|z_r| ed + |z_d| er + er ed) + rounding
// (algebraic square; quaternion norms multiply), so a step's exact modulus lies
// within 2 (|z_r| er + |z_d| ed) + er^2 + ed^2 of the FP32 one.  Where every
// step decides clear of that, the count is the exact sample's and FP64 can only
// give the same: `certain`.  Otherwise the count returned means nothing.
//
// Rounding of a step, u = 2^-24, term by term of dq_iter: the real half errs by
// at most u (5.1 |z_r|^2 + 4.3 |c|), the dual half by u (4.5 (|z_r|^2 + |z_d|^2)
// + 4 |c|) (the rounding of c included); the modulus by 8 u of itself.
template <int SQ, int MOD>
__device__ __forceinline__ int count_bound(const FrameDesc &fd, float (&z)[8], float er, float ed, bool &certain)
{
    const FrameT<float> &F = fd.f;
    constexpr float u = 5.9604645e-8f;
    certain = false;
    if (!fd.bounds) return 0;
    const float hi = F.R2 * (1.f + 2.f * u), lo = F.R2 * (1.f - 2.f * u);
    float sp = dq_sp<float>(z);
    float r2 = fmaf(z[0], z[0], sp), d2 = fmaf(z[7], z[7], fmaf(z[6], z[6], fmaf(z[5], z[5], z[4] * z[4])));
    float ar = sqrt_approx(r2), ad = sqrt_approx(d2);
    certain = true;
#pragma unroll 1
    for (int n = 1; n <= fd.max_iter; ++n) {
        const float round = 5.6f * u * ((MOD == 0 ? r2 + d2 : r2) + fd.settle_cn);
        bound_step<SQ, MOD>(er, ed, ar, ad, round);
        dq_iter<float, SQ, MOD>(z, z, sp, F.c);
        r2 = fmaf(z[0], z[0], sp);
        d2 = fmaf(z[7], z[7], fmaf(z[6], z[6], fmaf(z[5], z[5], z[4] * z[4])));
        ar = sqrt_approx(r2);
        ad = sqrt_approx(d2);
        const float m = MOD == 0 ? r2 + d2 : r2;
        // 1 % covers the roundings of the bound itself
        float dev = er * fmaf(2.f, ar, er);
        if (MOD == 0) dev = fmaf(ed, fmaf(2.f, ad, ed), dev);
        dev = fmaf(1.01f, dev, 10.f * u * m);
        if (m - dev > hi) return n;
        if (!(m + dev < lo)) {
            certain = false;
            return 0;
        }
    }
    return 0;
}

// count_bound of a FP64 point: its FP32 image lies within u of every component.
template <int SQ, int MOD>
__device__ __forceinline__ int count_bound64(const FrameDesc &fd, const double (&z64)[8], bool &certain)
{
    float z[8];
#pragma unroll
    for (int j = 0; j < 3; ++j) z[j] = (float)z64[j];
#pragma unroll
    for (int j = 3; j < 8; ++j) z[j] = 0.f;
    if (!fd.axis_slice) {
#pragma unroll
        for (int j = 3; j < 8; ++j) z[j] = (float)z64[j];
    }
    float n2 = z[0] * z[0];
#pragma unroll
    for (int j = 1; j < 8; ++j) n2 = fmaf(z[j], z[j], n2);
    const float e0 = 6.1e-8f * sqrt_approx(n2);
    return count_bound<SQ, MOD>(fd, z, e0, e0, certain);
}

// A sum of products kept in two floats h + l: every product's and every
// addition's rounding error is computed exactly by FMA and two-sum (Dekker 1971,
// Knuth) and gathered in l, whose own roundings are of the order u^2 of the
// terms.
struct Sum2 {
    float h, l;
    __device__ __forceinline__ void add(float p, float e)
    {
        // the _rn forms are never contracted into an FMA
        const float s = __fadd_rn(h, p), b = __fsub_rn(s, h);
        l += __fadd_rn(__fsub_rn(h, __fsub_rn(s, b)), __fsub_rn(p, b)) + e;
        h = s;
    }
    __device__ __forceinline__ void add_product(float ah, float al, float bh, float bl)
    {
        const float p = __fmul_rn(ah, bh);
        add(p, fmaf(ah, bl, fmaf(al, bh, fmaf(ah, bh, -p))));
    }
    __device__ __forceinline__ void store(float &oh, float &ol) const
    {
        oh = __fadd_rn(h, l);
        ol = __fsub_rn(l, __fsub_rn(oh, h));
    }
};

// count_bound of a FP64 point with the orbit in two floats per component (about
// 48 bits): for the samples whose FP32 orbit cannot decide, late orbits and samples next to the
// surface above all.  A step takes about 260 FP32 instructions, against 27 FP64
// instructions that hold the FP64 pipe for 1,728 cycles (512 x 512, max_iter 24:
// recheck pass 0.38 -> 0.18 ms).  The rounding of a step is below 30 u^2 of its
// terms, the bound takes 128 u^2 of |z_r|^2 + |z_d|^2 + |c|; the modulus needs the high
// parts only (14 u of itself), unless R^2 lies as close as that.
template <int SQ, int MOD>
__device__ __forceinline__ int count_bound2(const FrameDesc &fd, const double (&z64)[8], bool &certain)
{
    constexpr float u = 5.9604645e-8f;
    constexpr int nc = MOD == 0 ? 8 : 4;  // components that a test can see
    certain = false;
    if (!fd.bounds) return 0;
    const float R2 = fd.f.R2, hi = R2 * (1.f + 2.f * u), lo = R2 * (1.f - 2.f * u);
    float zh[8], zl[8];
#pragma unroll
    for (int j = 0; j < nc; ++j) {
        zh[j] = zl[j] = 0.f;
        if (j < 3 || !fd.axis_slice) {
            zh[j] = (float)z64[j];
            zl[j] = (float)(z64[j] - (double)zh[j]);
        }
    }
    auto norms = [&](float &r2, float &d2) {
        r2 = fmaf(zh[3], zh[3], fmaf(zh[2], zh[2], fmaf(zh[1], zh[1], zh[0] * zh[0])));
        d2 = MOD == 0 ? fmaf(zh[7], zh[7], fmaf(zh[6], zh[6], fmaf(zh[5], zh[5], zh[4] * zh[4]))) : 0.f;
    };
    float r2, d2;
    norms(r2, d2);
    float er = 4.f * u * u * (r2 + d2 + 1.f), ed = er;
    certain = true;
#pragma unroll 1
    for (int n = 1; n <= fd.max_iter; ++n) {
        bound_step<SQ, MOD>(er, ed, sqrt_approx(r2), sqrt_approx(d2), 128.f * u * u * (r2 + d2 + fd.settle_cn));
        float oh[8], ol[8];
        // component i starts from c_i
        auto from_c = [&](int i) {
            const float ch = fd.f.c[i];
            return Sum2{ch, (float)(fd.d.c[i] - (double)ch)};
        };
        const float t0h = zh[0] + zh[0], t0l = zl[0] + zl[0];
        {
            Sum2 a = from_c(0);
            a.add_product(zh[0], zl[0], zh[0], zl[0]);
#pragma unroll
            for (int i = 1; i < 4; ++i) a.add_product(-zh[i], -zl[i], zh[i], zl[i]);
            a.store(oh[0], ol[0]);
        }
#pragma unroll
        for (int i = 1; i < 4; ++i) {
            Sum2 a = from_c(i);
            a.add_product(t0h, t0l, zh[i], zl[i]);
            a.store(oh[i], ol[i]);
        }
        if (MOD == 0) {
            const float s0h = zh[4] + zh[4], s0l = zl[4] + zl[4];
            Sum2 a = from_c(4);
            if (SQ == 0) {
                a.add_product(t0h, t0l, zh[4], zl[4]);
#pragma unroll
                for (int i = 1; i < 4; ++i) a.add_product(-2.f * zh[i], -2.f * zl[i], zh[4 + i], zl[4 + i]);
            } else {
                a.add_product(zh[4], zl[4], zh[4], zl[4]);
#pragma unroll
                for (int i = 5; i < 8; ++i) a.add_product(-zh[i], -zl[i], zh[i], zl[i]);
            }
            a.store(oh[4], ol[4]);
#pragma unroll
            for (int i = 5; i < 8; ++i) {
                Sum2 b = from_c(i);
                if (SQ == 0) {
                    b.add_product(t0h, t0l, zh[i], zl[i]);
                    b.add_product(s0h, s0l, zh[i - 4], zl[i - 4]);
                } else {
                    b.add_product(s0h, s0l, zh[i], zl[i]);
                }
                b.store(oh[i], ol[i]);
            }
        }
#pragma unroll
        for (int i = 0; i < nc; ++i) {
            zh[i] = oh[i];
            zl[i] = ol[i];
        }
        norms(r2, d2);
        const float m = r2 + d2;
        float dev = er * fmaf(2.f, sqrt_approx(r2), er);
        if (MOD == 0) dev = fmaf(ed, fmaf(2.f, sqrt_approx(d2), ed), dev);
        dev = fmaf(1.01f, dev, 14.f * u * m);
        if (m - dev > hi) return n;
        if (!(m + dev < lo)) {
            certain = false;
            return 0;
        }
    }
    return 0;
}

// Escape count of a FP64 slice point, as FP64 evaluation gives it: by the
// two-float orbit where its bound decides, else in FP64.  An axis-aligned
// slice takes the axis form of the first step, whose operations are those of
// dq_iter on the zero components: the same iterate.
template <int SQ, int MOD>
__device__ __forceinline__ int count64(const FrameDesc &fd, double (&z)[8])
{
    bool certain;
    const int n = count_bound2<SQ, MOD>(fd, z, certain);
    if (certain) return n;
    return fd.axis_slice ? classify_scalar_axis<double, SQ, MOD>(z, fd.d, fd.max_iter)
                         : classify_scalar<double, SQ, MOD>(z, fd.d, fd.max_iter);
}

// FP64 recheck of one queued sample: the pixel is queued for an FP64 re-render
// when the sample's FP64 escape count differs from its FP32 one.
template <int SQ, int MOD>
__device__ __forceinline__ void recheck_entry(const FrameDesc &fd, const Scratch &sc, int4 e)
{
    double z[8];
    entry_point64(fd, e, z);
    if (count64<SQ, MOD>(fd, z) != e.w) mark_dirty(fd, sc, e.x);
}

// Lockstep classification of one sample per lane (classify_lockstep), FP64 by
// the bounds first: a lane whose count the FP32 orbit's bound proves needs no
// more, the others take count64.  FP32 samples are classified as they are.
template <typename T, int SQ, int MOD, bool RECHECK>
__device__ __forceinline__ int classify_sample(const FrameDesc &fd, T (&z)[8], bool part, bool &marginal)
{
    if constexpr (sizeof(T) == 8) {
        static_assert(!RECHECK, "the recheck mode classifies in FP32");
        marginal = false;
        bool certain = true;
        int n = 1;
        if (part) n = count_bound64<SQ, MOD>(fd, z, certain);
        if (part && !certain) n = count64<SQ, MOD>(fd, z);
        __syncwarp();
        return n;
    } else {
        return classify_lockstep<T, SQ, MOD, RECHECK>(z, frame<T>(fd), fd.max_iter, part, marginal);
    }
}

// Is the FP32 escape count n32 of march sample k of pixel (x, y) certain?  The
// sample is placed by FP32 arithmetic with a bound of its rounding: with
// u = 2^-24, the camera map's constants and three FMAs put w within 8 u m of
// the exact direction, m = 1 + |sx| + |sy| + 2 (|sxb| + |syb|) a bound of its
// terms; a face parameter tau = (face - eye) / w then lies within
// |tau| (8 u m / |w_a| + 8 u) + 3 u (|face| + |eye|) / |w_a| of its exact
// value, and the entry (a maximum) and exit (a minimum) within what the faces'
// upper and lower values give; the position A + tau W adds 8 u of its terms.
// A sample is flagged within 1e-3 of R^2 (by default); after the one to three
// steps of most flagged samples the bound is 1e-5 to 1e-4 of it.
template <int SQ, int MOD, bool AXIS>
__device__ __forceinline__ bool count_certain(const FrameDesc &fd, int x, int y, int k, int n32)
{
    const FrameT<float> &F = fd.f;
    constexpr float u = 5.9604645e-8f;
    float z[8], er, ed;
    {
        float w[3];
        ray_w<float>(F, x, y, w);
        const float sx = fmaf((float)x + 0.5f, F.sxa, F.sxb), sy = fmaf((float)y + 0.5f, F.sya, F.syb);
        // terms of sx and sy: up to twice their largest magnitude over the frame
        const float m = 1.f + fabsf(sx) + fabsf(sy) + 2.f * (fabsf(F.sxb) + fabsf(F.syb));
        const float dw = 8.f * u * m;
        float in = 0.f, in_hi = 0.f, in_lo = 0.f, out = tinf<float>(), out_hi = tinf<float>(), out_lo = tinf<float>();
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const float r = 1.f / w[a];
            const float p = (F.bmin[a] - F.eye[a]) * r, q = (F.bmax[a] - F.eye[a]) * r;
            const float near = fminf(p, q), far = fmaxf(p, q), rel = fmaf(dw, fabsf(r), 8.f * u);
            // the faces and the eye are rounded, and their difference may cancel
            const float abs_r = 3.f * u * fabsf(r) * (fabsf(F.eye[a]) + fmaxf(fabsf(F.bmin[a]), fabsf(F.bmax[a])));
            const float dn = fmaf(rel, fabsf(near), abs_r), df = fmaf(rel, fabsf(far), abs_r);
            in = fmaxf(in, near);
            in_hi = fmaxf(in_hi, near + dn);
            in_lo = fmaxf(in_lo, near - dn);
            out = fminf(out, far);
            out_hi = fminf(out_hi, far + df);
            out_lo = fminf(out_lo, far - df);
        }
        const float tau = fmaf((float)k * (float)fd.inv_n, out - in, in);
        const float dtau = fmaxf(fmaxf(in_hi - in, in - in_lo), fmaxf(out_hi - out, out - out_lo)) + 8.f * u * out;
        const float wn = sqrt_approx(fmaf(w[2], w[2], fmaf(w[1], w[1], w[0] * w[0])));
        // |A| <= settle_an; three FMAs per component of W, one of the position
        er = 1.01f * fmaf(dtau, wn, fmaf(out, dw, 8.f * u * fmaf(out, wn, fd.settle_an)));
        if (!(er < 1e-3f)) return false;  // far camera, grazing ray, overflow: FP64 decides
        ed = AXIS ? 0.f : er;
#pragma unroll
        for (int j = 0; j < (AXIS ? 3 : 8); ++j)
            z[j] = fmaf(tau, fmaf(w[0], F.E[0][j], fmaf(w[1], F.E[1][j], w[2] * F.E[2][j])), F.A[j]);
        if (AXIS) {
#pragma unroll
            for (int j = 3; j < 8; ++j) z[j] = 0.f;
        }
    }
    bool certain;
    const int n = count_bound<SQ, MOD>(fd, z, er, ed, certain);
    return certain && n == n32;
}

// A hit whose normal is evaluated in FP64: pixel x | y << 16, n*, FP64 depth.
__device__ __forceinline__ int4 late_hit(int x, int y, int n_star, double depth)
{
    const long long b = __double_as_longlong(depth);
    return make_int4(x | (y << 16), n_star, (int)(unsigned)(b & 0xffffffffll), (int)(b >> 32));
}

constexpr int kLateGroup = 5;  // hits whose normals a warp evaluates together, six lanes each

// FP64 normals and shading of late hits list[0, count), count <= 5 (all 32 lanes
// call): the six field evaluations of a hit on six lanes, on the hit's FP64 ray.
// An FP64 warp instruction takes the same time for one lane as for 32, so
// evaluating them on the hits' own lanes, or one hit at a time, wasted the
// others (512 x 512, max_iter 24, 55 % of the hits late: bisection pass 0.74 -> 0.63
// ms with the late hits of one step of a warp together, -> 0.52 ms gathered over
// its steps).  REF: the reference formula's order of operations for the points
// (the FP64 re-render), else the render's.  its: DQ iterations, on six-lane
// groups' first lanes.
template <int SQ, int MOD, bool REF>
__device__ __forceinline__ void late_normals(const FrameDesc &fd, const int4 *list, int count, unsigned long long &its)
{
    const FrameT<double> &F = fd.d;
    const int lane = threadIdx.x & 31;
    const int grp = lane / 6, q = lane - 6 * grp;  // lanes 30 and 31 idle
    const bool part = grp < count && grp < kLateGroup;
    int4 e = list[part ? grp : 0];
    const int ns = part ? e.y : 0;
    const int nmax = __reduce_max_sync(kFull, ns);
    const int x = e.x & 0xffff, y = e.x >> 16;
    const double t = __longlong_as_double(((long long)e.w << 32) | (long long)(unsigned)e.z);
    double d[3], t_in, t_out, z[8];
    camera_clip<double>(F, fd.W, fd.H, x, y, d, t_in, t_out);
    const int a = q >> 1;
    const double hs = (q & 1) == 0 ? F.h : -F.h;
    if (REF) {
        double p[3] = {F.eye[0] + t * d[0], F.eye[1] + t * d[1], F.eye[2] + t * d[2]};
#pragma unroll
        for (int i = 0; i < 3; ++i)
            if (i == a) p[i] += hs;
#pragma unroll
        for (int j = 0; j < 8; ++j) z[j] = F.O[j] + p[0] * F.E[0][j] + p[1] * F.E[1][j] + p[2] * F.E[2][j];
    } else {
        double D[8];
        slice_dir<double>(F, d, D);
#pragma unroll
        for (int i = 0; i < 8; ++i) z[i] = fma(hs, F.E[a][i], fma(t, D[i], F.A[i]));
    }
    double sp = dq_sp<double>(z);
#pragma unroll 1
    for (int n = 0; n < nmax; ++n)
        if (n < ns) dq_iter<double, SQ, MOD>(z, z, sp, F.c);
    const double fv = modulus<double, MOD>(z);
    const unsigned bad = __ballot_sync(kFull, !(fv <= normal_fmax(0.0)));
    double f[6];
#pragma unroll
    for (int i = 0; i < 6; ++i) f[i] = __shfl_sync(kFull, fv, min(6 * grp, 24) + i);
    if (part && q == 0) {
        const double g[3] = {f[0] - f[1], f[2] - f[3], f[4] - f[5]};
        its += 6ull * (unsigned)ns;
        shade_write<double>(fd, F, x, y, ns, t, g, ((bad >> (6 * grp)) & 63u) != 0, d);
    }
    __syncwarp();
}

// Add the lanes' late hits to the warp's list (room for kLateGroup - 1 + 32) and
// evaluate full groups; n: entries in the list (warp-uniform).
template <int SQ, int MOD>
__device__ __forceinline__ void push_late(const FrameDesc &fd, bool flag, int4 hit, int4 *list, int &n,
                                          unsigned long long &its)
{
    const unsigned m = __ballot_sync(kFull, flag);
    if (m == 0) return;
    if (flag) list[n + __popc(m & ((1u << (threadIdx.x & 31)) - 1u))] = hit;
    n += __popc(m);
    __syncwarp();
#pragma unroll 1
    while (n >= kLateGroup) {
        n -= kLateGroup;
        late_normals<SQ, MOD, false>(fd, list + n, kLateGroup, its);
    }
}

// Re-render of the pixels dirty_list[first, first + count), count <= 5, by one
// warp (all 32 lanes call), with the oracle's formulas for the sample positions
// (the reference sequence of steps) in FP64; a march or bisection sample is
// classified in FP32 where the rounding bound decides (count_bound), else by
// count64.  The pixels' camera rays are set up on one lane each, their samples
// are taken pixel by pixel: the lanes classify 32 consecutive march samples at
// a time, a ballot finds the first inside one and warp reductions give the
// largest escape count before it, so the result and the iteration count are
// those of the sample-by-sample loop; the bisection runs five levels per round
// across the lanes.  The hits' FP64 normals are evaluated together at the end
// (list: room for five entries).  A warp instruction in FP64 takes the same time
// for one lane as for 32: one pixel at a time the ray setup and the normal took
// most of the pass (1080p, default c, 9,940 pixels: 0.57 -> 0.36 ms).  Adds the
// iterations to its (per lane) and the pixels to npx (lane 0).
template <int SQ, int MOD>
__device__ __forceinline__ void fixup_pixels(const FrameDesc &fd, const Scratch &sc, unsigned first, int count,
                                             TileBox &box, int4 *list, unsigned long long &its,
                                             unsigned long long &npx)
{
    const FrameT<double> &F = fd.d;
    const int lane = threadIdx.x & 31;
    npx += lane == 0 ? (unsigned)count : 0;
    int px = 0, py = 0, hits = 0;
    double pd[3], p_in, p_out;
    {
        const int pixel = lane < count ? __ldcg(sc.dirty_list + first + lane) : 0;
        px = pixel % fd.W;
        py = pixel / fd.W;
    }
    const bool crosses = camera_clip<double>(F, fd.W, fd.H, px, py, pd, p_in, p_out);
    if (lane < count && !crosses) write_miss<double>(fd, px, py, 0);
    unsigned todo = __ballot_sync(kFull, lane < count && crosses);
#pragma unroll 1
    while (todo) {
        const int who = __ffs(todo) - 1;
        todo &= todo - 1;
        const int x = __shfl_sync(kFull, px, who), y = __shfl_sync(kFull, py, who);
        const double d[3] = {__shfl_sync(kFull, pd[0], who), __shfl_sync(kFull, pd[1], who),
                             __shfl_sync(kFull, pd[2], who)};
        const double t_in = __shfl_sync(kFull, p_in, who), t_out = __shfl_sync(kFull, p_out, who);
        const double delta = (t_out - t_in) / (double)fd.N;
        auto slice = [&](double t, double (&z)[8]) {
            auto comp = [&](int j) {
                z[j] = F.O[j] + (F.eye[0] + t * d[0]) * F.E[0][j] + (F.eye[1] + t * d[1]) * F.E[1][j] +
                       (F.eye[2] + t * d[2]) * F.E[2][j];
            };
#pragma unroll
            for (int j = 0; j < 3; ++j) comp(j);
#pragma unroll
            for (int j = 3; j < 8; ++j) z[j] = 0.0;
            if (!fd.axis_slice) {  // (zero on an axis-aligned slice)
#pragma unroll
                for (int j = 3; j < 8; ++j) comp(j);
            }
        };
        const float df[3] = {(float)d[0], (float)d[1], (float)d[2]};
        tile_box(fd, true, df, (float)t_in, (float)t_out, false, df, 0.f, 0.f, box);
        // a sample: by the FP32 orbit where its bound decides, else in FP64
        auto cls_march = [&](double t) {
            double z[8];
            slice(t, z);
            bool certain;
            const int n32 = count_bound64<SQ, MOD>(fd, z, certain);
            return certain ? n32 : count64<SQ, MOD>(fd, z);
        };
        int esc_max = 0, n_prev = 0, k_first = -1;
        unsigned w = 0;
        for (int k0 = 0; k0 <= fd.N; k0 += 32) {
            const int k = k0 + lane;
            const bool part = k <= fd.N;
            // the ray's settled samples (blocks of 16, chunks of 512: see
            // settle.cuh) have their counts; the others are classified
            if (fd.blocks && k0 % kSettleChunk == 0) {
                const int ke = min(k0 + kSettleChunk, fd.N + 1);
                w = fd.axis_slice ? settle_chunk<SQ, MOD, true>(fd, box, k0, ke, kSettlePairs)
                                  : settle_chunk<SQ, MOD, false>(fd, box, k0, ke, kSettlePairs);
            }
            const unsigned word = __shfl_sync(kFull, w, (k % kSettleChunk) / (2 * kSettlePairs));
            int n = (int)((word >> (4 * ((k % (2 * kSettlePairs)) >> 1))) & 15u);
            if (!part) n = 1;
            if (n == 0) n = cls_march(t_in + (double)k * delta);
            __syncwarp();
            const unsigned inside = __ballot_sync(kFull, part && n == 0);
            const int first = inside ? __ffs(inside) - 1 : 32;  // samples before it escaped
            if (part && lane <= first) its += n ? (unsigned)n : (unsigned)fd.max_iter;
            int m = part && lane < first ? n : 0;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(kFull, m, o));
            esc_max = max(esc_max, m);
            if (inside) {
                if (first > 0) n_prev = __shfl_sync(kFull, n, first - 1);  // else: last of the previous chunk
                k_first = k0 + first;
                break;
            }
            n_prev = __shfl_sync(kFull, n, 31);
        }
        if (k_first < 0) {
            if (lane == 0) write_miss<double>(fd, x, y, esc_max);
            continue;
        }
        double depth = t_in;
        int n_star = fd.max_iter;
        if (k_first > 0) {
            double lo = t_in + (double)(k_first - 1) * delta, hi = t_in + (double)k_first * delta;
            n_star = n_prev;
            // Bisection, up to five levels per round: lane j - 1 holds node j of the
            // level tree (node 1 the next midpoint, children 2j: inside -> [lo, mid],
            // 2j + 1: outside -> [mid, hi]), derives its interval with the same
            // operations as the sequential halvings and classifies its midpoint
            // (FP32 first, FP64 when marginal, as the march samples); the path is
            // then replayed, so the bracket is the sequential one.
            for (int b0 = 0; b0 < fd.B; b0 += 5) {
                const int levels = min(5, fd.B - b0);
                const int node = lane + 1;
                const int depth_j = 31 - __clz(node);  // level of the node
                int n = 1;
                if (depth_j < levels) {
                    double l = lo, h = hi;
                    for (int q = depth_j - 1; q >= 0; --q) {  // path bits below the leading one
                        const double mid = l + 0.5 * (h - l);
                        if ((node >> q) & 1)
                            l = mid;
                        else
                            h = mid;
                    }
                    n = cls_march(l + 0.5 * (h - l));
                }
                int cur = 1;
                for (int q = 0; q < levels; ++q) {
                    const int nq = __shfl_sync(kFull, n, cur - 1);
                    const double mid = lo + 0.5 * (hi - lo);
                    if (lane == 0) its += nq ? (unsigned)nq : (unsigned)fd.max_iter;
                    if (nq == 0) {
                        hi = mid;
                        cur = 2 * cur;
                    } else {
                        lo = mid;
                        n_star = nq;
                        cur = 2 * cur + 1;
                    }
                }
            }
            depth = lo + 0.5 * (hi - lo);
        }
        if (lane == 0) list[hits] = late_hit(x, y, n_star, depth);
        ++hits;
    }
    __syncwarp();
    if (hits) late_normals<SQ, MOD, true>(fd, list, hits, its);
}

// Device clock in nanoseconds, for the time limits of bounded waits.
__device__ __forceinline__ unsigned long long globaltimer_ns()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
    return t;
}

// Recheck entries of one warp are staged in shared memory.  At the end of its
// tile the warp drops those whose FP32 count a rounding bound proves
// (recheck_staged); the others go to the frame's queue for the recheck pass, in
// blocks of 32 (one atomic).  A tile that fills the stage (kQStage entries per
// warp; a round adds at most 128) appends the staged entries to the queue as
// they are.
constexpr int kQStage = 320;
// Ray parameter of a half without a sample in the recheck march: its first
// iterate overflows (modulus +inf) and the later ones are infinite or NaN, so
// its distance from R^2 never falls within a recheck band.
constexpr float kFarT = 1e18f;

// Entry `at` of the recheck queue.  One beyond the queue's capacity is counted as
// an overflow, and its pixel is re-rendered in FP64 instead.
__device__ __forceinline__ void queue_entry(const FrameDesc &fd, const Scratch &sc, unsigned at, int4 e)
{
    if (at < sc.queue_cap) {
        sc.queue[at] = e;
    } else {
        atomicAdd(&sc.ctr->stats[7], 1ull);
        mark_dirty(fd, sc, e.x);
    }
}

// Append a warp's staged entries qs[0, qn) to the recheck queue (qn warp-uniform)
// and count those from `counted` on as rechecks.
__device__ __forceinline__ void flush_staged(const FrameDesc &fd, const Scratch &sc, const int4 *qs, int qn,
                                             int counted)
{
    const int lane = threadIdx.x & 31;
    __syncwarp();
    unsigned base = 0;
    if (lane == 0) {
        base = atomicAdd(&sc.ctr->queue_count, (unsigned)qn);
        atomicAdd(&sc.ctr->stats[4], (unsigned long long)(qn - counted));
    }
    base = __shfl_sync(kFull, base, 0);
    for (int i = lane; i < qn; i += 32) {
        queue_entry(fd, sc, base + (unsigned)i, qs[i]);
    }
    __syncwarp();
}

// Recheck of a warp's staged entries qs[0, qn) (qn warp-uniform), counted as
// rechecks from entry `counted` on: entries whose FP32 count is certain are done;
// the others are gathered at the front and appended to the frame's queue 32 at a
// time, for the recheck pass.  (Evaluating them here put the FP64 and two-float
// code between a warp's tiles: instruction fetch then stalled the march, 0.76
// against 0.60 ms at 1080p, 1.51 against 0.97 ms on a random slice.)  Returns how many are left in qs (fewer than 32);
// they stay staged for the warp's next tile (flush_rest after its last).
template <int SQ, int MOD, bool AXIS>
__device__ __forceinline__ int recheck_staged(const FrameDesc &fd, const Scratch &sc, int4 *qs, int qn, int counted)
{
    const int lane = threadIdx.x & 31;
    __syncwarp();
    if (lane == 0) atomicAdd(&sc.ctr->stats[4], (unsigned long long)(qn - counted));
    int out = counted;
    for (int base = counted; base < qn; base += 32) {
        const int i = base + lane;
        int4 e = make_int4(0, 0, 0, 0);
        bool keep = false;
        if (i < qn) {
            e = qs[i];
            keep = !count_certain<SQ, MOD, AXIS>(fd, e.z & 0xffff, e.z >> 16, e.y & 0xffff, e.w);
        }
        const unsigned m = __ballot_sync(kFull, keep);
        if (keep) qs[out + __popc(m & ((1u << lane) - 1u))] = e;  // out <= base: read by now
        out += __popc(m);
        __syncwarp();
        if (out >= 32) {  // fewer than 32 were left, at most 32 came: one batch
            out -= 32;
            const int4 v = qs[out + lane];
            unsigned at = 0;
            if (lane == 0) at = atomicAdd(&sc.ctr->queue_count, 32u);
            queue_entry(fd, sc, __shfl_sync(kFull, at, 0) + lane, v);
            __syncwarp();
        }
    }
    return out;
}

// Recheck of queue entries [base, base + 32) clipped to nq by one warp (all 32
// lanes call), positions in FP64: entries whose FP32 count the rounding bound
// proves are done, the others join those in qs[0, left) and are evaluated in
// FP64 in full batches.  Returns the new number left in qs (room for 64).
template <int SQ, int MOD>
__device__ __forceinline__ int recheck_batch(const FrameDesc &fd, const Scratch &sc, unsigned base, unsigned nq,
                                             int4 *qs, int left)
{
    const int lane = threadIdx.x & 31;
    int4 e = make_int4(0, 0, 0, 0);
    bool keep = false;
    if (base + lane < nq) {
        e = __ldcg(sc.queue + base + lane);
        double z[8];
        entry_point64(fd, e, z);
        bool certain;
        const int n = count_bound64<SQ, MOD>(fd, z, certain);
        keep = !(certain && n == e.w);
    }
    const unsigned m = __ballot_sync(kFull, keep);
    if (keep) qs[left + __popc(m & ((1u << lane) - 1u))] = e;
    left += __popc(m);
    __syncwarp();
    if (left >= 32) {
        left -= 32;
        recheck_entry<SQ, MOD>(fd, sc, qs[left + lane]);
        __syncwarp();
    }
    return left;
}

// The entries a warp has left (already counted), to the recheck queue.
__device__ __forceinline__ void flush_rest(const FrameDesc &fd, const Scratch &sc, const int4 *qs, int qn)
{
    const int lane = threadIdx.x & 31;
    __syncwarp();
    unsigned base = 0;
    if (lane == 0 && qn > 0) base = atomicAdd(&sc.ctr->queue_count, (unsigned)qn);
    base = __shfl_sync(kFull, base, 0);
    if (lane < qn) queue_entry(fd, sc, base + (unsigned)lane, qs[lane]);
    __syncwarp();
}

// One 64-ray tile of the paired march (see march2_kernel); all 32 lanes call.
// A lane holds tile slots `lane` and `lane + 32`.  RECHECK: qs is the warp's
// staging buffer of kQStage entries in shared memory, filtered by a rounding bound
// at the end of the tile (recheck_staged); *left of them stay staged for the warp's
// next tile.  SPLIT: only samples
// [kb, ke) of each ray, with the range's partial result written to sc.part
// (range r = kb / fd.k_chunk) for march_merge_kernel instead of the outputs;
// a ray for which a lower range has already found an inside sample is
// skipped (the merge stops at that range), and a range that finds one records
// itself in sc.part_hit.
template <int SQ, int MOD, bool RECHECK, bool AXIS = false, bool SPLIT = false>
__device__ __forceinline__ void march2_tile(const FrameDesc &fd, const PairConsts &P, const Scratch &sc, unsigned tile,
                                            LaneStats &st, int4 *qs = nullptr, int *left = nullptr, int kb = 0,
                                            int ke = 0)
{
    const FrameT<float> &F = fd.f;
    const int lane = threadIdx.x & 31;
    const int N = fd.N, max_iter = fd.max_iter;
    const int tx = (int)(tile % (unsigned)fd.tiles_x), ty = (int)(tile / (unsigned)fd.tiles_x);
    // pixel of tile slot s; formed again at the end of the tile rather than kept
    // live across the march loop (the recheck mode keeps the linear indices)
    auto px = [&](int slot) { return tx * fd.tile_w + slot % fd.tile_w; };
    auto py = [&](int slot) { return ty * fd.tile_h + slot / fd.tile_w; };
    int pixa = 0, pixb = 0, xya = 0, xyb = 0;
    bool acta, actb, skipa = false, skipb = false;
    // Axis-aligned slice: zeta_0 = A + t D (components 0..2).  Otherwise the
    // first-iterate form (first_iterate_coeffs): zeta_1 = Q0 + s (Q1 + s Q2),
    // s = t + dot, with Q0 kept in D and t + dot in tin.
    float2 D[8], tin, dl;
    float2 Q1[AXIS ? 1 : 8], Q2[AXIS ? 1 : 8];
    {
        const int xa = px(lane), ya = py(lane), xb = px(lane + 32), yb = py(lane + 32);
        if (RECHECK) {
            pixa = ya * fd.W + xa;
            pixb = yb * fd.W + xb;
            xya = xa | (ya << 16);
            xyb = xb | (yb << 16);
        }
        const bool va = xa < fd.W && ya < fd.H, vb = xb < fd.W && yb < fd.H;
        float da[3] = {0.f, 0.f, 1.f}, db[3] = {0.f, 0.f, 1.f};
        float tia = 0.f, toa = 0.f, tib = 0.f, tob = 0.f;
        acta = va && camera_clip<float>(F, fd.W, fd.H, xa, ya, da, tia, toa);
        actb = vb && camera_clip<float>(F, fd.W, fd.H, xb, yb, db, tib, tob);
        if constexpr (SPLIT) {
            const unsigned r = (unsigned)(kb / fd.k_chunk);
            skipa = va && __ldcg(sc.part_hit + ya * fd.W + xa) < r;
            skipb = vb && __ldcg(sc.part_hit + yb * fd.W + xb) < r;
            acta = acta && !skipa;
            actb = actb && !skipb;
        }
        if (!acta) tia = toa = 0.f;
        if (!actb) tib = tob = 0.f;
        dl = make_float2((toa - tia) / (float)N, (tob - tib) / (float)N);
        if (RECHECK) {  // a half without a ray samples far away: never within the recheck band
            if (!acta) tia = kFarT;
            if (!actb) tib = kFarT;
        }
        float Da[8], Db[8];
        slice_dir<float>(F, da, Da);
        slice_dir<float>(F, db, Db);
#pragma unroll
        for (int i = 0; i < 8; ++i) D[i] = make_float2(Da[i], Db[i]);
        tin = make_float2(tia, tib);
        if constexpr (!AXIS) {
            // each ray's coefficients by the scalar code of march_kernel and
            // bisect_chunk (same operations, so the same values), then paired
            float Qa[3][8], Qb[3][8], dota, dotb;
            first_iterate_coeffs<float, SQ>(F.A, Da, F.c, dota, Qa[0], Qa[1], Qa[2]);
            first_iterate_coeffs<float, SQ>(F.A, Db, F.c, dotb, Qb[0], Qb[1], Qb[2]);
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                D[i] = make_float2(Qa[0][i], Qb[0][i]);
                Q1[i] = make_float2(Qa[1][i], Qb[1][i]);
                Q2[i] = make_float2(Qa[2][i], Qb[2][i]);
            }
            tin = make_float2(vadd(tia, dota), vadd(tib, dotb));
        }
    }
    const bool boxa = acta, boxb = actb;
    int suma = 0, sumb = 0, maxa = 0, maxb = 0, kfa = -1, kfb = -1;
    int qn = RECHECK ? *left : 0, counted = qn;  // staged recheck entries (warp-uniform); left: of earlier tiles
    const int k0 = SPLIT ? kb : 0, k1 = SPLIT ? ke : N + 1;
    float2 kf = make_float2((float)k0, (float)k0);
    // `more`: some ray of the warp still marches.  It changes only in a round
    // that found a ray inside, so it is voted on only then.
    bool more = __any_sync(kFull, acta || actb);
    for (int k = k0; k < k1 && more; ++k) {
        const float2 t = f2fma(kf, dl, tin);
        kf = f2add(kf, make_float2(1.f, 1.f));
        float2 z[8];
        bool ina = acta, inb = actb, live;
        int ca, cb;
        float2 dm;
        if constexpr (AXIS) {
#pragma unroll
            for (int i = 0; i < 3; ++i) z[i] = f2fma(t, D[i], P.A[i]);  // the rest are 0
            classify_lockstep2<SQ, MOD, RECHECK, true>(z, P, F.R2, max_iter, ina, inb, ca, cb, dm, live);
        } else {
            first_iterate<float2, 8>(t, D, Q1, Q2, z);
            classify_lockstep2_it1<SQ, MOD, RECHECK>(z, P, F.R2, max_iter, ina, inb, ca, cb, dm, live);
        }
        if (RECHECK && __any_sync(kFull, fminf(dm.x, dm.y) <= P.margin_t)) {
            // a marginal sample in this round (rare): stage it
            const bool pa = acta && dm.x <= P.margin_t, pb = actb && dm.y <= P.margin_t;
            const unsigned ba = __ballot_sync(kFull, pa), bb = __ballot_sync(kFull, pb);
            const unsigned below = (1u << lane) - 1u;
            const int nqa = __popc(ba), nq = nqa + __popc(bb);
            if (pa) qs[qn + __popc(ba & below)] = make_int4(pixa, k | (kMarchSample << 16), xya, ina ? 0 : ca + 1);
            if (pb) qs[qn + nqa + __popc(bb & below)] = make_int4(pixb, k | (kMarchSample << 16), xyb, inb ? 0 : cb + 1);
            qn += nq;
            if (qn > kQStage - 64) {
                flush_staged(fd, sc, qs, qn, counted);
                qn = counted = 0;
            }
        }
        // ina / inb imply acta / actb (they start equal and only clear)
        suma += ca;
        sumb += cb;
        maxa = max(maxa, ca);
        maxb = max(maxb, cb);
        if (live) {  // some half stayed bounded: those rays are inside at sample k
            if (ina) kfa = k;
            if (inb) kfb = k;
            if (RECHECK) {  // a finished ray samples far away from now on (see above)
                if (ina) tin.x = kFarT;
                if (inb) tin.y = kFarT;
            }
            acta = acta && !ina;
            actb = actb && !inb;
            more = __any_sync(kFull, acta || actb);
        }
    }
    if (RECHECK) *left = qn > counted ? recheck_staged<SQ, MOD, AXIS>(fd, sc, qs, qn, counted) : qn;
    const bool hita = kfa >= 0, hitb = kfb >= 0;
    // iterations = sum of (escape count) over escaped samples + max_iter per inside sample
    //            = sum of bounded steps + number of escaped samples
    const int nesca = (hita ? kfa : k1) - k0, nescb = (hitb ? kfb : k1) - k0;
    if constexpr (SPLIT) {  // this range's partial result per ray (see march_merge_kernel)
        const int xa = px(lane), ya = py(lane), xb = px(lane + 32), yb = py(lane + 32);
        const unsigned r = (unsigned)(kb / fd.k_chunk);
        const int64_t npx = (int64_t)fd.W * fd.H, base = (int64_t)r * npx;
        if (xa < fd.W && ya < fd.H && !skipa) {
            const int pa = ya * fd.W + xa;
            sc.part[base + pa] = boxa ? make_int4(kfa, suma + nesca, maxa + 1, nesca + (hita ? 1 : 0))
                                      : make_int4(-1, 0, 0, 0);
            if (hita) atomicMin(sc.part_hit + pa, r);
        }
        if (xb < fd.W && yb < fd.H && !skipb) {
            const int pb = yb * fd.W + xb;
            sc.part[base + pb] = boxb ? make_int4(kfb, sumb + nescb, maxb + 1, nescb + (hitb ? 1 : 0))
                                      : make_int4(-1, 0, 0, 0);
            if (hitb) atomicMin(sc.part_hit + pb, r);
        }
        return;
    }
    st.iters += (boxa ? suma + nesca : 0) + (boxb ? sumb + nescb : 0);
    st.samples += (boxa ? nesca + (hita ? 1 : 0) : 0) + (boxb ? nescb + (hitb ? 1 : 0) : 0);
    st.hits += (hita ? 1 : 0) + (hitb ? 1 : 0);
    const int xa = px(lane), ya = py(lane), xb = px(lane + 32), yb = py(lane + 32);
    const bool va = xa < fd.W && ya < fd.H, vb = xb < fd.W && yb < fd.H;
    if (va && !hita) write_miss<float>(fd, xa, ya, boxa ? maxa + 1 : 0);
    if (vb && !hitb) write_miss<float>(fd, xb, yb, boxb ? maxb + 1 : 0);
    warp_push(hita, make_int4(ya * fd.W + xa, kfa, 0, 0), sc.hits, sc.hit_cap, &sc.ctr->hit_count);
    warp_push(hitb, make_int4(yb * fd.W + xb, kfb, 0, 0), sc.hits, sc.hit_cap, &sc.ctr->hit_count);
}

// march2_tile with two samples of each ray per round (samples k and k + 1,
// classify_lockstep4_axis / classify_lockstep4_it1): the same per-sample
// arithmetic, so the same results, iteration counts and recheck entries.  A
// sample k + 1 after an inside sample k is classified but not counted or
// staged, as the one-sample march never reaches it.  SPLIT: samples [kb, ke)
// of each ray with the range's partial result, as in march2_tile.
// The tile's samples are taken 512 at a time: blocks of them whose escape
// count a bound proves (settle_chunk) only add to the counts, the rounds of
// the others are marched in order.  Without SETTLE all of them are (a split
// march's ranges and frames of few, wide samples do not pay for the bound, and
// the loop without it is the shorter one).  box: the warp's, in shared memory.
template <int SQ, int MOD, bool RECHECK, bool AXIS, bool SPLIT, bool SETTLE>
__device__ __forceinline__ void march4_tile(const FrameDesc &fd, const PairConsts &P, const Scratch &sc, unsigned tile,
                                            LaneStats &st, TileBox &box, int4 *qs = nullptr, int *left = nullptr,
                                            int kb = 0, int ke = 0)
{
    const FrameT<float> &F = fd.f;
    const int lane = threadIdx.x & 31;
    const int N = fd.N, max_iter = fd.max_iter;
    // pixels of the tile slots `lane` and `lane + 32`, x | y << 16 (no division
    // at the end of the tile, where they are needed again)
    int xya, xyb;
    {
        const int ty = (int)(tile / (unsigned)fd.tiles_x), tx = (int)tile - ty * fd.tiles_x;
        const int sya = lane / fd.tile_w, syb = (lane + 32) / fd.tile_w;
        xya = (tx * fd.tile_w + lane - sya * fd.tile_w) | ((ty * fd.tile_h + sya) << 16);
        xyb = (tx * fd.tile_w + lane + 32 - syb * fd.tile_w) | ((ty * fd.tile_h + syb) << 16);
    }
    const int xa = xya & 0xffff, ya = xya >> 16, xb = xyb & 0xffff, yb = xyb >> 16;
    int pixa = 0, pixb = 0;
    bool acta, actb, skipa = false, skipb = false;
    // as in march2_tile: zeta_0 = A + t D on an axis slice, else the first
    // iterate Q0 + s (Q1 + s Q2) with Q0 in D and s = t + dot
    float2 D[AXIS ? 3 : 8], tin, dl;
    float2 Q1[AXIS ? 1 : 8], Q2[AXIS ? 1 : 8];
    {
        if (RECHECK) {
            pixa = ya * fd.W + xa;
            pixb = yb * fd.W + xb;
        }
        const bool va = xa < fd.W && ya < fd.H, vb = xb < fd.W && yb < fd.H;
        float da[3] = {0.f, 0.f, 1.f}, db[3] = {0.f, 0.f, 1.f};
        float tia = 0.f, toa = 0.f, tib = 0.f, tob = 0.f;
        acta = va && camera_clip<float>(F, fd.W, fd.H, xa, ya, da, tia, toa);
        actb = vb && camera_clip<float>(F, fd.W, fd.H, xb, yb, db, tib, tob);
        if constexpr (SPLIT) {
            const unsigned r = (unsigned)(kb / fd.k_chunk);
            skipa = va && __ldcg(sc.part_hit + ya * fd.W + xa) < r;
            skipb = vb && __ldcg(sc.part_hit + yb * fd.W + xb) < r;
            acta = acta && !skipa;
            actb = actb && !skipb;
        }
        if (!acta) tia = toa = 0.f;
        if (!actb) tib = tob = 0.f;
        if (SETTLE && fd.settle) tile_box(fd, acta, da, tia, toa, actb, db, tib, tob, box);
        dl = make_float2((toa - tia) / (float)N, (tob - tib) / (float)N);
        if (RECHECK) {  // a half without a ray samples far away: never within the recheck band
            if (!acta) tia = kFarT;
            if (!actb) tib = kFarT;
        }
        float Da[8], Db[8];
        slice_dir<float>(F, da, Da);
        slice_dir<float>(F, db, Db);
        if constexpr (AXIS) {
#pragma unroll
            for (int i = 0; i < 3; ++i) D[i] = make_float2(Da[i], Db[i]);
            tin = make_float2(tia, tib);
        } else {
            float Qa[3][8], Qb[3][8], dota, dotb;
            first_iterate_coeffs<float, SQ>(F.A, Da, F.c, dota, Qa[0], Qa[1], Qa[2]);
            first_iterate_coeffs<float, SQ>(F.A, Db, F.c, dotb, Qb[0], Qb[1], Qb[2]);
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                D[i] = make_float2(Qa[0][i], Qb[0][i]);
                Q1[i] = make_float2(Qa[1][i], Qb[1][i]);
                Q2[i] = make_float2(Qa[2][i], Qb[2][i]);
            }
            tin = make_float2(vadd(tia, dota), vadd(tib, dotb));
        }
    }
    const bool boxa = acta, boxb = actb;
    int suma = 0, sumb = 0, maxa = 0, maxb = 0, kfa = -1, kfb = -1;
    int qn = RECHECK ? *left : 0, counted = qn;  // staged recheck entries (warp-uniform); left: of earlier tiles
    if (RECHECK) {
        __syncwarp();
        if (lane == 0) box.staged = qn;
        __syncwarp();
    }
    const int k0 = SPLIT ? kb : 0, k1 = SPLIT ? ke : N + 1;
    const float2 far = make_float2(kFarT, kFarT);
    bool more = __any_sync(kFull, acta || actb);
    // settled samples: the chunk [kc, kce) in hand, its
    // words of settled counts, the blocks and pairs of it still to march
    const bool settle = SETTLE && fd.settle && k1 > kSettleMin;
    int kc = k0 - kSettleChunk, kce = kc, pairs = 1, b = 0, p = 0;
    unsigned w = 0, open = 0, blocks = 0, ob = 0;
    float kf = (float)k0;  // k, carried along: a conversion would head every round's chain
    for (int k = k0; more; k += 2, kf += 2.f) {
        if (settle) {
            while (!ob) {
                if (!blocks) {  // the chunk is through: its settled samples, then the next chunk
                    if (kce > k0) {
                        int s, m;
                        settled_before(w, kc, kce, pairs, 32, 0, s, m);
                        suma += acta ? s : 0;
                        sumb += actb ? s : 0;
                        maxa = max(maxa, acta ? m : 0);
                        maxb = max(maxb, actb ? m : 0);
                    }
                    kc += kSettleChunk;
                    if (kc >= k1) break;
                    kce = min(kc + kSettleChunk, k1);
                    pairs = settle_pairs(kce - kc);
                    w = kce - kc > kSettleMin ? settle_chunk<SQ, MOD, AXIS>(fd, box, kc, kce, pairs) : 0u;
                    open = open_pairs(w, kc, kce, pairs);
                    blocks = __ballot_sync(kFull, open != 0);
                    continue;
                }
                b = __ffs(blocks) - 1;
                blocks &= blocks - 1;
                ob = __shfl_sync(kFull, open, b);
            }
            if (!ob) break;  // no chunk is left
            p = (__ffs(ob) - 1) >> 2;
            ob &= ob - 1;
            k = kc + 2 * (pairs * b + p);
            kf = (float)k;
        }
        if (k >= k1) break;
        const bool has2 = k + 1 < k1;  // warp-uniform: an odd number of samples ends in a round of one
        const float kf2 = kf + 1.f;
        const float2 t = f2fma(make_float2(kf, kf), dl, tin);
        const float2 t2 = has2 ? f2fma(make_float2(kf2, kf2), dl, tin) : far;
        float2 z[8], y[8];
        bool ina = acta, inb = actb, ina2 = acta && has2, inb2 = actb && has2, live;
        int ca, cb, ca2, cb2;
        float2 dm, dm2;
        if constexpr (AXIS) {
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                z[i] = f2fma(t, D[i], P.A[i]);
                y[i] = f2fma(t2, D[i], P.A[i]);
            }
            classify_lockstep4_axis<SQ, MOD, RECHECK>(z, y, P, F.R2, max_iter, ina, inb, ina2, inb2, ca, cb, ca2,
                                                      cb2, dm, dm2, live);
        } else {
            first_iterate<float2, 8>(t, D, Q1, Q2, z);
            first_iterate<float2, 8>(t2, D, Q1, Q2, y);
            classify_lockstep4_it1<SQ, MOD, RECHECK>(z, y, P, F.R2, max_iter, ina, inb, ina2, inb2, ca, cb, ca2,
                                                     cb2, dm, dm2, live);
        }
        if (RECHECK && __any_sync(kFull, fminf(fminf(dm.x, dm.y), fminf(dm2.x, dm2.y)) <= P.margin_t)) {
            // marginal samples in this round: staged by the lanes that hold them (a
            // few), through the warp's shared counter
            const bool pa = acta && dm.x <= P.margin_t, pb = actb && dm.y <= P.margin_t;
            const bool pa2 = acta && has2 && !ina && dm2.x <= P.margin_t;
            const bool pb2 = actb && has2 && !inb && dm2.y <= P.margin_t;
            const int np = (pa ? 1 : 0) + (pb ? 1 : 0) + (pa2 ? 1 : 0) + (pb2 ? 1 : 0);
            if (np) {
                int at = atomicAdd(&box.staged, np);
                const int kk = k | (kMarchSample << 16);
                if (pa) qs[at++] = make_int4(pixa, kk, xya, ina ? 0 : ca + 1);
                if (pb) qs[at++] = make_int4(pixb, kk, xyb, inb ? 0 : cb + 1);
                if (pa2) qs[at++] = make_int4(pixa, kk + 1, xya, ina2 ? 0 : ca2 + 1);
                if (pb2) qs[at++] = make_int4(pixb, kk + 1, xyb, inb2 ? 0 : cb2 + 1);
            }
            __syncwarp();
            qn = *(volatile int *)&box.staged;
            if (qn > kQStage - 128) {
                flush_staged(fd, sc, qs, qn, counted);
                if (lane == 0) box.staged = 0;
                __syncwarp();
                qn = counted = 0;
            }
        }
        // sample k + 1 counts only after an outside sample k (ca2 = 0 without a sample)
        suma += ca + (ina ? 0 : ca2);
        sumb += cb + (inb ? 0 : cb2);
        maxa = max(maxa, max(ca, ina ? 0 : ca2));
        maxb = max(maxb, max(cb, inb ? 0 : cb2));
        if (live) {  // some half stayed bounded: those rays are inside at sample k or k + 1
            const bool da = ina || ina2, db = inb || inb2;
            if (da) kfa = ina ? k : k + 1;
            if (db) kfb = inb ? k : k + 1;
            if (RECHECK) {  // a finished ray samples far away from now on (see above)
                if (da) tin.x = kFarT;
                if (db) tin.y = kFarT;
            }
            if (settle) {  // rays that end here: their settled samples of this chunk so far
                int s, m;
                settled_before(w, kc, kce, pairs, b, p, s, m);
                if (da) {
                    suma += s;
                    maxa = max(maxa, m);
                }
                if (db) {
                    sumb += s;
                    maxb = max(maxb, m);
                }
            }
            acta = acta && !da;
            actb = actb && !db;
            more = __any_sync(kFull, acta || actb);
        }
    }
    if (RECHECK) *left = qn > counted ? recheck_staged<SQ, MOD, AXIS>(fd, sc, qs, qn, counted) : qn;
    const bool hita = kfa >= 0, hitb = kfb >= 0;
    const int nesca = (hita ? kfa : k1) - k0, nescb = (hitb ? kfb : k1) - k0;
    if constexpr (SPLIT) {  // this range's partial result per ray (see march_merge_kernel)
        const unsigned r = (unsigned)(kb / fd.k_chunk);
        const int64_t npx = (int64_t)fd.W * fd.H, base = (int64_t)r * npx;
        if (xa < fd.W && ya < fd.H && !skipa) {
            const int pa = ya * fd.W + xa;
            sc.part[base + pa] = boxa ? make_int4(kfa, suma + nesca, maxa + 1, nesca + (hita ? 1 : 0))
                                      : make_int4(-1, 0, 0, 0);
            if (hita) atomicMin(sc.part_hit + pa, r);
        }
        if (xb < fd.W && yb < fd.H && !skipb) {
            const int pb = yb * fd.W + xb;
            sc.part[base + pb] = boxb ? make_int4(kfb, sumb + nescb, maxb + 1, nescb + (hitb ? 1 : 0))
                                      : make_int4(-1, 0, 0, 0);
            if (hitb) atomicMin(sc.part_hit + pb, r);
        }
        return;
    }
    st.iters += (boxa ? suma + nesca : 0) + (boxb ? sumb + nescb : 0);
    st.samples += (boxa ? nesca + (hita ? 1 : 0) : 0) + (boxb ? nescb + (hitb ? 1 : 0) : 0);
    st.hits += (hita ? 1 : 0) + (hitb ? 1 : 0);
    const bool va = xa < fd.W && ya < fd.H, vb = xb < fd.W && yb < fd.H;
    if (va && !hita) write_miss<float>(fd, xa, ya, boxa ? maxa + 1 : 0);
    if (vb && !hitb) write_miss<float>(fd, xb, yb, boxb ? maxb + 1 : 0);
    warp_push(hita, make_int4(ya * fd.W + xa, kfa, 0, 0), sc.hits, sc.hit_cap, &sc.ctr->hit_count);
    warp_push(hitb, make_int4(yb * fd.W + xb, kfb, 0, 0), sc.hits, sc.hit_cap, &sc.ctr->hit_count);
}

// Normal (central differences of F(p) = modulus(zeta_{n*}(p)) at p +- h e_a,
// iterated n* times from zeta0 = A + depth D +- h E_a, the slice image of
// eye + depth d +- h e_a), shading and the pixel's outputs for a hit at depth;
// lanes with part == false only join the warp-wide loop bound.
template <typename T, int SQ, int MOD>
__device__ __forceinline__ void normal_shade(const FrameDesc &fd, const FrameT<T> &F, int x, int y, const T (&d)[3],
                                             const T (&D)[8], T depth, int n_star, bool part, LaneStats &st)
{
    int nmax = part ? n_star : 0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) nmax = max(nmax, __shfl_xor_sync(kFull, nmax, o));
    T g[3];
    bool guard = false;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        T fv[2];
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            const T hs = s == 0 ? F.h : -F.h;
            T z[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) z[i] = dfma(hs, F.E[a][i], dfma(depth, D[i], F.A[i]));
            T sp = dq_sp<T>(z);
#pragma unroll 1
            for (int n = 0; n < nmax; ++n)
                if (n < n_star) dq_iter<T, SQ, MOD>(z, z, sp, F.c);
            fv[s] = modulus<T, MOD>(z);
            guard = guard || !(fv[s] <= normal_fmax(T(0)));
        }
        g[a] = fv[0] - fv[1];
    }
    if (part) {
        st.niters += 6ull * (unsigned)n_star;
        shade_write<T>(fd, F, x, y, n_star, depth, g, guard, d);
    }
}

// Bisection, normal and shading of hit-list entries [base, base + 32) clipped to
// nhits, one per lane (see bisect_kernel); all 32 lanes call.  Late hits of the
// recheck mode join the warp's list late[0, nlate) (push_late); the caller
// evaluates what is left in it.
template <typename T, int SQ, int MOD, bool RECHECK>
__device__ __forceinline__ void bisect_chunk(const FrameDesc &fd, const Scratch &sc, unsigned base, unsigned nhits,
                                             LaneStats &st, int4 *late, int &nlate)
{
    const FrameT<T> &F = frame<T>(fd);
    const int lane = threadIdx.x & 31;
    const unsigned idx = base + lane;
    const bool part = idx < nhits;
    int4 e = make_int4(0, 0, 0, 0);
    if (part) e = __ldcg(sc.hits + idx);  // L2: the list may be rewritten within one serving launch
    const int pixel = e.x, k_first = e.y;
    const int x = pixel % fd.W, y = pixel / fd.W;
    T d[3] = {T(0), T(0), T(1)};
    T t_in = T(0), t_out = T(0);
    if (part) camera_clip<T>(F, fd.W, fd.H, x, y, d, t_in, t_out);
    T D[8];
    slice_dir<T>(F, d, D);
    const T delta = (t_out - t_in) / T(fd.N);
    bool bis = part && k_first > 0;
    T lo = bis ? dfma(T(k_first - 1), delta, t_in) : t_in;
    T hi = bis ? dfma(T(k_first), delta, t_in) : t_in;
    // n* starts as the escape count of the last outside march sample, k_first - 1:
    // the march keeps no per-sample counts, so it is classified again here, with
    // the march's own position and arithmetic (not counted as new iterations)
    int n_lo = fd.max_iter;
    {
        T z[8];
        bool mg;
        int n;
        bool it1 = false;
        if constexpr (sizeof(T) == 4) {
            if (!fd.axis_slice) {  // the FP32 march's first-iterate form and sample position
                it1 = true;
                float Q0[8], Q1[8], Q2[8], dot;
                first_iterate_coeffs<float, SQ>(F.A, D, F.c, dot, Q0, Q1, Q2);
                first_iterate<float, 8>(vfma((float)(k_first - 1), delta, vadd(t_in, dot)), Q0, Q1, Q2, z);
            }
        }
        if (it1) {
            n = classify_lockstep_it1<T, SQ, MOD, false>(z, F, fd.max_iter, bis, mg);
        } else {
#pragma unroll
            for (int i = 0; i < 8; ++i) z[i] = dfma(lo, D[i], F.A[i]);
            n = classify_sample<T, SQ, MOD, false>(fd, z, bis, mg);
        }
        if (bis) n_lo = n;
    }
    unsigned path = 0;
    unsigned iters = 0, samples = 0;
    for (int b = 0; b < fd.B; ++b) {
        const T mid = lo + T(0.5) * (hi - lo);
        T z[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) z[i] = dfma(mid, D[i], F.A[i]);
        bool mg;
        const int n = classify_sample<T, SQ, MOD, RECHECK>(fd, z, bis, mg);
        if (RECHECK) {
            const bool push = bis && mg;
            if (warp_push(push, make_int4(pixel, k_first | (b << 16), (int)path, n), sc.queue, sc.queue_cap,
                          &sc.ctr->queue_count)) {
                atomicAdd(&sc.ctr->stats[7], 1ull);
                mark_dirty(fd, sc, pixel);
            }
            st.rechecks += push ? 1 : 0;
        }
        if (bis) {
            iters += n ? (unsigned)n : (unsigned)fd.max_iter;
            samples += 1;
            if (n == 0) {
                hi = mid;
            } else {
                lo = mid;
                n_lo = n;
                path |= 1u << b;
            }
        }
    }
    const T depth = bis ? lo + T(0.5) * (hi - lo) : t_in;
    // RECHECK: the FP32 field of a normal of more than late_step steps carries
    // its rounding amplified along the orbit, so those normals are evaluated in
    // FP64 (on the FP64 ray, at the bisection's depth); the others in FP32
    const bool n64 = RECHECK && sizeof(T) == 4 && part && n_lo > late_step<MOD>();
    normal_shade<T, SQ, MOD>(fd, F, x, y, d, D, depth, n_lo, part && !n64, st);
    if constexpr (RECHECK && sizeof(T) == 4)
        push_late<SQ, MOD>(fd, n64, late_hit(x, y, n_lo, (double)depth), late, nlate, st.niters);
    st.iters += iters;
    st.samples += samples;
}

// Normal and shading of the hits of an L-lane group (see bisect_group):
// evaluation q = 2a + s (F at depth -+ h e_a, s = 0: +h) runs on lane q mod L of
// the group, in round q / L; `part` is uniform within a group.  All 32 lanes
// call.  Same values as normal_shade<U>.
template <typename U, int SQ, int MOD, int L>
__device__ __forceinline__ void group_normal(const FrameDesc &fd, const FrameT<U> &F, int x, int y, const U (&d)[3],
                                             const U (&D)[8], U depth, int n_lo, bool part, LaneStats &st)
{
    const int lane = threadIdx.x & 31;
    const int j = lane & (L - 1), gb = lane & ~(L - 1);
    int nmax = part ? n_lo : 0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) nmax = max(nmax, __shfl_xor_sync(kFull, nmax, o));
    U fvq[6];
    bool guard = false;
#pragma unroll
    for (int q0 = 0; q0 < 6; q0 += L) {
        const int q = q0 + j;
        const int a = q < 6 ? q >> 1 : 0;
        const U hs = (q & 1) == 0 ? F.h : -F.h;
        U z[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) z[i] = dfma(hs, F.E[a][i], dfma(depth, D[i], F.A[i]));
        U sp = dq_sp<U>(z);
        const int ns = part && q < 6 ? n_lo : 0;
#pragma unroll 1
        for (int n = 0; n < nmax; ++n)
            if (n < ns) dq_iter<U, SQ, MOD>(z, z, sp, F.c);
        const U fv = modulus<U, MOD>(z);
        const unsigned bad = __ballot_sync(kFull, q < 6 && !(fv <= normal_fmax(U(0))));
        guard = guard || ((bad >> gb) & ((1u << L) - 1u)) != 0;
#pragma unroll
        for (int i = 0; i < L; ++i)
            if (q0 + i < 6) fvq[q0 + i] = __shfl_sync(kFull, fv, gb + i);
    }
    if (part && j == 0) {
        U g[3] = {fvq[0] - fvq[1], fvq[2] - fvq[3], fvq[4] - fvq[5]};
        st.niters += 6ull * (unsigned)n_lo;
        shade_write<U>(fd, F, x, y, n_lo, depth, g, guard, d);
    }
}

// The same bisection, normal and shading for hit-list entries [base, base +
// 32 / L) clipped to nhits, L lanes per hit (L = 4 or 8; lane group g = lane / L
// takes entry base + g; all 32 lanes call).  For frames with few hits per SM,
// where one lane per hit leaves the bisection's dependent chain of B + 7
// classifications exposed: here the lanes of a group classify the midpoints of
// log2(L) levels of the bisection tree at once (lane j < L - 1 holds node j + 1:
// node 1 the next midpoint, children 2i inside -> [lo, mid] and 2i + 1 outside
// -> [mid, hi]), each deriving its interval with the sequential halvings' own
// operations, and the group replays the path; the six normal evaluations are
// spread over the group's lanes.  Brackets, n*, depths, normals, queued
// rechecks and the counted iterations (only the nodes on the path count) are
// those of bisect_chunk.
template <typename T, int SQ, int MOD, bool RECHECK, int L>
__device__ __forceinline__ void bisect_group(const FrameDesc &fd, const Scratch &sc, unsigned base, unsigned nhits,
                                             LaneStats &st, int4 *late, int &nlate)
{
    static_assert(L == 4 || L == 8, "four or eight lanes per hit");
    constexpr int kLevels = L == 8 ? 3 : 2;  // tree levels per round
    const FrameT<T> &F = frame<T>(fd);
    const int lane = threadIdx.x & 31;
    const int j = lane & (L - 1), gb = lane & ~(L - 1);  // lane in the group, the group's first lane
    const unsigned idx = base + (unsigned)(lane / L);
    const bool part = idx < nhits;
    int4 e = make_int4(0, 0, 0, 0);
    if (part) e = __ldcg(sc.hits + idx);  // L2: the list may be rewritten within one serving launch
    const int pixel = e.x, k_first = e.y;
    const int x = pixel % fd.W, y = pixel / fd.W;
    T d[3] = {T(0), T(0), T(1)};
    T t_in = T(0), t_out = T(0);
    if (part) camera_clip<T>(F, fd.W, fd.H, x, y, d, t_in, t_out);
    T D[8];
    slice_dir<T>(F, d, D);
    const T delta = (t_out - t_in) / T(fd.N);
    const bool bis = part && k_first > 0;
    T lo = bis ? dfma(T(k_first - 1), delta, t_in) : t_in;
    T hi = bis ? dfma(T(k_first), delta, t_in) : t_in;
    // n* starts as the escape count of march sample k_first - 1, classified
    // again with the march's position and arithmetic (not counted): on the
    // group's last lane, in the first round where that form is the midpoints'
    // form, else (the FP32 march's first-iterate form of a general slice) before
    int n_lo = fd.max_iter;
    bool lo_in_round0 = true;
    if constexpr (sizeof(T) == 4) {
        if (!fd.axis_slice) {
            lo_in_round0 = false;
            T z[8];
            float Q0[8], Q1[8], Q2[8], dot;
            first_iterate_coeffs<float, SQ>(F.A, D, F.c, dot, Q0, Q1, Q2);
            first_iterate<float, 8>(vfma((float)(k_first - 1), delta, vadd(t_in, dot)), Q0, Q1, Q2, z);
            bool mg;
            const int n = classify_lockstep_it1<T, SQ, MOD, false>(z, F, fd.max_iter, bis && j == L - 1, mg);
            const int nl = __shfl_sync(kFull, n, gb + L - 1);
            if (bis) n_lo = nl;
        }
    }
    unsigned path = 0;
    unsigned iters = 0, samples = 0, rechecks = 0;
    const int node = j + 1, level = 31 - __clz(node);  // last lane: node L, level kLevels (no node)
    for (int b0 = 0; b0 < fd.B || (b0 == 0 && lo_in_round0); b0 += kLevels) {
        const int levels = min(kLevels, fd.B - b0);
        const bool lo_lane = b0 == 0 && lo_in_round0 && j == L - 1;
        T l = lo, h = hi;
        for (int q = level - 1; q >= 0; --q) {  // path bits below the node's leading one
            const T mid = l + T(0.5) * (h - l);
            if ((node >> q) & 1)
                l = mid;
            else
                h = mid;
        }
        const T pos = lo_lane ? lo : l + T(0.5) * (h - l);
        const bool act = bis && (lo_lane || level < levels);
        T z[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) z[i] = dfma(pos, D[i], F.A[i]);
        bool mg;
        const int n = classify_sample<T, SQ, MOD, RECHECK>(fd, z, act, mg);
        if (b0 == 0 && lo_in_round0) {
            const int nl = __shfl_sync(kFull, n, gb + L - 1);
            if (bis) n_lo = nl;
        }
        // replay the path through the levels of this round
        int cur = 1;
        for (int lv = 0; lv < kLevels; ++lv) {
            const int nc = __shfl_sync(kFull, n, gb + cur - 1);
            const bool mc = RECHECK ? __shfl_sync(kFull, mg, gb + cur - 1) : false;
            if (lv >= levels) break;  // warp-uniform
            const int b = b0 + lv;
            if (RECHECK) {
                const bool push = bis && mc && j == 0;
                if (warp_push(push, make_int4(pixel, k_first | (b << 16), (int)path, nc), sc.queue, sc.queue_cap,
                              &sc.ctr->queue_count)) {
                    atomicAdd(&sc.ctr->stats[7], 1ull);
                    mark_dirty(fd, sc, pixel);
                }
                rechecks += push ? 1 : 0;
            }
            const T mid = lo + T(0.5) * (hi - lo);
            if (bis) {
                iters += nc ? (unsigned)nc : (unsigned)fd.max_iter;
                samples += 1;
                if (nc == 0) {
                    hi = mid;
                } else {
                    lo = mid;
                    n_lo = nc;
                    path |= 1u << b;
                }
            }
            cur = 2 * cur + (nc != 0 ? 1 : 0);
        }
    }
    const T depth = bis ? lo + T(0.5) * (hi - lo) : t_in;
    // RECHECK: a normal of more than late_step steps is evaluated in FP64 (see
    // bisect_chunk), the others in T
    const bool n64 = RECHECK && sizeof(T) == 4 && part && n_lo > late_step<MOD>();
    group_normal<T, SQ, MOD, L>(fd, F, x, y, d, D, depth, n_lo, part && !n64, st);
    if constexpr (RECHECK && sizeof(T) == 4)
        push_late<SQ, MOD>(fd, n64 && j == 0, late_hit(x, y, n_lo, (double)depth), late, nlate, st.niters);
    if (part && j == 0) {
        st.iters += iters;
        st.samples += samples;
        if (RECHECK) st.rechecks += rechecks;
    }
}

// Add a warp's lane counters to the frame's stats.
template <bool RECHECK>
__device__ __forceinline__ void flush_lane_stats(const Scratch &sc, const LaneStats &st, bool march)
{
    flush_count(&sc.ctr->stats[0], st.iters);
    if (march) flush_count(&sc.ctr->stats[8], st.iters);
    if (!march) flush_count(&sc.ctr->stats[1], st.niters);  // a march evaluates no normals
    flush_count(&sc.ctr->stats[2], st.samples);
    flush_count(&sc.ctr->stats[3], st.hits);
    if (RECHECK) flush_count(&sc.ctr->stats[4], st.rechecks);
}

}  // namespace dqj
