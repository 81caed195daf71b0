// voxel_render.cu -- image of a voxel occupancy grid from the scene camera
// (Fig. voxels: the paper sets its ray-traced image beside renders of 50^3 and
// 100^3 voxel grids).  The grid is drawn as the union of its occupied cells,
// each a closed axis-aligned cube of the march box; a pixel shows the first cube
// its camera ray crosses, found by walking the ray cell by cell (Amanatides and
// Woo's grid traversal, 1987): start in the cell of the box entry point, then
// step to the neighbour across whichever cell face the ray reaches first.  On
// grids of 24 cells a side or more, blocks of cells without an occupied one are
// crossed in one step (voxel_render_blocks_kernel), with the same image.
//
// One pixel per thread, 16 x 8 pixel tiles per CTA, so a warp's rays walk
// neighbouring cells and share the occupancy bytes through L1/L2.  The camera
// ray, the start cell and the hit depth are FP64; the per-step choice of the
// next face compares FP32 face distances against a rigorous error bound and
// falls back to FP64 within it, so every choice is the one an FP64 walk makes
// except where two faces lie within FP64 rounding of each other (FP64 runs at
// 1/64 of the FP32 rate on this part).  A ray crosses at most 3 g - 2 cells.
#include "render_common.cuh"
#include "runtime.h"

namespace dqj {

namespace {

constexpr int kVrTileW = 16, kVrTileH = 8;
static_assert(kVrTileW * kVrTileH == kBlock, "one pixel per thread");

// Grid-uniform FP64 constants, computed once on the host.
struct GridGeom {
    double size[3];      // cell edge per axis, (box_max - box_min) / g
    double inv_size[3];  // g / (box_max - box_min)
    double lo_e[3];      // box_min - eye
    double hi_e[3];      // box_max - eye
    double sxa, sxb;     // screen x = (x + 0.5) sxa + sxb  (pinhole camera)
    double sya, syb;     // screen y = (y + 0.5) sya + syb
};

// Hit pixel: the entered face's outward normal (-d when the eye is inside the
// hit cube) and the ambient, diffuse and specular terms of Eq. phong, shaded in
// FP32 (the FP32 frame constants; the normal is exact and the depth FP64).
__device__ __forceinline__ void write_face_hit(const FrameDesc &fd, int x, int y, int iter, double depth, int axis,
                                               const double (&d)[3])
{
    const FrameT<float> &F = fd.f;
    float n[3], df[3];
#pragma unroll
    for (int b = 0; b < 3; ++b) {
        df[b] = (float)d[b];
        n[b] = axis < 0 ? -df[b] : (axis == b ? (d[b] > 0.0 ? -1.f : 1.f) : 0.f);
    }
    float ndl = n[0] * F.light[0] + n[1] * F.light[1] + n[2] * F.light[2];
    float spec = 0.f;
    if (F.ks > 0.f && ndl > 0.f) {  // reflected light r = 2n(n.l) - l against v = -d
        const float rv = -((2.f * ndl * n[0] - F.light[0]) * df[0] + (2.f * ndl * n[1] - F.light[1]) * df[1] +
                           (2.f * ndl * n[2] - F.light[2]) * df[2]);
        if (rv > 0.f) spec = F.ks * powf(rv, F.shin);
    }
    ndl = ndl > 0.f ? ndl : 0.f;
    float v = F.ka + F.kd * ndl + spec;
    v = v < 0.f ? 0.f : (v > 1.f ? 1.f : v);
    const int64_t o = (int64_t)y * fd.pitch + x;
    if (fd.iter) fd.iter[o] = iter;
    if (fd.depth) fd.depth[o] = (float)depth;
    if (fd.normal) {
        fd.normal[3 * o + 0] = n[0];
        fd.normal[3 * o + 1] = n[1];
        fd.normal[3 * o + 2] = n[2];
    }
    if (fd.rgba)
        *reinterpret_cast<uchar4 *>(fd.rgba + 4 * o) =
            make_uchar4(to_u8(v * F.albedo[0]), to_u8(v * F.albedo[1]), to_u8(v * F.albedo[2]), 255);
}

// A pixel's ray through the grid.  Per axis: the ray reaches cell plane k (bmin +
// k size) at t = base + k sd, base = (bmin - eye) / d, sd = size / d.
struct Walk {
    double d[3], b64[3], d64[3], t_in;
    float b32[3], d32[3];
    float E[3], tol;  // error bounds of an axis's FP32 plane distances, and their sum
    int st[3], s[3];  // start cell; step per axis (0: the ray crosses no plane of it)
    int axis;         // face of the box entry (-1: the eye is inside the box)
};

// FP64 camera ray (the pinhole formula of the march) with reciprocals instead of
// divisions, box entry and start cell; false when the ray misses the box.  FP64
// runs at 1/64 of the FP32 rate here, and this per-pixel setup, not the walk,
// bounds small grids: only the values that the walk and the depth need are FP64
// (about 75 instructions; with the comparisons and the start cell in FP64 too it
// took 105).  Which face is entered, whether the box is met and the start cell
// are decided in FP32 where its error bounds allow, else by the FP64 values.
__device__ __forceinline__ bool walk_setup(const FrameDesc &fd, const GridGeom &geo, int g, int x, int y, Walk &W)
{
    const FrameT<double> &F = fd.d;
    const double sx = fma((double)x + 0.5, geo.sxa, geo.sxb);
    const double sy = fma((double)y + 0.5, geo.sya, geo.syb);
#pragma unroll
    for (int a = 0; a < 3; ++a) W.d[a] = F.fwd[a] + sx * F.right[a] + sy * F.upv[a];
    const double il = rsqrt(W.d[0] * W.d[0] + W.d[1] * W.d[1] + W.d[2] * W.d[2]);
    double tb[3];
    float df[3], te[3], in = -tinf<float>(), mid = -tinf<float>(), out = tinf<float>();
    bool in_box = true, finite = true;
    W.tol = 0.f;
    W.axis = -1;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        W.d[a] *= il;
        df[a] = (float)W.d[a];
        W.s[a] = df[a] > 0.f ? 1 : (df[a] < 0.f ? -1 : 0);
        if (W.s[a] == 0) {  // parallel to the slab
            if (F.eye[a] < F.bmin[a] || F.eye[a] > F.bmax[a]) in_box = false;
            W.b64[a] = W.d64[a] = tb[a] = 0.0;
            W.b32[a] = W.d32[a] = W.E[a] = 0.f;
            te[a] = -tinf<float>();
            continue;
        }
        const double id = __drcp_rn(W.d[a]);
        W.b64[a] = geo.lo_e[a] * id;
        W.d64[a] = geo.size[a] * id;
        tb[a] = geo.hi_e[a] * id;
        W.b32[a] = (float)W.b64[a];
        W.d32[a] = (float)W.d64[a];
        const float far = fmaf((float)g, W.d32[a], W.b32[a]);
        te[a] = W.s[a] > 0 ? W.b32[a] : far;
        out = fminf(out, W.s[a] > 0 ? far : W.b32[a]);
        if (te[a] > in) {
            mid = in;
            in = te[a];
            W.axis = a;
        } else {
            mid = fmaxf(mid, te[a]);
        }
        // The walk compares the FP32 values m = fma(k, sd, base) of the plane
        // distances; each lies within E = 2^-21 (g |sd| + |base|) of its FP64 value
        // (three roundings of at most 2^-24 relative each, with a factor 2 to
        // spare), so when the two nearest planes differ by more than the sum of the
        // bounds the FP32 order is the FP64 order; otherwise the choice is FP64's.
        // An axis whose FP32 plane distances overflow (|d| below ~1e-38) crosses no
        // cell plane inside the box, like an axis the ray runs parallel to; whether
        // the ray meets the box at all is then left to the FP64 distances.
        const bool cross = isfinite(W.d32[a]) && isfinite(W.b32[a]);
        W.E[a] = cross ? 4.76837158203125e-7f * ((float)g * fabsf(W.d32[a]) + fabsf(W.b32[a])) : 0.f;
        W.tol += W.E[a];
        if (!cross) {
            W.s[a] = 0;
            finite = false;
        }
    }
    W.t_in = in > 0.f ? (W.axis == 0 ? (W.s[0] > 0 ? W.b64[0] : tb[0])
                                     : (W.axis == 1 ? (W.s[1] > 0 ? W.b64[1] : tb[1]) : (W.s[2] > 0 ? W.b64[2] : tb[2])))
                      : 0.0;
    bool crosses = in_box;
    if (!(finite && in - mid > W.tol && fabsf(in) > W.tol && out - fmaxf(in, 0.f) > W.tol)) {
        // too close for FP32: entry and exit by the FP64 distances
        double t0 = -tinf<double>(), t1 = tinf<double>();
        W.axis = -1;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            if (df[a] == 0.f) continue;
            const double ta = W.b64[a], e = ta < tb[a] ? ta : tb[a], f = ta < tb[a] ? tb[a] : ta;
            if (e > t0) {
                t0 = e;
                W.axis = a;
            }
            t1 = f < t1 ? f : t1;
        }
        if (t0 < 0.0) {
            t0 = 0.0;
            W.axis = -1;
        }
        W.t_in = t0;
        crosses = crosses && t0 < t1;
    } else if (in < 0.f) {
        W.axis = -1;
    }
    if (!crosses) return false;
    const float t32 = (float)W.t_in;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const float off = -(float)geo.lo_e[a], inv = (float)geo.inv_size[a];
        const float c = fmaf(t32, df[a], off) * inv, tc = 2e-6f * inv * (fabsf(t32 * df[a]) + fabsf(off)) + 1e-6f * fabsf(c);
        int i = (int)floorf(c);
        if (W.axis == a && W.s[a] != 0) {
            i = W.s[a] > 0 ? 0 : g - 1;  // at the face itself
        } else if (!(fabsf(c - rintf(c)) > tc)) {
            const double p = F.eye[a] + W.t_in * W.d[a];
            i = (int)fmin(fmax(floor((p - F.bmin[a]) * geo.inv_size[a]), -1.0), (double)g);
        }
        W.st[a] = min(max(i, 0), g - 1);
    }
    return true;
}

__global__ void __launch_bounds__(kBlock) voxel_render_kernel(const __grid_constant__ FrameDesc fd,
                                                              const uint8_t *__restrict__ occ, int g,
                                                              const __grid_constant__ GridGeom geo)
{
    const int x = blockIdx.x * kVrTileW + (int)(threadIdx.x % kVrTileW);
    const int y = blockIdx.y * kVrTileH + (int)(threadIdx.x / kVrTileW);
    if (x >= fd.W || y >= fd.H) return;
    Walk W;
    if (!walk_setup(fd, geo, g, x, y, W)) {
        write_miss<double>(fd, x, y, 0);
        return;
    }
    const double(&d)[3] = W.d, (&b64)[3] = W.b64, (&d64)[3] = W.d64;
    const float(&b32)[3] = W.b32, (&d32)[3] = W.d32;
    const double t_in = W.t_in;
    const float tol = W.tol;
    const int s0 = W.s[0], s1 = W.s[1], s2 = W.s[2];
    int i0 = W.st[0], i1 = W.st[1], i2 = W.st[2];
    int k0 = i0 + (s0 > 0 ? 1 : 0), k1 = i1 + (s1 > 0 ? 1 : 0), k2 = i2 + (s2 > 0 ? 1 : 0);
    const float m[3] = {s0 ? fmaf((float)k0, d32[0], b32[0]) : tinf<float>(),
                        s1 ? fmaf((float)k1, d32[1], b32[1]) : tinf<float>(),
                        s2 ? fmaf((float)k2, d32[2], b32[2]) : tinf<float>()};
    // Each step moves to the neighbour across the nearest face.  The step is
    // written without branches: neighbouring lanes choose different axes, and
    // a three-way branch would run all three paths for the warp.  A cell
    // records how it was entered (code = axis | plane << 2 for a step across
    // cell plane `plane` of `axis`; 3 for the start cell, entered at the box
    // entry through face axis0).  g <= 1024, so cell indices fit in 32 bits.
    // (Measured and not kept: walking a few cells ahead to batch their loads,
    // plane indices carried as floats, and the FP64 choice out of line; each
    // was slower.)
    const int axis0 = W.axis;
    float m0 = m[0], m1 = m[1], m2 = m[2];
    const uint32_t gu = (uint32_t)g;
    const int32_t st0 = s0, st1 = s1 * g, st2 = s2 * g * g;
    uint32_t lin = ((uint32_t)i2 * gu + (uint32_t)i1) * gu + (uint32_t)i0;
    uint32_t code = 3u;
    int n = 0;  // cells tested
    bool hit = false;
    const int max_cells = 3 * g;  // a ray crosses at most 3 g - 2 cells
    while (n < max_cells) {
        ++n;
        if (__ldg(occ + lin)) {
            hit = true;
            break;
        }
        // the nearest face, ties to the lower axis
        int a = (m0 <= m1 && m0 <= m2) ? 0 : (m1 <= m2 ? 1 : 2);
        const float lo = fminf(m0, fminf(m1, m2));
        const float mid = fmaxf(fminf(m0, m1), fminf(fmaxf(m0, m1), m2));
        if (mid - lo <= tol) {  // too close for FP32: decide in FP64
            const double t0 = m[0] != tinf<float>() ? fma((double)k0, d64[0], b64[0]) : tinf<double>();
            const double t1 = m[1] != tinf<float>() ? fma((double)k1, d64[1], b64[1]) : tinf<double>();
            const double t2 = m[2] != tinf<float>() ? fma((double)k2, d64[2], b64[2]) : tinf<double>();
            a = (t0 <= t1 && t0 <= t2) ? 0 : (t1 <= t2 ? 1 : 2);
        }
        const bool x0 = a == 0, x1 = a == 1, x2 = a == 2;
        i0 += x0 ? s0 : 0;
        i1 += x1 ? s1 : 0;
        i2 += x2 ? s2 : 0;
        const bool out = ((unsigned)i0 >= gu) | ((unsigned)i1 >= gu) | ((unsigned)i2 >= gu);
        const int kc = x0 ? k0 : (x1 ? k1 : k2);
        const int sa = x0 ? s0 : (x1 ? s1 : s2);
        code = (uint32_t)a | ((uint32_t)kc << 2);
        k0 += x0 ? s0 : 0;
        k1 += x1 ? s1 : 0;
        k2 += x2 ? s2 : 0;
        lin += (uint32_t)(x0 ? st0 : (x1 ? st1 : st2));
        const float mk = fmaf((float)(kc + sa), x0 ? d32[0] : (x1 ? d32[1] : d32[2]), x0 ? b32[0] : (x1 ? b32[1] : b32[2]));
        m0 = x0 ? mk : m0;
        m1 = x1 ? mk : m1;
        m2 = x2 ? mk : m2;
        if (out) break;  // the cell just tested was the last inside the grid
    }
    if (!hit) {
        write_miss<double>(fd, x, y, n);
        return;
    }
    const int sa = (int)(code & 3u);
    const double kc = (double)(code >> 2);
    double t = t_in;  // the start cell is entered at the box entry
    if (sa == 0) t = fma(kc, d64[0], b64[0]);
    if (sa == 1) t = fma(kc, d64[1], b64[1]);
    if (sa == 2) t = fma(kc, d64[2], b64[2]);
    write_face_hit(fd, x, y, n, t, sa == 3 ? axis0 : sa, d);
}

// The same walk on a grid with block occupancy mip (one byte per block of 2^SHIFT
// cells a side, non-zero where some cell of it is occupied; blocks gb a side):
// empty blocks are crossed whole, plane by block plane, and the walk goes cell by
// cell only from the first cell of a block that is not empty.  The pixel's values
// are the walk's own: plane crossings happen in the order of (distance, axis), so
// the cell in which the ray enters a block, and the number of cells it crossed
// until there, follow from the crossing alone.  1080p, default c, cell by cell /
// by blocks (ms): 24^3 0.30 / 0.30, 64^3 0.37 / 0.32, 100^3 0.50 / 0.33, 200^3 1.0 / 0.37,
// 512^3 3.1 / 0.64, 1024^3 8.0 / 1.3 (more, and grids on which blocks only cost, at
// mip_shift).
template <int SHIFT>
__global__ void __launch_bounds__(kBlock) voxel_render_blocks_kernel(const __grid_constant__ FrameDesc fd,
                                                                     const uint8_t *__restrict__ occ, int g,
                                                                     const __grid_constant__ GridGeom geo,
                                                                     const uint8_t *__restrict__ mip, int gb)
{
    const int x = blockIdx.x * kVrTileW + (int)(threadIdx.x % kVrTileW);
    const int y = blockIdx.y * kVrTileH + (int)(threadIdx.x / kVrTileW);
    if (x >= fd.W || y >= fd.H) return;
    Walk W;
    if (!walk_setup(fd, geo, g, x, y, W)) {
        write_miss<double>(fd, x, y, 0);
        return;
    }
    const double(&d)[3] = W.d, (&b64)[3] = W.b64, (&d64)[3] = W.d64;
    const float(&b32)[3] = W.b32, (&d32)[3] = W.d32, (&E)[3] = W.E;
    const double t_in = W.t_in;
    const float tol = W.tol;
    const int s0 = W.s[0], s1 = W.s[1], s2 = W.s[2];
    int i0 = W.st[0], i1 = W.st[1], i2 = W.st[2];
    constexpr int B = 1 << SHIFT;
    const float inf = tinf<float>();
    const int c0 = i0, c1 = i1, c2 = i2;  // start cell
    // next block plane per axis (in cell planes) and its distance; block
    int q0 = s0 > 0 ? min((i0 & -B) + B, g) : (i0 & -B), q1 = s1 > 0 ? min((i1 & -B) + B, g) : (i1 & -B),
        q2 = s2 > 0 ? min((i2 & -B) + B, g) : (i2 & -B);
    float n0 = s0 ? fmaf((float)q0, d32[0], b32[0]) : inf, n1 = s1 ? fmaf((float)q1, d32[1], b32[1]) : inf,
          n2 = s2 ? fmaf((float)q2, d32[2], b32[2]) : inf;
    uint32_t blk = ((uint32_t)(i2 >> SHIFT) * (uint32_t)gb + (uint32_t)(i1 >> SHIFT)) * (uint32_t)gb + (uint32_t)(i0 >> SHIFT);
    const int32_t bs1 = s1 * gb, bs2 = s2 * gb * gb;
    const int32_t st1 = s1 * g, st2 = s2 * g * g;
    // the nearest of three planes, ties to the lower axis
    auto nearest = [&](float m0, float m1, float m2, int k0, int k1, int k2) {
        int a = (m0 <= m1 && m0 <= m2) ? 0 : (m1 <= m2 ? 1 : 2);
        const float lo = fminf(m0, fminf(m1, m2));
        const float mid = fmaxf(fminf(m0, m1), fminf(fmaxf(m0, m1), m2));
        if (mid - lo <= tol) {  // too close for FP32: decide in FP64
            const double t0 = s0 ? fma((double)k0, d64[0], b64[0]) : tinf<double>();
            const double t1 = s1 ? fma((double)k1, d64[1], b64[1]) : tinf<double>();
            const double t2 = s2 ? fma((double)k2, d64[2], b64[2]) : tinf<double>();
            a = (t0 <= t1 && t0 <= t2) ? 0 : (t1 <= t2 ? 1 : 2);
        }
        return a;
    };
    // the walk crosses block plane kc of axis a in direction sa: next plane, next block
    auto next_block = [&](int a, int kc, int sa) {
        const bool x0 = a == 0, x1 = a == 1, x2 = a == 2;
        const int kn = sa > 0 ? min(kc + B, g) : kc - B;
        const float mn = fmaf((float)kn, x0 ? d32[0] : (x1 ? d32[1] : d32[2]), x0 ? b32[0] : (x1 ? b32[1] : b32[2]));
        q0 = x0 ? kn : q0;
        q1 = x1 ? kn : q1;
        q2 = x2 ? kn : q2;
        n0 = x0 ? mn : n0;
        n1 = x1 ? mn : n1;
        n2 = x2 ? mn : n2;
        blk += (uint32_t)(x0 ? s0 : (x1 ? bs1 : bs2));
    };
    // Cell index on axis q where the walk crosses plane ke of axis e (FP32 distance
    // te, FP64 tq on demand): the planes crossed by then are those whose
    // (distance, axis) precedes the crossing's, and their number follows from its
    // position in planes, decided in FP64 where that lies within the error bound
    // of a plane.  Never behind the start cell, whose position is rounded too.
    auto index_at = [&](int q, int sq, int start, int e, int ke, float te) {
        if (sq == 0) return start;
        const float inv = 1.f / d32[q];
        const float xp = (te - b32[q]) * inv, tx = 2.f * ((e == 0 ? E[0] : (e == 1 ? E[1] : E[2])) + E[q]) * fabsf(inv);
        int r = (int)floorf(xp);
        if (fabsf(xp - rintf(xp)) <= tx || !(tx < 0.25f)) {
            const double t = fma((double)ke, e == 0 ? d64[0] : (e == 1 ? d64[1] : d64[2]),
                                 e == 0 ? b64[0] : (e == 1 ? b64[1] : b64[2]));
            const int p = (int)fmin(fmax(rint((t - b64[q]) / d64[q]), -4.0), (double)g + 4.0);
            const double tp = fma((double)p, d64[q], b64[q]);
            const bool crossed = tp < t || (tp == t && q < e);
            r = (sq > 0) == crossed ? p : p - 1;
        }
        r = min(max(r, 0), g - 1);
        return sq > 0 ? max(r, start) : min(r, start);
    };
    // into its block on an axis: between the block planes behind and ahead
    auto in_block = [&](int i, int sq, int q) {
        return sq > 0 ? max(min(i, q - 1), (q - 1) & -B) : (sq < 0 ? min(max(i, q), min(q + B, g) - 1) : i);
    };
    const int axis0 = W.axis;
    uint32_t code = 3u;
    bool hit = false, out = false;
    bool cells = __ldg(mip + blk) != 0;  // cell by cell from here (the start cell's block), else by blocks
    int left = 4 * g + 8;                // steps of either kind: a ray crosses at most 3 g - 2 cells
    for (;;) {
        if (!cells) {
            int a, kc, sa;
            do {
                a = nearest(n0, n1, n2, q0, q1, q2);
                kc = a == 0 ? q0 : (a == 1 ? q1 : q2);
                sa = a == 0 ? s0 : (a == 1 ? s1 : s2);
                out = sa > 0 ? kc >= g : kc <= 0;
                if (!out) next_block(a, kc, sa);
            } while (!out && --left > 0 && !__ldg(mip + blk));
            code = (uint32_t)a | ((uint32_t)kc << 2);
            // the cell behind the plane, or the last one before it where the walk leaves the grid
            const float te = fmaf((float)kc, a == 0 ? d32[0] : (a == 1 ? d32[1] : d32[2]),
                                  a == 0 ? b32[0] : (a == 1 ? b32[1] : b32[2]));
            const int ia = (sa > 0) != out ? kc : kc - 1;
            i0 = a == 0 ? ia : index_at(0, s0, c0, a, kc, te);
            i1 = a == 1 ? ia : index_at(1, s1, c1, a, kc, te);
            i2 = a == 2 ? ia : index_at(2, s2, c2, a, kc, te);
            if (out || left <= 0) break;
            i0 = in_block(i0, s0, q0);
            i1 = in_block(i1, s1, q1);
            i2 = in_block(i2, s2, q2);
            cells = true;
        }
        int k0 = i0 + (s0 > 0 ? 1 : 0), k1 = i1 + (s1 > 0 ? 1 : 0), k2 = i2 + (s2 > 0 ? 1 : 0);
        float m0 = s0 ? fmaf((float)k0, d32[0], b32[0]) : inf, m1 = s1 ? fmaf((float)k1, d32[1], b32[1]) : inf,
              m2 = s2 ? fmaf((float)k2, d32[2], b32[2]) : inf;
        uint32_t lin = ((uint32_t)i2 * (uint32_t)g + (uint32_t)i1) * (uint32_t)g + (uint32_t)i0;
        while (--left > 0) {
            if (__ldg(occ + lin)) {
                hit = true;
                break;
            }
            const int a = nearest(m0, m1, m2, k0, k1, k2);
            const bool x0 = a == 0, x1 = a == 1, x2 = a == 2;
            const int kc = x0 ? k0 : (x1 ? k1 : k2), sa = x0 ? s0 : (x1 ? s1 : s2);
            const bool leaves = kc == (x0 ? q0 : (x1 ? q1 : q2));
            code = (uint32_t)a | ((uint32_t)kc << 2);
            out = leaves && (sa > 0 ? kc >= g : kc <= 0);
            if (out) break;  // the cell just tested was the last inside the grid
            i0 += x0 ? s0 : 0;
            i1 += x1 ? s1 : 0;
            i2 += x2 ? s2 : 0;
            k0 += x0 ? s0 : 0;
            k1 += x1 ? s1 : 0;
            k2 += x2 ? s2 : 0;
            lin += (uint32_t)(x0 ? s0 : (x1 ? st1 : st2));
            const float mk = fmaf((float)(kc + sa), x0 ? d32[0] : (x1 ? d32[1] : d32[2]), x0 ? b32[0] : (x1 ? b32[1] : b32[2]));
            m0 = x0 ? mk : m0;
            m1 = x1 ? mk : m1;
            m2 = x2 ? mk : m2;
            if (leaves) {
                next_block(a, kc, sa);
                cells = __ldg(mip + blk) != 0;
                if (!cells) break;
            }
        }
        if (hit || out || left <= 0) break;
    }
    // every step crosses one plane, so the cells tested follow from the last one
    const int n = 1 + abs(i0 - c0) + abs(i1 - c1) + abs(i2 - c2);
    if (!hit) {
        write_miss<double>(fd, x, y, n);
        return;
    }
    const int sa = (int)(code & 3u);
    const double kc = (double)(code >> 2);
    double t = t_in;  // the start cell is entered at the box entry
    if (sa == 0) t = fma(kc, d64[0], b64[0]);
    if (sa == 1) t = fma(kc, d64[1], b64[1]);
    if (sa == 2) t = fma(kc, d64[2], b64[2]);
    write_face_hit(fd, x, y, n, t, sa == 3 ? axis0 : sa, d);
}

// One byte per block of 2^shift cells a side: is some cell of it occupied?  A CTA
// takes 32 blocks, one per lane, so that a row's loads of `wide` bytes (8, 4 or 1:
// g and occ are multiples of it, so every row segment is aligned and whole) are
// contiguous over a warp; its warps take the z slabs in turn.  1024^3: 0.17 ms, the
// 1.07 GB it reads at the measured copy rate.
__global__ void __launch_bounds__(kBlock) voxel_mip_kernel(const uint8_t *__restrict__ occ, int g, int shift, int wide,
                                                           uint8_t *__restrict__ mip)
{
    __shared__ uint32_t s_any[kBlock / 32][32];
    const int B = 1 << shift, gb = (g + B - 1) >> shift;
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const uint32_t id = blockIdx.x * 32u + (uint32_t)lane;
    const bool part = id < (uint32_t)gb * (uint32_t)gb * (uint32_t)gb;
    uint32_t any = 0;
    if (part) {
        const uint32_t row = id / (uint32_t)gb;
        const int x0 = (int)(id - row * (uint32_t)gb) << shift, y0 = (int)(row % (uint32_t)gb) << shift;
        const int z0 = (int)(row / (uint32_t)gb) << shift;
        const int nx = min(B, g - x0), ny = min(B, g - y0), nz = min(B, g - z0);
        for (int z = wib; z < nz; z += kBlock / 32) {
            const uint8_t *p = occ + ((uint32_t)(z0 + z) * (uint32_t)g + (uint32_t)y0) * (uint32_t)g + (uint32_t)x0;
#pragma unroll 4
            for (int y = 0; y < ny; ++y, p += g) {
                if (wide == 8) {
                    const uint2 v = __ldg(reinterpret_cast<const uint2 *>(p));
                    any |= v.x | v.y;
                } else if (wide == 4) {
                    for (int x = 0; x < nx; x += 4) any |= __ldg(reinterpret_cast<const uint32_t *>(p + x));
                } else {
                    for (int x = 0; x < nx; ++x) any |= __ldg(p + x);
                }
            }
        }
    }
    s_any[wib][lane] = any;
    __syncthreads();
    if (wib == 0 && part) {
#pragma unroll
        for (int w = 1; w < kBlock / 32; ++w) any |= s_any[w][lane];
        mip[id] = any ? 1 : 0;
    }
}

// Block size of the walk, 2^shift cells a side (0: cell by cell): a ray crosses
// about 3 g / 2^shift blocks, and every block it meets that is not empty costs
// the search of its first cell.  Cell by cell / by blocks, default c, at 1080p and at
// 64x48 (us, the block occupancy included): 24^3 277 / 281 and 21 / 26, 32^3 289 / 282 and
// 27 / 26, 50^3 337 / 295 and 38 / 36, 96^3 555 / 313 and 78 / 54, 200^3 1128 / 364 and 192 /
// 86, 1024^3 9337 / 1360 and 1406 / 515; solids (a ball, a shell) 0.9 to 2.5 times as
// fast.  Scattered cells, which a Julia grid does not have, lose: noise of 3e-4 of the
// cells at 200^3 1263 / 714, of 1e-3 1247 / 1260, of 0.01 901 / 1345, of 0.1 at 1024^3 455 / 730.
// (Measured and not kept: judging the grid from 1,024 sampled rows first, which took
// 6 to 8 us of every image and left the noise 0.8 to 0.9 times as fast as cell by
// cell; going cell by cell on a ray that met too few empty blocks, 364 -> 418 us at
// 200^3.)
int mip_shift(int g) { return g >= 96 ? 3 : (g >= 24 ? 2 : 0); }

// Allocates from the stream's pool without disturbing a capture under way on
// another stream or thread: in the default mode the pool's calls are not allowed
// beside one (they fail and invalidate it), although nothing here is captured.
struct BesideCaptures {
    cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
    BesideCaptures() { swap(); }
    ~BesideCaptures() { swap(); }
    void swap() { (void)cudaThreadExchangeStreamCaptureMode(&mode); }
};

// The context's pool for block occupancies: it keeps its memory between calls (at
// most 2 MiB for each call in flight), until dqj_destroy.
bool ensure_mip_pool(dqj_ctx *ctx)
{
    if (ctx->mip_pool) return true;
    cudaMemPoolProps props{};
    props.allocType = cudaMemAllocationTypePinned;
    props.location.type = cudaMemLocationTypeDevice;
    props.location.id = ctx->device;
    cudaMemPool_t pool = nullptr;
    if (cudaMemPoolCreate(&pool, &props) != cudaSuccess) {
        (void)cudaGetLastError();
        return false;
    }
    uint64_t keep = ~0ull;
    if (cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep) != cudaSuccess) (void)cudaGetLastError();
    ctx->mip_pool = pool;
    return true;
}

}  // namespace

}  // namespace dqj

using namespace dqj;

extern "C" dqj_status dqj_render_voxels(dqj_ctx *ctx, const dqj_params *p, int32_t grid_n, const uint8_t *occupancy,
                                        const dqj_outputs *out, void *cuda_stream)
{
    return dqj::guarded([&]() -> dqj_status {
        if (!ctx) return fail(DQJ_ERR_INVALID, "ctx is NULL");
        dqj_status s = validate(p);
        if (s != DQJ_OK) return s;
        if (grid_n < 1 || grid_n > DQJ_VOXEL_MAX_GRID)
            return fail(DQJ_ERR_INVALID, "grid_n must be in 1.." + std::to_string(DQJ_VOXEL_MAX_GRID));
        if (!occupancy) return fail(DQJ_ERR_INVALID, "occupancy is NULL");
        s = check_outputs(*p, out);
        if (s != DQJ_OK) return s;
        if (ctx->device == DQJ_DEVICE_MOCK) return fail(DQJ_ERR_INVALID, "a mock context cannot render voxels");
        std::lock_guard<std::mutex> lk(ctx->mu);
        cudaError_t e = cudaSetDevice(ctx->device);
        if (e != cudaSuccess) return cuda_fail(e, "render_voxels: cudaSetDevice");
        FrameDesc fd;
        derive_frame(*p, fd, 8, 8);
        fd.pitch = out->pitch_px;
        fd.iter = out->iter;
        fd.depth = out->depth;
        fd.normal = out->normal;
        fd.rgba = out->rgba;
        GridGeom geo;
        for (int a = 0; a < 3; ++a) {
            const double ext = p->box_max[a] - p->box_min[a];
            geo.size[a] = ext / (double)grid_n;
            geo.inv_size[a] = (double)grid_n / ext;
            geo.lo_e[a] = p->box_min[a] - p->eye[a];
            geo.hi_e[a] = p->box_max[a] - p->eye[a];
        }
        // the pinhole map of the FP64 camera, 2 (x + 0.5) / W - 1 and
        // 1 - 2 (y + 0.5) / H scaled by tan(fov_y / 2) (and the aspect for x)
        geo.sxa = 2.0 * fd.d.th * fd.d.aspect / (double)p->width;
        geo.sxb = -fd.d.th * fd.d.aspect;
        geo.sya = -2.0 * fd.d.th / (double)p->height;
        geo.syb = fd.d.th;
        const dim3 grid((unsigned)((p->width + kVrTileW - 1) / kVrTileW), (unsigned)((p->height + kVrTileH - 1) / kVrTileH));
        const cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
        // The block occupancy lives for this call, allocated in stream order from
        // the context's pool (calls on several streams do not share it).  Without
        // it, under stream capture or where the pool has no memory, the walk goes
        // cell by cell.
        const int shift = mip_shift(grid_n);
        uint8_t *mip = nullptr;
        const int gb = shift ? (grid_n + (1 << shift) - 1) >> shift : 0;
        const uint32_t blocks = (uint32_t)gb * (uint32_t)gb * (uint32_t)gb;
        const BesideCaptures relaxed;
        if (shift) {
            (void)cudaGetLastError();
            cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
            e = cudaStreamIsCapturing(st, &cap);
            if (e != cudaSuccess) return cuda_fail(e, "render_voxels: cudaStreamIsCapturing");
            if (cap == cudaStreamCaptureStatusNone && ensure_mip_pool(ctx) &&
                cudaMallocFromPoolAsync(reinterpret_cast<void **>(&mip), blocks, ctx->mip_pool, st) != cudaSuccess) {
                (void)cudaGetLastError();
                mip = nullptr;
            }
        }
        if (mip) {
            const uintptr_t at = reinterpret_cast<uintptr_t>(occupancy);
            const int wide = shift == 3 && grid_n % 8 == 0 && at % 8 == 0 ? 8 : (grid_n % 4 == 0 && at % 4 == 0 ? 4 : 1);
            voxel_mip_kernel<<<(blocks + 31u) / 32u, kBlock, 0, st>>>(occupancy, grid_n, shift, wide, mip);
            if (shift == 3)
                voxel_render_blocks_kernel<3><<<grid, kBlock, 0, st>>>(fd, occupancy, grid_n, geo, mip, gb);
            else
                voxel_render_blocks_kernel<2><<<grid, kBlock, 0, st>>>(fd, occupancy, grid_n, geo, mip, gb);
            e = cudaFreeAsync(mip, st);
            if (e != cudaSuccess) return cuda_fail(e, "render_voxels: cudaFreeAsync");
        } else {
            voxel_render_kernel<<<grid, kBlock, 0, st>>>(fd, occupancy, grid_n, geo);
        }
        e = cudaGetLastError();
        if (e != cudaSuccess) return cuda_fail(e, "render_voxels: launch");
        return DQJ_OK;
    });
}
