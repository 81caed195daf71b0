// settle.cuh -- settled blocks: runs of march samples whose escape count is
// proved by a bound instead of iterated.
//
// Far from the set the escape count is the same over long stretches of a ray
// and over all rays of a screen tile: of the 257 rounds of 128 samples of a
// 1080p tile only about 8 see two different counts.  The samples of a tile in
// the range [ka, kb] lie in a box of scene space: centre p, half extents h, on
// the lines between the rays' box entries and exits.  Its slice image is
//     zeta_0 = z + sum_a u_a g_a + e,   |u_a| <= 1,  |e_r| <= er, |e_d| <= ed
// (g_a = h_a E_a; e collects rounding), and one step of the iteration maps such
// a set into one of the same form:
//     z   <- z^2 + c                 (the centre's own orbit)
//     g_a <- z g_a + g_a z           (the derivative, exact to first order)
//     er  <- 2 |z_r| er + (Gr + er)^2          Gr >= |sum_a u_a g_a| (real half)
//     ed  <- 2 (|z_r| ed + |z_d| er) + 2 (Gr + er)(Gd + ed)   (algebraic square)
// because quaternion norms multiply.  The modulus over the set then lies in
//     |z|^2 +- 2 (sum_a |z . g_a| + |z_r| er + |z_d| ed)  [+ (Gr + er)^2 + (Gd + ed)^2].
// When the lower end exceeds R^2 at step n, after every earlier upper end
// stayed below it, every sample of the block escapes at exactly step n; with
// the recheck margin added to both comparisons, none of them is marginal
// either.  Rounding: er and ed grow each step by far more than FP32 (or FP64)
// evaluation of the samples and of this bound can err, so a settled count is
// the count the march computes, bit for bit, in every precision.  Whatever the
// bound cannot prove (any NaN or overflow included) is marched as before.
#pragma once

#include "dq_math.cuh"

namespace dqj {

constexpr int kSettleCap = 6;     // deepest escape step proved: deeper shells are thinner than a pair of samples
constexpr int kSettleInside = 15; // count of a box without an escape (settle_box<INSIDE>)
constexpr int kSettlePairs = 8;   // sample pairs per block at most
constexpr int kSettleChunk = 32 * 2 * kSettlePairs;  // samples settled at a time by a warp
constexpr int kSettleMin = 8;     // chunks of this many samples or fewer are marched outright
static_assert(kSettleCap < 12 && kSettleCap <= 15, "a settled count is no late step and fits four bits");

// Bounding box of a tile's samples: the samples of index k lie within
// h0 + (k / N) dh of the centre c0 + (k / N) dc, per scene axis.
struct TileBox {
    float c0[3], dc[3], h0[3], dh[3];
    float rho, e1;  // bounds of the rounding of a sample's position and of its first iterate
    int staged;     // recheck entries the warp has staged (march4_tile; not part of the box)
};

__device__ __forceinline__ float warp_min(float v)
{
    float r;
    asm volatile("redux.sync.min.f32 %0, %1, 0xffffffff;" : "=f"(r) : "f"(v));
    return r;
}
__device__ __forceinline__ float warp_max(float v)
{
    float r;
    asm volatile("redux.sync.max.f32 %0, %1, 0xffffffff;" : "=f"(r) : "f"(v));
    return r;
}
// Square root to 1e-6 relative; arguments below 1e-38 count as zero, which the
// bounds' additive rounding terms cover.
__device__ __forceinline__ float sqrt_approx(float v)
{
    float r;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(v));
    return r;
}

// Per scene axis, the range of the entry (or exit) points of a lane's rays;
// a lane without a ray passes an empty range.
__device__ __forceinline__ void box_side(const float (&lo)[3], const float (&hi)[3], float (&c)[3], float (&h)[3])
{
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const float l = warp_min(lo[a]), u = warp_max(hi[a]);
        c[a] = 0.5f * (l + u);
        h[a] = 0.5f * (u - l);
    }
}

// The box of two rays per lane (act: the half has a ray from t_in to t_out in
// direction d), written to the warp's box in shared memory (all lanes call).
__device__ __forceinline__ void tile_box(const FrameDesc &fd, bool acta, const float (&da)[3], float tia, float toa,
                                         bool actb, const float (&db)[3], float tib, float tob, TileBox &box)
{
    const float inf = __int_as_float(0x7f800000);
    TileBox B;
    float cN[3], hN[3];
#pragma unroll
    for (int s = 0; s < 2; ++s) {
        const float ta = s ? toa : tia, tb = s ? tob : tib;
        float lo[3], hi[3];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const float pa = fmaf(ta, da[a], fd.f.eye[a]), pb = fmaf(tb, db[a], fd.f.eye[a]);
            lo[a] = fminf(acta ? pa : inf, actb ? pb : inf);
            hi[a] = fmaxf(acta ? pa : -inf, actb ? pb : -inf);
        }
        if (s == 0)
            box_side(lo, hi, B.c0, B.h0);
        else
            box_side(lo, hi, cN, hN);
    }
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        B.dc[a] = cN[a] - B.c0[a];
        B.dh[a] = hN[a] - B.h0[a];
    }
    const float r = fd.settle_an + warp_max(fmaxf(acta ? toa : 0.f, actb ? tob : 0.f));
    B.rho = 4e-6f * r;
    B.e1 = 8e-6f * r * r;
    __syncwarp();  // the warp's readers of its previous tile's box are done
    if ((threadIdx.x & 31) == 0) {
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            box.c0[a] = B.c0[a];
            box.dc[a] = B.dc[a];
            box.h0[a] = B.h0[a];
            box.dh[a] = B.dh[a];
        }
        box.rho = B.rho;
        box.e1 = B.e1;
    }
    __syncwarp();
}

// Centre and half extents of the box of samples [ka, kb].
__device__ __forceinline__ void block_box(const TileBox &B, float inv_n, int ka, int kb, float (&p)[3], float (&h)[3])
{
    const float fm = 0.5f * inv_n * (float)(ka + kb), fh = 0.5f * inv_n * (float)(kb - ka);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        p[a] = fmaf(fm, B.dc[a], B.c0[a]);
        h[a] = fmaf(fh, fabsf(B.dh[a]) + fabsf(B.dc[a]), fmaf(fm, B.dh[a], B.h0[a])) + B.rho;
    }
}

// The escape count shared by every sample of the box (p, h), or 0 when it is
// not proved.  INSIDE: counts to 14, and 15 when no sample of the box escapes by
// max_iter.  The centre and the first generator advance in the halves of u,
// the other two generators in those of v.  AXIS: components 3..7 of the slice
// are zero, so the first step needs only components 0..2.
template <int SQ, int MOD, bool AXIS, bool INSIDE = false>
__device__ __forceinline__ int settle_box(const FrameDesc &fd, const float (&p)[3], const float (&h)[3], float rho,
                                          float e1)
{
    const FrameT<float> &F = fd.f;
    const float hi = fd.settle_hi, lo = fd.settle_lo, cn = fd.settle_cn;
    constexpr int nc = AXIS ? 3 : 8;
    float2 u[8], v[8];
#pragma unroll
    for (int i = 0; i < nc; ++i) {
        u[i].x = fmaf(p[2], F.E[2][i], fmaf(p[1], F.E[1][i], fmaf(p[0], F.E[0][i], F.O[i])));
        u[i].y = h[0] * F.E[0][i];
        v[i] = make_float2(h[1] * F.E[1][i], h[2] * F.E[2][i]);
    }
    // the basis is orthonormal: |sum_a u_a g_a| <= |h|
    float Gr = sqrt_approx(fmaf(h[2], h[2], fmaf(h[1], h[1], h[0] * h[0])));
    float Gd = AXIS ? 0.f : Gr;
    float er = rho, ed = AXIS ? 0.f : rho;
    float ar, ad;
    {
        float r = u[0].x * u[0].x, d = 0.f;
#pragma unroll
        for (int i = 1; i < (AXIS ? 3 : 4); ++i) r = fmaf(u[i].x, u[i].x, r);
        if (!AXIS) {
#pragma unroll
            for (int i = 4; i < 8; ++i) d = fmaf(u[i].x, u[i].x, d);
        }
        ar = sqrt_approx(r);
        ad = AXIS ? 0.f : sqrt_approx(d);
    }
    const int cap = INSIDE ? fd.max_iter : min(kSettleCap, fd.max_iter);
    const float2 two = make_float2(2.f, 2.f), neg = make_float2(-1.f, -1.f), one_two = make_float2(1.f, 2.f);
#pragma unroll 1
    for (int n = 1; n <= cap; ++n) {
        // the remainder, from the norms of this step's set
        {
            const float gr = Gr + er, gd = Gd + ed;
            const float round = 8e-6f * fmaf(ar, ar, fmaf(ad, ad, cn));
            const float ner = fmaf(1.0002f, fmaf(2.f * ar, er, gr * gr), round);
            float ned;
            if (SQ == 0)
                ned = 2.0004f * fmaf(ar, ed, fmaf(ad, er, gr * gd));
            else
                ned = 1.0002f * fmaf(2.f * ad, ed, gd * gd);
            er = ner;
            ed = ned + round;
            if (n == 1) {
                er += e1;
                ed += e1;
            }
        }
        float2 z[8];
        if (AXIS && n == 1) {
            const float2 z0 = make_float2(u[0].x, u[0].x), z1 = make_float2(u[1].x, u[1].x),
                         z2 = make_float2(u[2].x, u[2].x);
            const float2 qu = f2fma(z2, u[2], f2mul(z1, u[1])), qv = f2fma(z2, v[2], f2mul(z1, v[1]));
            const float2 u0 = make_float2(u[0].x, u[0].y), v0 = v[0];
            u[0] = f2fma(f2fma(z0, u0, f2mul(qu, neg)), one_two, make_float2(F.c[0], 0.f));
            u[1] = f2fma(f2fma(z0, u[1], f2mul(u0, z1)), one_two, make_float2(F.c[1], 0.f));
            u[2] = f2fma(f2fma(z0, u[2], f2mul(u0, z2)), one_two, make_float2(F.c[2], 0.f));
            v[0] = f2mul(f2fma(z0, v0, f2mul(qv, neg)), two);
            v[1] = f2mul(f2fma(z0, v[1], f2mul(v0, z1)), two);
            v[2] = f2mul(f2fma(z0, v[2], f2mul(v0, z2)), two);
#pragma unroll
            for (int i = 3; i < 8; ++i) {
                u[i] = make_float2(F.c[i], 0.f);
                v[i] = make_float2(0.f, 0.f);
            }
        } else {
#pragma unroll
            for (int i = 0; i < 8; ++i) z[i] = make_float2(u[i].x, u[i].x);
            // (z b + b z) / 2 of b = (z, g_0) and b = (g_1, g_2)
            auto half_sym = [&](float2(&b)[8]) {
                float2 o[8];
                float2 q = f2fma(z[3], b[3], f2fma(z[2], b[2], f2mul(z[1], b[1])));
                o[0] = f2fma(z[0], b[0], f2mul(q, neg));
#pragma unroll
                for (int i = 1; i < 4; ++i) o[i] = f2fma(z[0], b[i], f2mul(b[0], z[i]));
                if (SQ == 0) {
                    q = f2mul(z[1], b[5]);
                    q = f2fma(z[2], b[6], q);
                    q = f2fma(z[3], b[7], q);
                    q = f2fma(z[5], b[1], q);
                    q = f2fma(z[6], b[2], q);
                    q = f2fma(z[7], b[3], q);
                    o[4] = f2fma(z[0], b[4], f2fma(z[4], b[0], f2mul(q, neg)));
#pragma unroll
                    for (int i = 1; i < 4; ++i)
                        o[4 + i] = f2fma(z[0], b[4 + i], f2fma(b[4], z[i], f2fma(z[4], b[i], f2mul(b[0], z[4 + i]))));
                } else {
                    q = f2fma(z[7], b[7], f2fma(z[6], b[6], f2mul(z[5], b[5])));
                    o[4] = f2fma(z[4], b[4], f2mul(q, neg));
#pragma unroll
                    for (int i = 5; i < 8; ++i) o[i] = f2fma(z[4], b[i], f2mul(b[4], z[i]));
                }
#pragma unroll
                for (int i = 0; i < 8; ++i) b[i] = o[i];
            };
            half_sym(v);
            half_sym(u);
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                u[i] = f2fma(u[i], one_two, make_float2(F.c[i], 0.f));
                v[i] = f2mul(v[i], two);
            }
        }
        // norms of the halves and the products z . g_a
        float2 su, sv, tu, tv;
        float gr, gd;
        {
            const float2 z0 = make_float2(u[0].x, u[0].x), z4 = make_float2(u[4].x, u[4].x);
            su = f2mul(z0, u[0]);
            sv = f2mul(z0, v[0]);
            tu = f2mul(z4, u[4]);
            tv = f2mul(z4, v[4]);
            gr = fmaf(v[0].y, v[0].y, fmaf(v[0].x, v[0].x, u[0].y * u[0].y));
            gd = fmaf(v[4].y, v[4].y, fmaf(v[4].x, v[4].x, u[4].y * u[4].y));
#pragma unroll
            for (int i = 1; i < 4; ++i) {
                const float2 zi = make_float2(u[i].x, u[i].x), zj = make_float2(u[4 + i].x, u[4 + i].x);
                su = f2fma(zi, u[i], su);
                sv = f2fma(zi, v[i], sv);
                tu = f2fma(zj, u[4 + i], tu);
                tv = f2fma(zj, v[4 + i], tv);
                gr = fmaf(v[i].y, v[i].y, fmaf(v[i].x, v[i].x, fmaf(u[i].y, u[i].y, gr)));
                gd = fmaf(v[4 + i].y, v[4 + i].y, fmaf(v[4 + i].x, v[4 + i].x, fmaf(u[4 + i].y, u[4 + i].y, gd)));
            }
        }
        // |sum_a u_a g_a|^2 <= 3 sum_a |g_a|^2
        Gr = sqrt_approx(3.f * gr);
        Gd = sqrt_approx(3.f * gd);
        ar = sqrt_approx(su.x);
        ad = sqrt_approx(tu.x);
        float m, dev, sq;
        {
            const float xr = Gr + er;
            if (MOD == 0) {
                const float xd = Gd + ed;
                m = su.x + tu.x;
                dev = fabsf(su.y + tu.y) + fabsf(sv.x + tv.x) + fabsf(sv.y + tv.y) + fmaf(ar, er, ad * ed);
                sq = fmaf(xr, xr, xd * xd);
            } else {
                m = su.x;
                dev = fabsf(su.y) + fabsf(sv.x) + fabsf(sv.y) + ar * er;
                sq = xr * xr;
            }
        }
        dev = fmaf(2.0004f, dev, 1e-5f * (m + sq));
        if (m - dev > hi) return !INSIDE || n < kSettleInside ? n : 0;
        if (!(fmaf(1.0002f, sq, m + dev) < lo)) return 0;
    }
    return INSIDE ? kSettleInside : 0;
}

// Settled counts of the samples [kc, ke) of a tile, ke - kc <= kSettleChunk, in
// blocks of 2 * pairs samples (pairs = settle_pairs(ke - kc)): lane b's word
// holds the counts of block b's pairs, four bits each (0: not settled).  Whole
// blocks first, one per lane; the pairs of the blocks left over then, four
// blocks at a time.
__device__ __forceinline__ int settle_pairs(int samples) { return min(kSettlePairs, ((samples + 1) / 2 + 31) / 32); }

template <int SQ, int MOD, bool AXIS>
__device__ __forceinline__ unsigned settle_chunk(const FrameDesc &fd, const TileBox &B, int kc, int ke, int pairs)
{
    const int lane = threadIdx.x & 31;
    const float inv_n = 1.f / (float)fd.N;
    unsigned w = 0, todo = 0;
#pragma unroll 1
    for (bool whole = true;; whole = false) {
        int ka, kb, src = -1;
        bool valid;
        if (whole) {
            ka = kc + 2 * pairs * lane;
            kb = min(ka + 2 * pairs, ke) - 1;
            valid = ka < ke;
        } else {
            if (todo == 0) break;
            int blk = 32;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int bj = todo ? __ffs(todo) - 1 : 32;
                todo &= todo - 1;
                if ((lane >> 3) == j) blk = bj;
                if (lane == bj) src = 8 * j;
            }
            ka = kc + 2 * pairs * blk + 2 * (lane & 7);
            kb = min(ka + 1, ke - 1);
            valid = blk < 32 && (lane & 7) < pairs && ka < ke;
        }
        int n = 0;
        if (valid) {
            float p[3], h[3];
            block_box(B, inv_n, ka, kb, p, h);
            n = settle_box<SQ, MOD, AXIS>(fd, p, h, B.rho, B.e1);
        }
        __syncwarp();
        if (whole) {
            w = (unsigned)n * 0x11111111u;
            if (pairs == 1) break;
            todo = __ballot_sync(0xffffffffu, valid && n == 0);
        } else {
            unsigned v = (unsigned)n << (4 * (lane & 7));
            v |= __shfl_xor_sync(0xffffffffu, v, 1);
            v |= __shfl_xor_sync(0xffffffffu, v, 2);
            v |= __shfl_xor_sync(0xffffffffu, v, 4);
            const unsigned t = __shfl_sync(0xffffffffu, v, src < 0 ? 0 : src);
            if (src >= 0) w = t;
        }
    }
    return w;
}

// Bits 4p set: pair p of a lane's block has samples in [kc, ke) and is not settled.
__device__ __forceinline__ unsigned open_pairs(unsigned w, int kc, int ke, int pairs)
{
    const int ka = kc + 2 * pairs * (int)(threadIdx.x & 31);
    const int np = min(max((ke - ka + 1) / 2, 0), pairs);
    const unsigned t = w | (w >> 1);
    const unsigned open = ~(t | (t >> 2)) & 0x11111111u;
    return np >= 8 ? open : open & ((1u << (4 * np)) - 1u);
}

// Over the settled pairs p < p_end of a lane's block: the sum of (count - 1)
// over their samples, and the largest count - 1.
__device__ __forceinline__ void settled_sum(unsigned w, int kc, int ke, int pairs, int p_end, int &sum, int &mx)
{
    const int ka = kc + 2 * pairs * (int)(threadIdx.x & 31);
    sum = mx = 0;
#pragma unroll
    for (int p = 0; p < kSettlePairs; ++p) {
        const int n = (int)((w >> (4 * p)) & 15u), left = ke - (ka + 2 * p);
        if (n && p < p_end && p < pairs && left > 0) {
            sum += (n - 1) * min(left, 2);
            mx = max(mx, n - 1);
        }
    }
}

// The settled samples of the chunk before pair p of block b (b = 32: all of
// them), over the warp; every lane gets the same values.
__device__ __forceinline__ void settled_before(unsigned w, int kc, int ke, int pairs, int b, int p, int &sum, int &mx)
{
    const int lane = threadIdx.x & 31;
    settled_sum(w, kc, ke, pairs, lane < b ? kSettlePairs : (lane == b ? p : 0), sum, mx);
    sum = __reduce_add_sync(0xffffffffu, sum);
    mx = __reduce_max_sync(0xffffffffu, mx);
}

}  // namespace dqj
