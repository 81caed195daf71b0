// bounds_probe.cu -- the render kernels' device functions behind the recheck, one
// call per thread or warp, for tests/test_gpu_bounds.py: built beside libdqj
// from the same headers, with the library's own per-frame constants.
#include "../paper_2303_14827_gb300/csrc/render_common.cuh"
#include "../paper_2303_14827_gb300/csrc/runtime.h"

using namespace dqj;

namespace {

// t0, t1 (in units of the ray w) of ray_clip64 and the ray itself.
__global__ void clip_kernel(const __grid_constant__ FrameDesc fd, const int *x, const int *y, int n, double *t0,
                            double *t1, double *w)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    double v[3];
    ray_w<double>(fd.d, x[i], y[i], v);
    ray_clip64(fd, v, t0[i], t1[i]);
    for (int a = 0; a < 3; ++a) w[3 * i + a] = v[a];
}

// FP64 slice points of march samples (entry_point64).
__global__ void position_kernel(const __grid_constant__ FrameDesc fd, const int *x, const int *y, const int *k, int n,
                                double *out)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    double z[8];
    entry_point64(fd, make_int4(y[i] * fd.W + x[i], k[i] | (kMarchSample << 16), x[i] | (y[i] << 16), 0), z);
    for (int j = 0; j < 8; ++j) out[8 * i + j] = z[j];
}

// which: 0 count_bound64, 1 count_bound2, 2 FP64 evaluation, 3 count64.
template <int SQ, int MOD>
__global__ void count_kernel(const __grid_constant__ FrameDesc fd, int which, const double *zs, int n, int *count,
                             int *certain)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    double z[8];
    for (int j = 0; j < 8; ++j) z[j] = zs[8 * i + j];
    bool ok = true;
    int c;
    if (which == 0)
        c = count_bound64<SQ, MOD>(fd, z, ok);
    else if (which == 1)
        c = count_bound2<SQ, MOD>(fd, z, ok);
    else if (which == 2)
        c = classify_scalar<double, SQ, MOD>(z, fd.d, fd.max_iter);
    else
        c = count64<SQ, MOD>(fd, z);
    count[i] = c;
    certain[i] = ok;
}

// March sample k of pixel (x, y): its FP64 count from its FP64 position, and
// whether count_certain vouches for that count and for the next one.
template <int SQ, int MOD, bool AXIS>
__global__ void sample_kernel(const __grid_constant__ FrameDesc fd, const int *x, const int *y, const int *k, int n,
                              int *count, int *right, int *wrong)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    double z[8];
    entry_point64(fd, make_int4(y[i] * fd.W + x[i], k[i] | (kMarchSample << 16), x[i] | (y[i] << 16), 0), z);
    const int c = classify_scalar<double, SQ, MOD>(z, fd.d, fd.max_iter);
    count[i] = c;
    right[i] = count_certain<SQ, MOD, AXIS>(fd, x[i], y[i], k[i], c);
    wrong[i] = count_certain<SQ, MOD, AXIS>(fd, x[i], y[i], k[i], c + 1);
}

// The integer doublings: 2 x and 4 x of every bit pattern.
__global__ void twice_kernel(const double *x, long n, double *two, double *four)
{
    const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    two[i] = twice(x[i]);
    four[i] = four_times(x[i]);
}

// One warp: n staged entries of march samples whose FP32 count is wrong by one,
// against a queue of `cap` entries; ctr, flags and list as in a frame's scratch.
__global__ void staged_kernel(const __grid_constant__ FrameDesc fd, Scratch sc, const int4 *entries, int n)
{
    __shared__ int4 qs[kQStage];
    for (int i = threadIdx.x; i < n; i += 32) qs[i] = entries[i];
    __syncwarp();
    const int left = recheck_staged<0, 0, true>(fd, sc, qs, n, 0);
    flush_rest(fd, sc, qs, left);
}

// Samples of the frame's 8 x 8 tiles [0, tiles) that the settled blocks cover.
template <int SQ, int MOD, bool AXIS>
__global__ void settled_kernel(const __grid_constant__ FrameDesc fd, int tiles, unsigned long long *out)
{
    __shared__ TileBox box;
    const int lane = threadIdx.x, tile = blockIdx.x;
    const int x0 = tile % fd.tiles_x * fd.tile_w, y0 = tile / fd.tiles_x * fd.tile_h;
    float d[2][3], ti[2] = {0.f, 0.f}, to[2] = {0.f, 0.f};
    bool act[2];
    for (int s = 0; s < 2; ++s) {
        const int slot = lane + 32 * s, x = x0 + slot % fd.tile_w, y = y0 + slot / fd.tile_w;
        act[s] = x < fd.W && y < fd.H && camera_clip<float>(fd.f, fd.W, fd.H, x, y, d[s], ti[s], to[s]);
    }
    tile_box(fd, act[0], d[0], ti[0], to[0], act[1], d[1], ti[1], to[1], box);
    unsigned samples = 0;
    for (int kc = 0; kc <= fd.N; kc += kSettleChunk) {
        const int ke = min(kc + kSettleChunk, fd.N + 1), pairs = settle_pairs(ke - kc);
        const unsigned w = ke - kc > kSettleMin ? settle_chunk<SQ, MOD, AXIS>(fd, box, kc, ke, pairs) : 0u;
        for (int p = 0; p < pairs; ++p)
            if ((w >> (4 * p)) & 15u) samples += (unsigned)max(0, min(2, ke - (kc + 2 * (pairs * lane + p))));
    }
    samples = __reduce_add_sync(kFull, samples);
    if (lane == 0) atomicAdd(out, (unsigned long long)samples);
}

FrameDesc frame_of(const dqj_params *p)
{
    FrameDesc fd;
    derive_frame(*p, fd, 8, 8);
    return fd;
}

int done()
{
    const cudaError_t e = cudaDeviceSynchronize();
    return (int)(e != cudaSuccess ? e : cudaGetLastError());
}

}  // namespace

extern "C" {

int probe_clip(const dqj_params *p, const int *x, const int *y, int n, double *t0, double *t1, double *w)
{
    clip_kernel<<<(n + 127) / 128, 128>>>(frame_of(p), x, y, n, t0, t1, w);
    return done();
}

// The library's camera constants: forward, right and up, tan(fov_y / 2), aspect.
void probe_camera(const dqj_params *p, double *out)
{
    const FrameDesc fd = frame_of(p);
    for (int a = 0; a < 3; ++a) {
        out[a] = fd.d.fwd[a];
        out[3 + a] = fd.d.right[a];
        out[6 + a] = fd.d.upv[a];
    }
    out[9] = fd.d.th;
    out[10] = fd.d.aspect;
}

int probe_positions(const dqj_params *p, const int *x, const int *y, const int *k, int n, double *z)
{
    position_kernel<<<(n + 127) / 128, 128>>>(frame_of(p), x, y, k, n, z);
    return done();
}

int probe_count(const dqj_params *p, int which, const double *z, int n, int *count, int *certain)
{
    const FrameDesc fd = frame_of(p);
    const int g = (n + 127) / 128;
    switch (2 * p->square_mode + p->modulus_mode) {
    case 0: count_kernel<0, 0><<<g, 128>>>(fd, which, z, n, count, certain); break;
    case 1: count_kernel<0, 1><<<g, 128>>>(fd, which, z, n, count, certain); break;
    case 2: count_kernel<1, 0><<<g, 128>>>(fd, which, z, n, count, certain); break;
    default: count_kernel<1, 1><<<g, 128>>>(fd, which, z, n, count, certain); break;
    }
    return done();
}

int probe_samples(const dqj_params *p, const int *x, const int *y, const int *k, int n, int *count, int *right,
                  int *wrong)
{
    const FrameDesc fd = frame_of(p);
    const int g = (n + 127) / 128;
    auto run = [&](auto sq, auto mod) {
        if (fd.axis_slice)
            sample_kernel<sq(), mod(), true><<<g, 128>>>(fd, x, y, k, n, count, right, wrong);
        else
            sample_kernel<sq(), mod(), false><<<g, 128>>>(fd, x, y, k, n, count, right, wrong);
    };
    using Z = std::integral_constant<int, 0>;
    using O = std::integral_constant<int, 1>;
    switch (2 * p->square_mode + p->modulus_mode) {
    case 0: run(Z{}, Z{}); break;
    case 1: run(Z{}, O{}); break;
    case 2: run(O{}, Z{}); break;
    default: run(O{}, O{}); break;
    }
    return done();
}

int probe_twice(const double *x, long n, double *two, double *four)
{
    twice_kernel<<<(unsigned)((n + 127) / 128), 128>>>(x, n, two, four);
    return done();
}

// stats (DQJ_NSTATS), queue_count and dirty_count of the scratch after n <= 320
// staged entries; queue: room for `cap` entries, flags and list: one per pixel.
int probe_staged(const dqj_params *p, const int *entries, int n, int *queue, int cap, unsigned *flags, int *list,
                 unsigned long long *counters)
{
    FrameDesc fd = frame_of(p);
    fd.epoch = 1;
    Scratch sc{};
    sc.ctr = reinterpret_cast<Counters *>(counters);
    sc.queue = reinterpret_cast<int4 *>(queue);
    sc.queue_cap = (uint32_t)cap;
    sc.dirty_flag = flags;
    sc.dirty_list = list;
    sc.dirty_cap = (uint32_t)(fd.W * fd.H);
    staged_kernel<<<1, 32>>>(fd, sc, reinterpret_cast<const int4 *>(entries), n);
    return done();
}

int probe_counter_offsets(int *queue_count, int *dirty_count)
{
    *queue_count = (int)offsetof(Counters, queue_count);
    *dirty_count = (int)offsetof(Counters, dirty_count);
    return (int)sizeof(Counters);
}

// Whether the frame settles blocks, and the samples they cover (all tiles).
int probe_settled(const dqj_params *p, int *settles, unsigned long long *samples)
{
    const FrameDesc fd = frame_of(p);
    *settles = fd.settle;
    const int tiles = fd.tiles_x * fd.tiles_y;
    auto run = [&](auto sq, auto mod) {
        if (fd.axis_slice)
            settled_kernel<sq(), mod(), true><<<tiles, 32>>>(fd, tiles, samples);
        else
            settled_kernel<sq(), mod(), false><<<tiles, 32>>>(fd, tiles, samples);
    };
    using Z = std::integral_constant<int, 0>;
    using O = std::integral_constant<int, 1>;
    switch (2 * p->square_mode + p->modulus_mode) {
    case 0: run(Z{}, Z{}); break;
    case 1: run(Z{}, O{}); break;
    case 2: run(O{}, Z{}); break;
    default: run(O{}, O{}); break;
    }
    return done();
}

}  // extern "C"
