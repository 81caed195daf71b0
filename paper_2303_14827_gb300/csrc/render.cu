// render.cu -- launches of a frame's passes: the algebraic square's kernels
// (render_passes.cuh), and the choices that hold for every form.  The
// component-wise square's kernels compile beside it in render_componentwise.cu.
#include "render_passes.cuh"

namespace dqj {

namespace {
int march_samples_env()  // DQJ_MARCH_SAMPLES, or -1
{
    static const int n = [] {
        const char *e = std::getenv("DQJ_MARCH_SAMPLES");
        return e ? (int)std::strtol(e, nullptr, 10) : -1;
    }();
    return n;
}
}  // namespace

int march_samples_per_round() { return march_samples_env() == 1 ? 1 : 2; }

bool bounds_decide()
{
    static const bool on = [] {
        const char *e = std::getenv("DQJ_BOUNDS");
        return !(e && e[0] == '0');
    }();
    return on;
}

bool march_settles() { return bounds_decide() && march_samples_env() != 0 && march_samples_env() != 1; }

int march_split(const FrameDesc &fd, int num_sms)
{
    static std::atomic<int> g_occ{0};
    if (fd.precision != DQJ_FP32 || fd.march_variant != 1 || fd.traversal != DQJ_TRAVERSAL_MARCH) return 1;
    if (const char *e = std::getenv("DQJ_MARCH_SPLIT")) {  // 0: never split; n > 1: n ranges
        const long n = std::strtol(e, nullptr, 10);
        if (n <= 1) return 1;
        return (int)std::min<long>(std::min<long>(n, 64), (long)fd.N + 1);
    }
    static std::atomic<int> g_occ4{0};
    const int per_sm = fd.march_samples == 2 ? resident_per_sm(g_occ4, march4_split_kernel<0, 0, true>)
                                             : resident_per_sm(g_occ, march2_split_kernel<0, 0, true>);
    const long long warps = (long long)num_sms * per_sm * (kBlock / 32);
    const long long tiles = subset_tiles(fd, (unsigned)fd.tiles_x * (unsigned)fd.tiles_y);
    if (tiles >= warps || tiles == 0) return 1;
    // about four waves of items: later waves skip the rays earlier ranges hit
    const long long p = (4 * warps + tiles - 1) / tiles;
    return (int)std::min<long long>(std::min<long long>(p, 16), (long long)fd.N + 1);
}

cudaError_t launch_frame(const FrameDesc &fd, const Scratch &sc, cudaStream_t st, int num_sms, cudaEvent_t *ev)
{
    if (fd.traversal == DQJ_TRAVERSAL_DE) return launch_de(fd, sc, st, num_sms, ev);
    if (fd.square_mode != DQJ_SQUARE_ALGEBRAIC) return launch_componentwise(fd, sc, st, num_sms, ev);
    return fd.modulus_mode == DQJ_MODULUS_EUCLID8 ? launch_mode<0, 0>(fd, sc, st, num_sms, ev)
                                                  : launch_mode<0, 1>(fd, sc, st, num_sms, ev);
}

}  // namespace dqj
