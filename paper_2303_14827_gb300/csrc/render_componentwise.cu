// render_componentwise.cu -- the passes of a frame with the component-wise square
// (DQJ_SQUARE_PAPER_COMPONENTWISE), a translation unit of its own so that the
// two squares compile in parallel.
#include "render_passes.cuh"

namespace dqj {

cudaError_t launch_componentwise(const FrameDesc &fd, const Scratch &sc, cudaStream_t st, int num_sms,
                                 cudaEvent_t *ev)
{
    return fd.modulus_mode == DQJ_MODULUS_EUCLID8 ? launch_mode<1, 0>(fd, sc, st, num_sms, ev)
                                                  : launch_mode<1, 1>(fd, sc, st, num_sms, ev);
}

}  // namespace dqj
