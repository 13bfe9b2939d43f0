// fft_tma_256.cu -- instantiations of the asynchronous-output stage kernel
// (fft_warp_tma.cuh) for 256-point lines.
#include "fft_warp_tma.cuh"

namespace ofg {

cudaError_t launch_warp_tma_256(const StageLaunch& L, cudaStream_t st, bool* handled)
{
    // tiles of 4 lines whether the plan asks for 4 or 8: a CTA of 8 waits at its
    // barriers for twice the warps (512^3 3785 us against 3757, 256^3 456 against 431,
    // with persistent CTAs)
    if (L.args.G >= 4) return launch_warp_tma_n<256, 4>(L, st, handled);
    *handled = false;
    return cudaSuccess;
}

}  // namespace ofg
