// fft_mix_f32.cu -- the any-length stage kernel (fft_mix.cuh) in FP32.
#include "fft_mix_launch.cuh"

namespace ofg {

cudaError_t launch_mix_f32(const StageLaunch& L, cudaStream_t st, bool* handled)
{
    *handled = false;
    if (L.args.n > kMaxLen) return cudaSuccess;
    // tiles of 8 lines: as fast as 16 up to 96 points, 5-15 % faster above
    return L.args.G >= 8 ? launch_mix_g<ArF32, 8>(L, st, handled) : cudaSuccess;
}

}  // namespace ofg
