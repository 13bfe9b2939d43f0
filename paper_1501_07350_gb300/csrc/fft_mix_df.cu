// fft_mix_df.cu -- the any-length stage kernel (fft_mix.cuh) in packed double-float.
#include "fft_mix_launch.cuh"

namespace ofg {

cudaError_t launch_mix_df(const StageLaunch& L, cudaStream_t st, bool* handled)
{
    *handled = false;
    if (L.args.n > kMaxLen) return cudaSuccess;
    // tiles of 8 lines (128-byte rows in the transposed output) while an SM holds four
    // of them, else of 4: 240^3 513 against 521 us, 448^3 3404 against 3800
    if (L.args.G >= 8 && mix_launch<ArDP, 8>(L.args.n).per_sm >= 4) return launch_mix_g<ArDP, 8>(L, st, handled);
    return L.args.G >= 4 ? launch_mix_g<ArDP, 4>(L, st, handled) : cudaSuccess;
}

}  // namespace ofg
