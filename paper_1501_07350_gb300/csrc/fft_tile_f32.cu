// fft_tile_f32.cu -- instantiations of the specialised stage kernels for one arithmetic:
// warp-per-line kernels for power-of-two lengths, tile kernels for the others.
#include "fft_tile.cuh"
#include "fft_warp.cuh"

namespace ofg {

cudaError_t launch_tile_f32(const StageLaunch& L, cudaStream_t st, bool* handled)
{
    *handled = false;
    // fft_mix also takes the longer power-of-two lengths (with the warp kernel 256^3 took
    // 172-198 us and 512^3 1590-1650, with fft_mix then 156 and 1460), and 64 and 128 points
    // where there are lines enough to fill the chip several times (512x64x512 161 against
    // 173, 512x128x512 310 against 321; 128^3, 16384 lines, 24.3 against 25.3).  64^3 (4096
    // lines) takes 10.1 against 7.3 us, 128x128x64 (8192 to 16384) 14.7 against 14.2.
    const int64_t lines = choice_lines(L);
    if (L.family == KERNEL_AUTO && (L.args.n >= 256 || (L.args.n == 64 && lines >= 32768) || (L.args.n == 128 && lines >= 16384))) {
        cudaError_t e = launch_mix_f32(L, st, handled);
        if (*handled || e) return e;
    }
    if ((L.family == KERNEL_AUTO || L.family == KERNEL_WARP) && (L.args.G == 8 || L.args.G == 16)) {
        cudaError_t e = L.args.G == 8 ? launch_warp_g<ArF32, 8>(L, st, handled) : launch_warp_g<ArF32, 16>(L, st, handled);
        if (*handled || e) return e;
    }
    if (L.family == KERNEL_AUTO) {
        cudaError_t e = launch_mix_f32(L, st, handled);
        if (*handled || e) return e;
    }
    if (L.family == KERNEL_WARP) return cudaSuccess;
    if (L.args.G == 8) return launch_tile_g<ArF32, 8>(L, st, handled);
    if (L.args.G == 16) return launch_tile_g<ArF32, 16>(L, st, handled);
    return cudaSuccess;
}

}  // namespace ofg
