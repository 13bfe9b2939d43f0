// fft_tile_df.cu -- instantiations of the specialised stage kernels for one arithmetic:
// warp-per-line kernels for power-of-two lengths, tile kernels for the others.
// The double-float warp kernels run the packed-lane policy (arith_pair.cuh);
// 256- and 512-point lines take the asynchronous-output kernel
// (fft_warp_tma.cuh, fft_tma_*.cu) whenever the stage's output has its view.
#include "fft_tile.cuh"
#include "fft_warp.cuh"

namespace ofg {

cudaError_t launch_tile_df(const StageLaunch& L, cudaStream_t st, bool* handled)
{
    *handled = false;
    if ((L.family == KERNEL_AUTO || L.family == KERNEL_WARP) && (L.args.n == 256 || L.args.n == 512)) {
        cudaError_t e = L.args.n == 256 ? launch_warp_tma_256(L, st, handled) : launch_warp_tma_512(L, st, handled);
        if (*handled || e) return e;
    }
    // a tile of the warp kernel is one warp of 32-point lines, two of 64-point ones: with
    // few lines it leaves the chip nearly empty, and fft_mix's tiles are faster (32^3 10.1
    // against 11.1 us, 64x32x32 11.4 against 12.2, 32x32x64 10.8 against 12.2, 64x64x32 12.3
    // against 12.8).  Above, the warp kernel: 64^3, 4096 lines, 13.6 against 15.2, 32x32x256,
    // 8192 of 32 points, 14.7 against 16.3, 128x128x32 21.7 against 25.6.
    const int64_t lines = choice_lines(L);
    if (L.family == KERNEL_AUTO && ((L.args.n == 32 && lines <= 4096) || (L.args.n == 64 && lines <= 2048))) {
        cudaError_t e = launch_mix_df(L, st, handled);
        if (*handled || e) return e;
    }
    if ((L.family == KERNEL_AUTO || L.family == KERNEL_WARP) && (L.args.G == 4 || L.args.G == 8)) {
        cudaError_t e = L.args.G == 4 ? launch_warp_g<ArDP, 4>(L, st, handled) : launch_warp_g<ArDP, 8>(L, st, handled);
        if (*handled || e) return e;
    }
    if (L.family == KERNEL_AUTO) {
        cudaError_t e = launch_mix_df(L, st, handled);
        if (*handled || e) return e;
    }
    if (L.family == KERNEL_WARP) return cudaSuccess;
    if (L.args.G == 4) return launch_tile_g<ArDF, 4>(L, st, handled);
    if (L.args.G == 8) return launch_tile_g<ArDF, 8>(L, st, handled);
    return cudaSuccess;
}

}  // namespace ofg
