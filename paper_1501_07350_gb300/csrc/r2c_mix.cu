// r2c_mix.cu -- launches of the real stages of any length (r2c_mix.cuh).
#include "fft_mix_launch.cuh"
#include "r2c_mix.cuh"

namespace ofg {

namespace {

template <class A, int G>
MixLaunch real_launch(int n)
{
    static std::atomic<const MixLaunch*> made[kMaxLen + 1] = {};
    return kept_launch(made, n, [](int len) {
        MixLaunch l;
        l.plan = mix_radix_plan(len, sizeof(typename A::C) >= 16);
        l.smem = real_tile_bytes<A, G>(len);
        size_launch(l, G);
        return l;
    });
}

template <class A, int G>
cudaError_t launch_real_g(const StageLaunch& L, cudaStream_t st, bool* handled)
{
    const MixLaunch ml = real_launch<A, G>(L.args.n);
    if (ml.plan.npass == 0) return cudaSuccess;
    const bool fwd = L.family == KERNEL_R2C;
    static int cached[2][kMaxDevices] = {};
    const void* kern = fwd ? (const void*)real_mix_kernel<A, G, true> : (const void*)real_mix_kernel<A, G, false>;
    if (cudaError_t e = prepare_kernel(kern, device_slot(cached[fwd]))) return e;
    *handled = true;
    const int64_t ntiles = (L.args.M1 + 2 * G - 1) / (2 * G);
    // 180x200x225 double forward 200 us with one share a CTA, 195 with 4, 201 with 8
    const unsigned grid = (unsigned)tile_grid<A>(ntiles, (int64_t)L.sms * ml.per_sm, 4);
    return fwd ? launch_chained(L, real_mix_kernel<A, G, true>, grid, ml.threads, ml.smem, st, L.args, ml.plan, ntiles)
               : launch_chained(L, real_mix_kernel<A, G, false>, grid, ml.threads, ml.smem, st, L.args, ml.plan, ntiles);
}

}  // namespace

cudaError_t launch_real_mix(const StageLaunch& L, cudaStream_t st, bool* handled)
{
    *handled = false;
    const int mid = L.arith == ARITH_F32 ? FMT_C64 : FMT_DF;
    if (L.arith == ARITH_F64 || L.args.n > kMaxLen || (L.family == KERNEL_C2R && L.args.in_fmt != mid)) return cudaSuccess;
    if (L.arith == ARITH_F32) return launch_real_g<ArF32, 8>(L, st, handled);
    if (real_launch<ArDP, 8>(L.args.n).per_sm >= 4) return launch_real_g<ArDP, 8>(L, st, handled);
    return launch_real_g<ArDP, 4>(L, st, handled);
}

}  // namespace ofg
