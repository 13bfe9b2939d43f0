// fft_mix_launch.cuh -- launch rule of the stage kernel of fft_mix.cuh.
#pragma once
#include <algorithm>
#include <atomic>
#include <new>

#include "fft_mix.cuh"

namespace ofg {

// What a launch on lines of one length needs.
struct MixLaunch {
    MixPlan plan;               // npass = 0: no launch
    int threads, per_sm;
    size_t smem;
};

// CTAs of 128 threads, or of 256 or 512 where an SM would hold fewer than 512
// threads, and no more than the passes have butterflies for.  Sweeps of every count
// on cubes of 36..448 points put 128 threads first or within 3 % almost
// everywhere: 320^3 complex64 330 us, 350 with 64 or 192; 448^3 complex128
// 3404 us with 256 (three CTAs per SM), 3561 with 128.
inline void size_launch(MixLaunch& l, int G)
{
    l.threads = l.per_sm = 0;
    if (l.smem > 200 * 1024) l.plan.npass = 0;
    if (l.plan.npass == 0) return;
    int nbf = 1;
    for (int p = 0; p < l.plan.npass; ++p) nbf = std::max(nbf, l.plan.pass[p].nbf);
    const int smem_ctas = (int)(227 * 1024 / (l.smem + 1024));
    int T = 128;
    while (T < kMixMaxThreads && smem_ctas * T < 512) T *= 2;
    T = std::min(T, (G * nbf + 31) / 32 * 32);
    l.threads = T;
    l.plan.slots = T / G;
    l.per_sm = std::min({32, 65536 / (64 * T), smem_ctas});
}

template <class A, int G>
MixLaunch make_launch(int n)
{
    MixLaunch l;
    l.plan = mix_radix_plan(n, sizeof(typename A::C) >= 16);
    l.smem = (2 * (size_t)G * Mix<A, G>::pitch(n) + n) * sizeof(typename A::C);
    size_launch(l, G);
    return l;
}

// The launch of length n that `make` makes, made on its first use and kept in `made`
// (kMaxLen + 1 entries); two threads may both make one, and one is kept.  Without host
// memory to keep it in, it is made again at the next call.
template <class Make>
MixLaunch kept_launch(std::atomic<const MixLaunch*>* made, int n, Make make)
{
    const MixLaunch* kept = made[n].load(std::memory_order_acquire);
    if (kept) return *kept;
    const MixLaunch l = make(n);
    const MixLaunch* mine = new (std::nothrow) MixLaunch(l);
    if (mine && !made[n].compare_exchange_strong(kept, mine, std::memory_order_acq_rel)) delete mine;
    return l;
}

template <class A, int G>
MixLaunch mix_launch(int n)
{
    static std::atomic<const MixLaunch*> made[kMaxLen + 1] = {};
    return kept_launch(made, n, make_launch<A, G>);
}

// A kernel's dynamic shared-memory limit and carveout, set once per device.
inline cudaError_t prepare_kernel(const void* kern, int* slot, int max_smem = 200 * 1024)
{
    if (slot && *slot) return cudaSuccess;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, max_smem);
    if (!e) e = cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
    if (!e && slot) *slot = 1;
    return e;
}

template <class A, int G, bool REPEAT>
cudaError_t launch_mix_r(const StageLaunch& L, cudaStream_t st, bool* handled)
{
    const MixLaunch ml = mix_launch<A, G>(L.args.n);
    if (ml.plan.npass == 0) return cudaSuccess;
    auto kern = fft_mix_kernel<A, G, REPEAT>;
    static int cached[kMaxDevices] = {};          // 1 once the kernel's attributes are set on the device
    if (cudaError_t e = prepare_kernel((const void*)kern, device_slot(cached))) return e;
    StageArgs a = L.args;
    const int64_t Mg = a.group_i2 ? a.M2 : a.M1;
    a.ngroups = (Mg + G - 1) / G;
    const int64_t ntiles = a.ngroups * (a.group_i2 ? a.M1 : a.M2) * (REPEAT ? a.M3 : 1);
    if (ntiles > 0x7fffffffLL) return cudaSuccess;      // tiles are counted in 32 bits
    *handled = true;
    const int64_t grid = tile_grid<A>(ntiles, (int64_t)L.sms * ml.per_sm);
    // FP32 stages of contiguous output: with lines across the lanes a warp's store of the
    // last pass touches 8 lines of 128 bytes, and the stage took 68 us of 256^3 (transposed
    // ones 53), bound by its stores' wavefronts; along a line it touches two, for a few
    // conflicts of its twiddle loads.  256^3 154.5 -> 138.5 us, 512^3 1450 -> 1311,
    // 240x288x320 213 -> 192, 180x200x225 83.8 -> 80.6; where the pass has butterflies for
    // fewer than 7 of 8 threads of a line it gains nothing.  A choice at run time: as a
    // kernel of its own, whose code each transform loads anew, 256^3 took 149.5.
    const bool rows = a.contig_store && ml.plan.pass[ml.plan.npass - 1].nbf * 8 >= ml.plan.slots * 7;
    return launch_chained(L, kern, (unsigned)grid, ml.threads, ml.smem, st, a, ml.plan, ntiles, rows);
}

template <class A, int G>
cudaError_t launch_mix_g(const StageLaunch& L, cudaStream_t st, bool* handled)
{
    return L.args.M3 > 1 ? launch_mix_r<A, G, true>(L, st, handled) : launch_mix_r<A, G, false>(L, st, handled);
}

}  // namespace ofg
