// fft_mix.cu -- radix plans, launch rule and instantiations of the stage kernel of
// fft_mix.cuh.
#include "fft_mix.cuh"

#include <algorithm>
#include <atomic>
#include <iterator>
#include <vector>

namespace ofg {

namespace {

// Radices the passes are compiled for, largest first.
constexpr int kRadixDF[] = {10, 8, 7, 6, 5, 4, 3, 2};
constexpr int kRadixF32[] = {16, 15, 12, 10, 9, 8, 7, 6, 5, 4, 3, 2};

// Plans of `rest` with radices no larger than the last one, the largest first (the
// first pass has no twiddles): the cheapest sum of radices and passes, each pass
// weighing `pass`.  FP32 takes the fewest passes (its passes are short and wait on
// shared memory) and among those similar radices: 288 = 8 6 6 took 246 us a 288^3
// transform, 12 12 2 317.  In double-float a pass weighs 6.5, 3.5 up to 100
// points and 1.5 up to 64, where more threads with less to do each win: 48^3 took
// 12.1 us as 4 4 3, 15.1 as 8 6; 80^3 29 as 5 4 4, 36 as 10 8; 144^3 110 as 8 6 3, 115
// as 4 4 3 3.
void mix_search(const int* radix, int count, int rest, float pass, std::vector<int>& cur, std::vector<int>& best)
{
    if (rest == 1) {
        auto cost = [pass](const std::vector<int>& v) { float s = pass * v.size(); for (int r : v) s += r; return s; };
        if (best.empty() || cost(cur) < cost(best)) best = cur;
        return;
    }
    for (int i = 0; i < count; ++i) {
        const int R = radix[i];
        if (rest % R || (!cur.empty() && R > cur.back())) continue;
        cur.push_back(R);
        mix_search(radix, count, rest / R, pass, cur, best);
        cur.pop_back();
    }
}

MixPlan make_plan(const int* radix, int count, float pass, int n)
{
    MixPlan pl;
    pl.npass = 0;
    pl.slots = 1;
    std::vector<int> cur, best;
    mix_search(radix, count, n, pass, cur, best);
    if (best.size() > (size_t)kMixMaxPasses) return pl;
    int m = 1;
    for (int R : best) {
        MixPass& ps = pl.pass[pl.npass++];
        ps.radix = R;
        ps.nbf = n / R;
        ps.m = m;
        ps.s = n / (m * R);
        ps.inv = ((1u << 20) + (uint32_t)m - 1) / (uint32_t)m;
        m *= R;
    }
    return pl;
}

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
template <class A, int G>
MixLaunch make_launch(const int* radix, int count, float pass, int n)
{
    MixLaunch l;
    l.plan = make_plan(radix, count, pass, n);
    l.smem = (2 * (size_t)G * Mix<A, G>::pitch(n) + n) * sizeof(typename A::C);
    l.threads = l.per_sm = 0;
    if (l.smem > 200 * 1024) l.plan.npass = 0;
    if (l.plan.npass == 0) return l;
    int nbf = 1;
    for (int p = 0; p < l.plan.npass; ++p) nbf = std::max(nbf, l.plan.pass[p].nbf);
    const int smem_ctas = (int)(227 * 1024 / (l.smem + 1024));
    int T = 128;
    while (T < kMixMaxThreads && smem_ctas * T < 512) T *= 2;
    T = std::min(T, (G * nbf + 31) / 32 * 32);
    l.threads = T;
    l.plan.slots = T / G;
    l.per_sm = std::min({32, 65536 / (64 * T), smem_ctas});
    return l;
}

// Each length's launch is made on its first use and kept (at most kMaxLen of them
// per arithmetic and tile width); two threads may both make one, and one is kept.
template <class A, int G>
const MixLaunch& mix_launch(int n)
{
    static std::atomic<const MixLaunch*> made[kMaxLen + 1] = {};
    const MixLaunch* l = made[n].load(std::memory_order_acquire);
    if (l) return *l;
    constexpr bool df = sizeof(typename A::C) >= 16;
    const MixLaunch* mine =
        new MixLaunch(df ? make_launch<A, G>(kRadixDF, (int)std::size(kRadixDF), n <= 64 ? 1.5f : (n <= 100 ? 3.5f : 6.5f), n)
                         : make_launch<A, G>(kRadixF32, (int)std::size(kRadixF32), 100.f, n));
    if (made[n].compare_exchange_strong(l, mine, std::memory_order_acq_rel)) return *mine;
    delete mine;
    return *l;
}

template <class A, int G, bool REPEAT>
cudaError_t launch_mix_r(const StageLaunch& L, cudaStream_t st, bool* handled)
{
    const MixLaunch& ml = mix_launch<A, G>(L.args.n);
    if (ml.plan.npass == 0) return cudaSuccess;
    auto kern = fft_mix_kernel<A, G, REPEAT>;
    static int cached[kMaxDevices] = {};          // 1 once the kernel's attributes are set on the device
    int* slot = device_slot(cached);
    if (!slot || !*slot) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
        if (!e) e = cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
        if (e) return e;
        if (slot) *slot = 1;
    }
    StageArgs a = L.args;
    const int64_t Mg = a.group_i2 ? a.M2 : a.M1;
    a.ngroups = (Mg + G - 1) / G;
    const int64_t ntiles = a.ngroups * (a.group_i2 ? a.M1 : a.M2) * (REPEAT ? a.M3 : 1);
    if (ntiles > 0x7fffffffLL) return cudaSuccess;      // tiles are counted in 32 bits
    *handled = true;
    const int64_t grid = std::max<int64_t>(1, std::min<int64_t>((int64_t)L.sms * ml.per_sm, ntiles));
    return launch_chained(kern, (unsigned)grid, ml.threads, ml.smem, st, a, ml.plan, ntiles);
}

template <class A, int G>
cudaError_t launch_mix_g(const StageLaunch& L, cudaStream_t st, bool* handled)
{
    return L.args.M3 > 1 ? launch_mix_r<A, G, true>(L, st, handled) : launch_mix_r<A, G, false>(L, st, handled);
}

}  // namespace

cudaError_t launch_mix_df(const StageLaunch& L, cudaStream_t st, bool* handled)
{
    *handled = false;
    if (L.args.n < 2 || L.args.n > kMaxLen) return cudaSuccess;
    // tiles of 8 lines (128-byte rows in the transposed output) while an SM holds four
    // of them, else of 4: 240^3 513 against 521 us, 448^3 3404 against 3800
    if (L.args.G >= 8 && mix_launch<ArDP, 8>(L.args.n).per_sm >= 4) return launch_mix_g<ArDP, 8>(L, st, handled);
    return L.args.G >= 4 ? launch_mix_g<ArDP, 4>(L, st, handled) : cudaSuccess;
}

cudaError_t launch_mix_f32(const StageLaunch& L, cudaStream_t st, bool* handled)
{
    *handled = false;
    if (L.args.n < 2 || L.args.n > kMaxLen) return cudaSuccess;
    // tiles of 8 lines: as fast as 16 up to 96 points, 5-15 % faster above
    return L.args.G >= 8 ? launch_mix_g<ArF32, 8>(L, st, handled) : cudaSuccess;
}

}  // namespace ofg
