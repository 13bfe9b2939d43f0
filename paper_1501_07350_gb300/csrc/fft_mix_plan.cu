// fft_mix_plan.cu -- radix plans of the stage kernel of fft_mix.cuh.
#include "fft_mix.cuh"

#include <iterator>

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
// Plans are made in the calls that execute transforms: no container, nothing that throws.
struct Radices {
    int r[kMixMaxPasses];
    int count = 0;
    float cost(float pass) const
    {
        float c = pass * count;
        for (int i = 0; i < count; ++i) c += r[i];
        return c;
    }
};

void mix_search(const int* radix, int kinds, int rest, float pass, Radices& cur, Radices& best)
{
    if (rest == 1) {
        if (best.count == 0 || cur.cost(pass) < best.cost(pass)) best = cur;
        return;
    }
    if (cur.count == kMixMaxPasses) return;
    for (int i = 0; i < kinds; ++i) {
        const int R = radix[i];
        if (rest % R || (cur.count && R > cur.r[cur.count - 1])) continue;
        cur.r[cur.count++] = R;
        mix_search(radix, kinds, rest / R, pass, cur, best);
        --cur.count;
    }
}

}  // namespace

MixPlan mix_radix_plan(int n, bool df)
{
    MixPlan pl;
    pl.npass = 0;
    pl.slots = 1;
    Radices cur, best;
    if (n == 1) best.r[best.count++] = 1;
    else if (df) mix_search(kRadixDF, (int)std::size(kRadixDF), n, n <= 64 ? 1.5f : (n <= 100 ? 3.5f : 6.5f), cur, best);
    else mix_search(kRadixF32, (int)std::size(kRadixF32), n, 100.f, cur, best);
    int m = 1;
    for (int i = 0; i < best.count; ++i) {
        const int R = best.r[i];
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

}  // namespace ofg
