// r2c_mix.cuh -- the real stages of the real transform (r2c.cu) for any line length,
// on the passes of the any-length stage kernel (fft_mix.cuh), in packed double-float
// and FP32.
//
// A tile is G complex lines, each a pair of real lines (see r2c.cu for the algebra).
//   Forward: 2G real lines are copied in as they are; the first pass reads two reals
//   per value, the last one leaves the spectra Z in shared memory, and the CTA
//   separates them and stores frequency k of the tile's 2G real lines as 2G
//   consecutive elements.
//   Inverse: 2G half lines are copied in; the first pass forms the Hermitian
//   extension as it reads (no pass of its own); the last leaves z in shared memory,
//   and each warp writes whole real lines.
// The copies of the next tile go into the raw buffer, free once the first pass has
// read it, and overlap all later passes and the stores.
//
// The forward stage moves n reals in and n/2 + 1 complex elements out a line, the
// inverse the reverse; both are bound by the passes' instructions and shared-memory
// traffic (180x200x225 inverse in float: the stage takes 31 us with 56 % of issue slots
// busy, 18.6 warps on an SM).  Whole real transforms, generic kernel before -> now:
// 240^3 double 338 -> 310 us, inverse 341 -> 315, float 111 -> 85, inverse 112 -> 89;
// 256x256x360 double 536 -> 422, float 196 -> 134; 180x200x225 inverse float 75 -> 61.
#pragma once
#include "fft_mix.cuh"

namespace ofg {

// Two real values <-> one complex element; scale in the form `part` applies it.
template <class A> struct MixReal;

template <> struct MixReal<ArF32> {
    using T = float;
    using Scale = float2;
    __device__ __forceinline__ static float2 make(float a, float b) { return make_float2(a, b); }
    // u + i v (up), conj u + i conj v (not up), or Re u + i Re v (edge)
    __device__ __forceinline__ static float2 extend(float2 u, float2 v, bool up, bool edge)
    {
        const float uy = edge ? 0.f : (up ? u.y : -u.y), vy = edge ? 0.f : (up ? v.y : -v.y);
        return make_float2(u.x - vy, uy + v.x);
    }
    __device__ __forceinline__ static Scale scale_of(const StageArgs& p) { return make_float2(p.scale_hi, p.scale_lo); }
    __device__ __forceinline__ static void parts(float2 z, Scale s, float& re, float& im)
    {
        re = fmaf(z.x, s.x, z.x * s.y);
        im = fmaf(z.y, s.x, z.y * s.y);
    }
};

template <> struct MixReal<ArDP> {
    using T = double;
    using Scale = float2;
    __device__ __forceinline__ static ArDP::C make(double a, double b)
    {
        const float2 ha = split_f64(a), hb = split_f64(b);
        return ArDP::make(p2_pack(ha.x, hb.x), p2_pack(ha.y, hb.y));
    }
    __device__ __forceinline__ static ArDP::C extend(ArDP::C u, ArDP::C v, bool up, bool edge)
    {
        // (u.re, +-u.im) + (-+v.im, v.re)
        const u64 ku = edge ? 0x00000000FFFFFFFFull : ~0ull, kv = edge ? 0xFFFFFFFF00000000ull : ~0ull;
        const u64 su = up ? 0ull : kSignHi, sv = up ? kSignLo : 0ull;
        return ArDP::add(ArDP::make((u.x ^ su) & ku, (u.y ^ su) & ku),
                         ArDP::make((p2_swap(v.x) ^ sv) & kv, (p2_swap(v.y) ^ sv) & kv));
    }
    __device__ __forceinline__ static Scale scale_of(const StageArgs& p)
    {
        const float kh = (float)p.scale;
        return make_float2(kh, (float)(p.scale - (double)kh));
    }
    // the product is formed in double-float on the FP32 units (exact kh hi plus
    // first-order terms) before the join's single FP64 addition
    __device__ __forceinline__ static void parts(ArDP::C z, Scale k, double& re, double& im)
    {
        const u64 kh = p2_splat(k.x), kl = p2_splat(k.y);
        const u64 ph = p2_mul(z.x, kh);
        const u64 pl = p2_fma(z.y, kh, p2_fma(z.x, kl, p2_fma(z.x, kh, ph ^ kSignBoth)));
        float a, b, c, d;
        p2_unpack(ph, a, b);
        p2_unpack(pl, c, d);
        re = join_f64(a, c);
        im = join_f64(b, d);
    }
};

// Copies of rows [row0, row0 + rows) of `len` elements of BYTES bytes, packed in memory,
// to dst with `ld` elements between rows; a warp per row, in 16-byte pieces where
// every row starts on 16 bytes on both sides, else element by element (8-byte
// pieces of 4-byte elements where those are aligned).
template <int BYTES>
__device__ __forceinline__ void copy_rows(unsigned char* dst, int ld, const void* src, int64_t row0, int rows, int len,
                                          int tid, int T)
{
    const int lane = tid & 31;
    const unsigned at = (unsigned)reinterpret_cast<uintptr_t>(src) | (unsigned)(len * BYTES) | (unsigned)(ld * BYTES);
    for (int r = tid >> 5; r < rows; r += T >> 5) {
        const char* s = static_cast<const char*>(src) + (row0 + r) * (int64_t)len * BYTES;
        unsigned char* d = dst + (size_t)r * ld * BYTES;
        if (BYTES == 16 || (at & 15) == 0) {
            for (int i = lane * 16; i < len * BYTES; i += 512) cp_async<16>(d + i, s + i);
        } else if (BYTES == 8 || (at & 7) == 0) {
            for (int i = lane * 8; i < len * BYTES; i += 256) cp_async<8>(d + i, s + i);
        } else {
            for (int i = lane * 4; i < len * BYTES; i += 128)
                asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"((uint32_t)__cvta_generic_to_shared(d + i)), "l"(s + i)
                             : "memory");
        }
    }
    cp_async_commit();
}

// Elements between raw rows: 16-byte rows, and consecutive rows 16 bytes apart in
// the banks.
__host__ __device__ inline int raw_pitch(int len, int bytes)
{
    const int per = 16 / bytes;
    const int l = (len + per - 1) / per * per;
    return l + (per - l % (128 / bytes) + 128 / bytes) % (128 / bytes);
}

template <class A, int G>
__host__ __device__ inline size_t real_tile_bytes(int n)
{
    const int raw_r2c = raw_pitch(n, (int)sizeof(typename MixReal<A>::T)) * (int)sizeof(typename MixReal<A>::T);
    const int raw_c2r = raw_pitch(n / 2 + 1, (int)sizeof(typename A::C)) * (int)sizeof(typename A::C);
    const size_t raw = 2 * (size_t)G * (raw_r2c > raw_c2r ? raw_r2c : raw_c2r);
    return raw + (2 * (size_t)G * Mix<A, G>::pitch(n) + n) * sizeof(typename A::C);
}

// The passes of a tile whose inputs the first pass takes from `in`; returns the
// buffer with the result (every thread past the barrier).
template <class A, int G, class In, class AfterFirst>
__device__ __forceinline__ typename A::C* real_passes(const StageArgs& p, const MixPlan& plan, typename A::C* a,
                                                      typename A::C* b, const typename A::C* tw, bool mine, int at, int g,
                                                      int slot, int slots, In in, AfterFirst after_first)
{
    using M = Mix<A, G>;
    const TileGeom tg{};
    if (mine) M::template dispatch<true>(p, plan.pass[0], false, tg, a + at, a + at, tw, g, slot, slots, in);
    __syncthreads();
    after_first();
    for (int ps = 1; ps < plan.npass; ++ps) {
        if (mine) M::template dispatch<false>(p, plan.pass[ps], false, tg, a + at, b + at, tw, g, slot, slots);
        __syncthreads();
        typename A::C* t = a; a = b; b = t;
    }
    return a;
}

template <class A, int G, bool FWD>
__global__ void __launch_bounds__(kMixMaxThreads, mix_min_ctas())
real_mix_kernel(const StageArgs p, const __grid_constant__ MixPlan plan, int64_t ntiles)
{
    using M = Mix<A, G>;
    using C = typename A::C;
    using RP = MixReal<A>;
    using T = typename RP::T;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int n = p.n, nh = n / 2 + 1, ld = M::pitch(n);
    C* ba = reinterpret_cast<C*>(smem_raw);
    C* bb = ba + G * ld;
    unsigned char* raw = reinterpret_cast<unsigned char*>(bb + G * ld);
    const int ldr = FWD ? raw_pitch(n, (int)sizeof(T)) : raw_pitch(nh, (int)sizeof(C));
    C* tw = reinterpret_cast<C*>(raw + 2 * (size_t)G * ldr * (FWD ? sizeof(T) : sizeof(C)));
    const int tid = threadIdx.x, TH = blockDim.x;
    const int g = M::line_of(tid), slot = M::slot_of(tid), slots = plan.slots;
    const int64_t L = p.M1;
    auto rows = [&](int64_t t) { return (int)(L - t * 2 * G < 2 * G ? L - t * 2 * G : 2 * G); };
    auto copy_in = [&](int64_t t) {
        if constexpr (FWD) copy_rows<sizeof(T)>(raw, ldr, p.in, t * 2 * G, rows(t), n, tid, TH);
        else copy_rows<sizeof(C)>(raw, ldr, p.in, t * 2 * G, rows(t), nh, tid, TH);
    };
    grid_wait();
    for (int i = tid; i < n; i += TH) cp_async<M::E>(tw + i, reinterpret_cast<const C*>(p.tw) + i);
    copy_in(blockIdx.x);
    const typename RP::Scale ks = RP::scale_of(p);
    for (int64_t t = blockIdx.x; t < ntiles; t += gridDim.x) {
        const int64_t l0 = t * 2 * G, next = t + gridDim.x;
        const int nrow = rows(t);
        const bool mine = 2 * g < nrow, both = 2 * g + 1 < nrow;
        auto refill = [&]() { if (next < ntiles) copy_in(next); };
        cp_async_wait_all();
        __syncthreads();
        const C* z;
        if constexpr (FWD) {
            const T* x1 = reinterpret_cast<const T*>(raw) + 2 * g * ldr;
            const T* x2 = x1 + ldr;
            z = real_passes<A, G>(p, plan, ba, bb, tw, mine, g * ld, g, slot, slots,
                                  [&](int pos) { return RP::make(x1[pos], both ? x2[pos] : T(0)); }, refill);
            // separate the two spectra: frequencies 0..n/2 of the tile's real lines,
            // consecutive threads on consecutive lines
            const int o = tid % (2 * G);
            const C* zl = z + (o >> 1) * ld;
            if (o < nrow)
                for (int k = tid / (2 * G); k < nh; k += TH / (2 * G)) {
                    const C zk = zl[k], zr = A::conj(zl[k == 0 ? 0 : n - k]);
                    const C X = A::scale((o & 1) ? A::mul_mi(A::sub(zk, zr)) : A::add(zk, zr), 0.5);
                    Io<A>::store(p.out, p.out_fmt, (int64_t)k * p.Sk + (l0 + o) * p.S1, X);
                }
        } else {
            const C* v1 = reinterpret_cast<const C*>(raw) + 2 * g * ldr;
            const C* v2 = v1 + ldr;
            z = real_passes<A, G>(p, plan, ba, bb, tw, mine, g * ld, g, slot, slots,
                                  [&](int pos) {
                                      const bool up = pos < nh;
                                      const int k = up ? pos : n - pos;
                                      return RP::extend(v1[k], both ? v2[k] : A::zero(), up, k == 0 || 2 * k == n);
                                  },
                                  refill);
            // a warp per pair of real lines
            for (int r = tid >> 5; 2 * r < nrow; r += TH >> 5) {
                const C* zl = z + r * ld;
                T* y1 = reinterpret_cast<T*>(p.out) + (l0 + 2 * r) * n;
                const bool two = 2 * r + 1 < nrow;
#pragma unroll 4
                for (int i = tid & 31; i < n; i += 32) {
                    T re, im;
                    RP::parts(zl[i], ks, re, im);
                    y1[i] = re;
                    if (two) y1[n + i] = im;
                }
            }
        }
    }
    cp_async_wait_all();
}

}  // namespace ofg
