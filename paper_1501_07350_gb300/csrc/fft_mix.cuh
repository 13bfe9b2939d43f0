// fft_mix.cuh -- FFT stage kernel for the line lengths that have no kernel
// compiled for them alone: any n with factors 2, 3, 5 and 7, in the packed double-float
// and the FP32 arithmetic.  The passes take every n <= 2048 (the batched form runs them
// all); as a stage of its own it goes as far as the plan's tile width, which comes from
// the generic kernel's two tiles of n (G + 1) elements in 200 KB: 8 lines in FP32 up to
// 1422 points, 4 in double-float up to 1280, and as many lines side by side in the output
// (five, three).  Longer lines and fewer of them run on the generic stage.
//
// A CTA takes tiles of G lines.  The radix plan is chosen on the host per length
// (mix_radix_plan): few passes of large radices (composite ones up to 10 in
// double-float, 16 in FP32, whose coprime factors need no twiddles between
// them), each pass compiled per radix, strides and counts at run time.
//
// Tile layout in shared memory: line after line, padded so that consecutive lines
// start one or two elements apart in the banks, and the lanes of a warp take
// consecutive lines at one position (two consecutive positions, where G lines do
// not fill the banks): every pass reads and writes without conflicts whatever the
// radix and the length, a twiddle is one broadcast load for the G lines (from the CTA's own
// copy of the length's table), the copies in run along the lines, and the last pass's
// results leave for global memory straight from registers, G consecutive elements per
// frequency (the transposed store).  FP32 lines of contiguous output have their last
// pass run along the line instead (fft_mix_launch.cuh).
//
// Passes alternate between two tile buffers, one barrier each (in place, with a barrier
// between a pass's reads and writes, the radix cases spilled).  The last pass reads
// one buffer and writes global memory, so the next tile's copies (cp.async) go into
// the other buffer while it runs.
//
// Registers: 64 a thread everywhere (the bound of 512-thread CTAs).  The double-float
// instances spill 44 bytes of stores and 96 of loads there, the real ones up to 216 and
// 212, the batched one 184 and 164; FP32 ones none.  The 512-thread batched kernel has
// 128 registers and no spills.
//
// In double-float the instructions bound it (6.5-8.5 a point and stage, 47-55 % of issue
// slots) with the barriers between passes; FP32 runs at 75-85 % of the copy bandwidth on
// large arrays.  Against the kernels before it (compile-time mixed radices, generic), us:
// 240x288x320 complex128 1317 -> 774, complex64 452 -> 193; 120x144x160 complex128 137 ->
// 99; 180x200x225 complex64 183 -> 81; 98x343x105 complex128 330 -> 172.
#pragma once
#include <type_traits>

#include "arith.cuh"
#include "arith_pair.cuh"
#include "fft_stage.h"
#include "fft_tile.cuh"
#include "stage_io.cuh"

namespace ofg {

constexpr int kMixMaxPasses = 11;

struct MixPass {
    int radix;
    int nbf;                    // butterflies of one line: n / radix
    int m;                      // product of the earlier radices
    int s;                      // nbf / m: twiddle exponent step
    uint32_t inv;               // ceil(2^20 / m): b / m = (b inv) >> 20 for b m < 2^20
};
struct MixPlan {
    int npass;
    int slots;                  // threads per line of a tile
    MixPass pass[kMixMaxPasses];
};

// threads per CTA at most, and the CTAs of that size the registers are sized for
constexpr int kMixMaxThreads = 512;
constexpr int mix_min_ctas() { return 2; }

// entry e of the tile's copy of the twiddle table
__device__ __forceinline__ ArF32::W mix_twiddle(const ArF32::C* tw, int e) { return tw[e]; }
__device__ __forceinline__ ArDP::W mix_twiddle(const ArDP::C* tw, int e)
{
    return ArDP::make_w(reinterpret_cast<const float4*>(tw)[e]);
}

// a complex128 element that was copied as the bits of a double-float one
__device__ __forceinline__ ArDP::C c128_bits(ArDP::C x)
{
    return Io<ArDP>::from_c128(make_double2(__longlong_as_double((long long)x.x), __longlong_as_double((long long)x.y)));
}

// Tiles of G lines (G = 0: a width w that is given at run time).
template <class A, int G>
struct Mix {
    using C = typename A::C;
    static constexpr int E = sizeof(C);
    // lanes of a warp: lines fastest, or (line, slot parity) with the parity fastest
    __host__ __device__ static constexpr bool pairs(int w) { return E * w != 128 || E == 8; }
    static constexpr int kUnits = 128 / E;                    // elements of one shared-memory wavefront

    __host__ __device__ static int pitch(int n, int w = G)
    {
        if (!pairs(w)) return n | 1;
        return n + (2 - n % kUnits + kUnits) % kUnits;
    }
    __device__ __forceinline__ static int line_of(int tid, int w = G) { return pairs(w) ? (tid >> 1) % w : tid % w; }
    __device__ __forceinline__ static int slot_of(int tid, int w = G)
    {
        return pairs(w) ? (tid & 1) + 2 * (tid / (2 * w)) : tid / w;
    }

    // Copies of a tile: `valid` lines, lstride apart from line0 on, a warp per line
    // in 16-byte pieces (8 bytes where an odd length or the array's address leaves
    // lines of complex64 unaligned).
    __device__ __forceinline__ static void issue_load(const StageArgs& p, int64_t line0, int64_t lstride, int valid, C* buf,
                                                      int ld, int tid, int T)
    {
        const int n = p.n, lane = tid & 31;
        const bool wide = ((n & 1) | (int)(reinterpret_cast<uintptr_t>(p.in) & 15)) == 0;
        for (int g = tid >> 5; g < valid; g += T >> 5) {
            const int64_t e = (line0 + g * lstride) * n;
            const char* src = reinterpret_cast<const char*>(p.in) + e * E;
            C* dst = buf + g * ld;
            if (E == 16 || !wide) {
#pragma unroll 4
                for (int i = lane; i < n; i += 32)
                    if (in_bounds(p.chk, e + i, p.in_elems)) cp_async<E>(dst + i, src + i * E);
            } else {
#pragma unroll 4
                for (int i = 2 * lane; i < n; i += 64)
                    if (in_bounds(p.chk, e + i, p.in_elems) && in_bounds(p.chk, e + i + 1, p.in_elems))
                        cp_async<16>(dst + i, src + i * E);
            }
        }
        cp_async_commit();
    }

    template <bool CONJ_SCALE, bool EXT, int R>
    __device__ __forceinline__ static void store(const StageArgs& p, int64_t o, int64_t step, const C* v)
    {
        constexpr int EB = EXT ? Io<A>::kExtBytes : Io<A>::kMidBytes;
        char* ptr = reinterpret_cast<char*>(p.out) + o * EB;
#pragma unroll
        for (int q = 0; q < R; ++q) {
            if (in_bounds(p.chk, o + q * step, p.out_elems)) put<A, CONJ_SCALE, EXT>(ptr, v[q], p);
            ptr += step * EB;
        }
    }

    // One pass from buffer src to buffer dst, or, the last one, to global memory.
    // The first pass takes its inputs from in(position) unless In is FromTile.
    struct FromTile {
        __device__ __forceinline__ C operator()(int) const { return A::zero(); }
    };
    template <int R, bool FIRST, class In>
    __device__ __forceinline__ static void pass(const StageArgs& p, const MixPass& ps, bool last, const TileGeom& tg,
                                                const C* src, C* dst, const C* tw, int g, int slot, int slots, In in)
    {
        constexpr bool kFromTile = std::is_same<In, FromTile>::value;
        // src, dst: this thread's line
        const int nbf = ps.nbf;
        for (int b = slot; b < nbf; b += slots) {
            C v[R];
            const C* x = src + b;
#pragma unroll
            for (int j = 0; j < R; ++j) {
                if constexpr (kFromTile || !FIRST) v[j] = x[j * nbf];
                else v[j] = in(b + j * nbf);
            }
            int pos = b * R;                               // of the first result: t m R + k, b = t m + k
            if constexpr (FIRST && kFromTile) {
                if constexpr (Io<A>::kConverts) {
                    if (p.in_fmt == FMT_C128) {
#pragma unroll
                        for (int j = 0; j < R; ++j) v[j] = c128_bits(v[j]);
                    }
                }
                if (p.conj_in) {
#pragma unroll
                    for (int j = 0; j < R; ++j) v[j] = A::conj(v[j]);
                }
            } else if constexpr (!FIRST) {
                const int t = (int)(((uint32_t)b * ps.inv) >> 20), k = b - t * ps.m;
                pos = t * ps.m * R + k;
                const int ks = k * ps.s;
#pragma unroll
                for (int j = 1; j < R; ++j) v[j] = A::mul(v[j], mix_twiddle(tw, j * ks));
            }
            Dft<A, R>::run(v);
            if (!last) {
                C* y = dst + pos;
#pragma unroll
                for (int q = 0; q < R; ++q) y[q * ps.m] = v[q];
            } else {
                const int64_t o = tg.obase + g * tg.ostride + b * p.Sk, step = ps.m * p.Sk;
                const bool ext = p.out_fmt != FMT_DF;
                if (p.conj_out) {
                    if (ext) store<true, true, R>(p, o, step, v);
                    else store<true, false, R>(p, o, step, v);
                } else {
                    if (ext) store<false, true, R>(p, o, step, v);
                    else store<false, false, R>(p, o, step, v);
                }
            }
        }
    }

    template <bool FIRST, class In = FromTile>
    __device__ __forceinline__ static void dispatch(const StageArgs& p, const MixPass& ps, bool last, const TileGeom& tg,
                                                    const C* src, C* dst, const C* tw, int g, int slot, int slots,
                                                    In in = In())
    {
        switch (ps.radix) {
        case 1:
            if constexpr (FIRST) pass<1, FIRST>(p, ps, last, tg, src, dst, tw, g, slot, slots, in);     // lines of one point
            break;
        case 2: pass<2, FIRST>(p, ps, last, tg, src, dst, tw, g, slot, slots, in); break;
        case 3: pass<3, FIRST>(p, ps, last, tg, src, dst, tw, g, slot, slots, in); break;
        case 4: pass<4, FIRST>(p, ps, last, tg, src, dst, tw, g, slot, slots, in); break;
        case 5: pass<5, FIRST>(p, ps, last, tg, src, dst, tw, g, slot, slots, in); break;
        case 6: pass<6, FIRST>(p, ps, last, tg, src, dst, tw, g, slot, slots, in); break;
        case 7: pass<7, FIRST>(p, ps, last, tg, src, dst, tw, g, slot, slots, in); break;
        case 8: pass<8, FIRST>(p, ps, last, tg, src, dst, tw, g, slot, slots, in); break;
        case 10: pass<10, FIRST>(p, ps, last, tg, src, dst, tw, g, slot, slots, in); break;
        default:
            if constexpr (E == 8) {
                switch (ps.radix) {
                case 9: pass<9, FIRST>(p, ps, last, tg, src, dst, tw, g, slot, slots, in); break;
                case 12: pass<12, FIRST>(p, ps, last, tg, src, dst, tw, g, slot, slots, in); break;
                case 15: pass<15, FIRST>(p, ps, last, tg, src, dst, tw, g, slot, slots, in); break;
                default: pass<16, FIRST>(p, ps, last, tg, src, dst, tw, g, slot, slots, in); break;
                }
            }
            break;
        }
    }
};

// Barrier of the threads that run a tile: the CTA's, or that of a group of its warps.
struct CtaSync {
    __device__ __forceinline__ void operator()() const { __syncthreads(); }
};
struct GroupSync {
    int id, threads;
    __device__ __forceinline__ void operator()() const
    {
        asm volatile("barrier.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
    }
};

// Tiles tile, tile + step, ... below end of a stage, by T threads (tid among them) that
// `sync` synchronises.  cur and oth: two tile buffers of G ld elements; tw: n elements
// for the length's twiddle table, copied in here.  rows: the last pass, whose lines go
// out as they are, takes consecutive threads along a line.  Returns with the threads
// still reading the buffers.
template <class A, int G, bool REPEAT, class Sync>
__device__ __forceinline__ void mix_run(const StageArgs& p, const MixPlan& plan, int64_t tile, int64_t step, int64_t end,
                                        typename A::C* cur, typename A::C* oth, typename A::C* tw, int ld, int slots, int tid,
                                        int T, bool rows, Sync sync)
{
    using M = Mix<A, G>;
    using C = typename A::C;
    const int w = G ? G : p.G;
    const int g = M::line_of(tid, w), slot = M::slot_of(tid, w), at = g * ld;
    const int gl = rows ? tid / slots : g, sl = rows ? tid - gl * slots : slot, al = gl * ld;      // of the last pass
    TileGeom tg = tile_geom<REPEAT>(p, tile, w);
    for (int i = tid; i < p.n; i += T) cp_async<M::E>(tw + i, reinterpret_cast<const C*>(p.tw) + i);
    M::issue_load(p, tg.line0, tg.lstride, tg.valid, cur, ld, tid, T);
    for (; tile < end; tile += step) {
        const int64_t next = tile + step;
        const TileGeom tn = tile_geom<REPEAT>(p, next < end ? next : tile, w);
        const bool mine = g < tg.valid;
        cp_async_wait_all();
        sync();
        const int np = plan.npass;
        if (np > 1) {
            if (mine) M::template dispatch<true>(p, plan.pass[0], false, tg, cur + at, oth + at, tw, g, slot, slots);
            sync();
            for (int ps = 1; ps < np - 1; ++ps) {
                C* t = cur; cur = oth; oth = t;
                if (mine) M::template dispatch<false>(p, plan.pass[ps], false, tg, cur + at, oth + at, tw, g, slot, slots);
                sync();
            }
            // every thread has read `cur`: it takes the next tile while the last pass runs
            if (next < end) M::issue_load(p, tn.line0, tn.lstride, tn.valid, cur, ld, tid, T);
            if (gl < tg.valid) M::template dispatch<false>(p, plan.pass[np - 1], true, tg, oth + al, cur + al, tw, gl, sl, slots);
        } else {
            if (next < end) M::issue_load(p, tn.line0, tn.lstride, tn.valid, oth, ld, tid, T);
            if (gl < tg.valid) M::template dispatch<true>(p, plan.pass[0], true, tg, cur + al, oth + al, tw, gl, sl, slots);
            C* t = cur; cur = oth; oth = t;
        }
        tg = tn;
    }
    cp_async_wait_all();
}

template <class A, int G, bool REPEAT>
__global__ void __launch_bounds__(kMixMaxThreads, mix_min_ctas())
fft_mix_kernel(const StageArgs p, const __grid_constant__ MixPlan plan, int64_t ntiles, bool rows)
{
    using C = typename A::C;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int ld = Mix<A, G>::pitch(p.n);
    C* buf = reinterpret_cast<C*>(smem_raw);
    grid_wait();
    // the grid has at most ntiles CTAs
    mix_run<A, G, REPEAT>(p, plan, blockIdx.x, gridDim.x, ntiles, buf, buf + G * ld, buf + 2 * G * ld, ld, plan.slots,
                          threadIdx.x, blockDim.x, sizeof(C) == 8 && rows, CtaSync());
}

// The radix plan of length n for a policy of 16-byte (double-float) or 8-byte (FP32)
// elements; npass = 0 if there is none.  pass[].radix etc. as the kernels read them.
MixPlan mix_radix_plan(int n, bool df);

}  // namespace ofg
