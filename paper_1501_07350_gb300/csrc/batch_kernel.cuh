// batch_kernel.cuh -- the persistent kernel of the batched form (batch.cu).
#pragma once
#include "../../include/openfft_gb.h"
#include "fft_mix.cuh"

namespace ofg {

// Threads of a CTA whose items' tiles all 128 threads share, and of one (WIDE) that
// splits into groups of warps with a tile each.
constexpr int kBatchThreads = 128;
constexpr int kBatchWideThreads = 512;
constexpr int kBatchWideGroups = 4;            // at most
template <bool WIDE>
constexpr int batch_threads() { return WIDE ? kBatchWideThreads : kBatchThreads; }

struct BatchCounters {
    unsigned long long next;   // queue head
    int status;                // OPENFFT_OK or OPENFFT_ERR_TIMEOUT
    int pad;
    // followed by done[3 * count]
};

// One stage of one transform; args.aux: the length's MixPlan.
struct BatchStage {
    StageArgs args;
    int tiles_per_item;
    int groups;                // of the CTA's threads, each with tiles of its own
    int group_elems;           // elements between the groups' buffers
    int pad;
};

struct BatchDev {
    const BatchStage* stages;      // [2 directions][3 stages][count]
    const int64_t* item_base;      // [3 * count + 1]: queue index of the first item of (stage, transform)
    const unsigned* need;          // [3 * count]: items of (stage, transform)
    void* const* ptrs;             // [2 * count]: in_i, out_i (device pointers)
    void* const* scratch;          // [count]
    BatchCounters* ctr;
    unsigned* done;                // [3 * count]
    int count;
    int dir_index;                 // 0 forward, 1 backward
    long long wait_budget;         // clock64 cycles
};

// Shared-memory layout of the batched kernel: [two tile buffers and the twiddle
// table, of each group, buf_bytes | queue prefix item_base (3 count + 1 int64) | item
// counts need (3 count uint32)].
template <class A, bool WIDE>
__global__ void __launch_bounds__(batch_threads<WIDE>(), WIDE ? 1 : 8)
batch_kernel(const BatchDev d, size_t buf_bytes)
{
    using C = typename A::C;
    constexpr int T = batch_threads<WIDE>();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ __align__(8) BatchStage s_st;
    __shared__ __align__(8) MixPlan s_plan;
    __shared__ int64_t s_item;        // the item's index in its (stage, transform)
    __shared__ int s_q, s_abort;
    const int tid = threadIdx.x;
    const int nq = 3 * d.count;
    int64_t* sh_base = reinterpret_cast<int64_t*>(smem_raw + buf_bytes);
    unsigned* sh_need = reinterpret_cast<unsigned*>(sh_base + nq + 1);
    for (int k = tid; k <= nq; k += T) sh_base[k] = d.item_base[k];
    for (int k = tid; k < nq; k += T) sh_need[k] = d.need[k];
    __syncthreads();
    const int64_t total = sh_base[nq];
    volatile int* status = &d.ctr->status;
    int64_t mine = 0;                 // thread 0: the next item
    if (tid == 0) mine = (int64_t)atomicAdd(&d.ctr->next, 1ull);

    for (;;) {
        if (tid == 0) {
            const int64_t j = mine;
            int abort = *status != OPENFFT_OK || j >= total;
            int q = 0;
            if (!abort) {
                mine = (int64_t)atomicAdd(&d.ctr->next, 1ull);
                // (stage, transform) of item j: last q with item_base[q] <= j
                int lo = 0, hi = nq - 1;
                while (lo < hi) {
                    const int mid = (lo + hi + 1) >> 1;
                    if (sh_base[mid] <= j) lo = mid; else hi = mid - 1;
                }
                q = lo;
                const int s = q / d.count;
                if (s > 0) {
                    volatile unsigned* cnt = &d.done[q - d.count];
                    const unsigned want = sh_need[q - d.count];
                    const long long t0 = clock64();
                    while (*cnt < want) {
                        if (*status != OPENFFT_OK) { abort = 1; break; }
                        if (clock64() - t0 > d.wait_budget) {
                            atomicCAS(&d.ctr->status, OPENFFT_OK, OPENFFT_ERR_TIMEOUT);
                            abort = 1;
                            break;
                        }
                        __nanosleep(128);
                    }
                    __threadfence();               // acquire: order the loads after the counter
                }
            }
            s_abort = abort;
            s_q = q;
            s_item = abort ? 0 : j - sh_base[q];
        }
        __syncthreads();
        if (s_abort) break;
        const int q = s_q, s = q / d.count, i = q - s * d.count;
        // the item's stage descriptor and radix plan, its arrays
        const BatchStage* gp = &d.stages[d.dir_index * nq + q];
        const MixPlan* gplan = reinterpret_cast<const MixPlan*>(__ldg(reinterpret_cast<const unsigned long long*>(&gp->args.aux)));
        for (int k = tid; k < (int)(sizeof(BatchStage) / 4); k += T)
            reinterpret_cast<int*>(&s_st)[k] = __ldg(reinterpret_cast<const int*>(gp) + k);
        for (int k = tid; k < (int)(sizeof(MixPlan) / 4); k += T)
            reinterpret_cast<int*>(&s_plan)[k] = __ldg(reinterpret_cast<const int*>(gplan) + k);
        const void* in_i = d.ptrs[2 * i];
        void* out_i = d.ptrs[2 * i + 1];
        void* sc = d.scratch[i];
        __syncthreads();
        C* buf = reinterpret_cast<C*>(smem_raw);
        StageArgs p = s_st.args;
        p.in = s == 0 ? in_i : (s == 1 ? sc : out_i);
        p.out = s == 0 ? sc : out_i;
        const int64_t ntile = p.ngroups * (p.group_i2 ? p.M1 : p.M2);
        const int64_t t0 = s_item * s_st.tiles_per_item;
        const int64_t t1 = t0 + s_st.tiles_per_item < ntile ? t0 + s_st.tiles_per_item : ntile;
        if constexpr (!WIDE) {
            constexpr int G = 8;
            const int ld = Mix<A, G>::pitch(p.n);
            mix_run<A, G, false>(p, s_plan, t0, 1, t1, buf, buf + G * ld, buf + 2 * G * ld, ld, T / G, tid, T, false, CtaSync());
        } else {
            // group grp of the CTA's threads takes tiles t0 + grp, t0 + grp + groups, ...
            const int groups = s_st.groups, threads = T / groups, grp = tid / threads;
            const int w = p.G, ld = Mix<A, 0>::pitch(p.n, w);
            C* b = buf + grp * s_st.group_elems;
            if (t0 + grp < t1)
                mix_run<A, 0, false>(p, s_plan, t0 + grp, groups, t1, b, b + w * ld, b + 2 * w * ld, ld, threads / w,
                                     tid - grp * threads, threads, false, GroupSync{1 + grp, threads});
        }
        __threadfence();                           // release this thread's stores
        __syncthreads();
        if (tid == 0) atomicAdd(&d.done[q], 1u);
    }
}

// Bytes of a group's tiles of G = 8, 4, 2 or 1 lines of n points with the twiddle table,
// and the kernels, per arithmetic (batch_df.cu, batch_f32.cu).
size_t batch_tile_bytes_df(int G, int n);
size_t batch_tile_bytes_f32(int G, int n);
const void* batch_kernel_df(bool wide);
const void* batch_kernel_f32(bool wide);

template <class A>
size_t batch_tile_bytes(int G, int n)
{
    return ((2 * (size_t)G * Mix<A, 0>::pitch(n, G) + n) * sizeof(typename A::C) + 15) & ~(size_t)15;
}

}  // namespace ofg
