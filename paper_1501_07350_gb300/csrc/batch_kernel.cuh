// batch_kernel.cuh -- the persistent kernel of the batched form (batch.cu).
#pragma once
#include "../../include/openfft_gb.h"
#include "fft_mix.cuh"

namespace ofg {

constexpr int kBatchThreads = 128;
struct BatchCounters {
    unsigned long long next;   // queue head
    int status;                // OPENFFT_OK or OPENFFT_ERR_TIMEOUT
    int pad;
    // followed by done[3 * count]
};

struct BatchDev {
    const StageArgs* stages;       // [2 directions][3 stages][count]; aux: the length's MixPlan
    const int64_t* item_base;      // [3 * count + 1]: queue index of the first tile of (stage, transform)
    const unsigned* need;          // [3 * count]: tiles of (stage, transform)
    void* const* ptrs;             // [2 * count]: in_i, out_i (device pointers)
    void* const* scratch;          // [count]
    BatchCounters* ctr;
    unsigned* done;                // [3 * count]
    int count;
    int tiles_per_item;
    int dir_index;                 // 0 forward, 1 backward
    long long wait_budget;         // clock64 cycles
};

// Shared-memory layout of the batched kernel: [two tile buffers and the twiddle
// table, buf_bytes | queue prefix item_base (3 count + 1 int64) | tile counts need
// (3 count uint32)].
template <class A, int G>
__global__ void __launch_bounds__(kBatchThreads, 8)
batch_kernel(const BatchDev d, size_t buf_bytes)
{
    using C = typename A::C;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ __align__(8) StageArgs s_p;
    __shared__ __align__(8) MixPlan s_plan;
    __shared__ int64_t s_tile;        // first tile of the item
    __shared__ int s_q, s_abort;
    const int tid = threadIdx.x;
    const int nq = 3 * d.count;
    int64_t* sh_base = reinterpret_cast<int64_t*>(smem_raw + buf_bytes);
    unsigned* sh_need = reinterpret_cast<unsigned*>(sh_base + nq + 1);
    for (int k = tid; k <= nq; k += kBatchThreads) sh_base[k] = d.item_base[k];
    for (int k = tid; k < nq; k += kBatchThreads) sh_need[k] = d.need[k];
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
            s_tile = abort ? 0 : (j - sh_base[q]) * d.tiles_per_item;
        }
        __syncthreads();
        if (s_abort) break;
        const int q = s_q, s = q / d.count, i = q - s * d.count;
        // the item's stage descriptor and radix plan, its arrays
        const StageArgs* gp = &d.stages[d.dir_index * nq + q];
        const MixPlan* gplan = reinterpret_cast<const MixPlan*>(__ldg(reinterpret_cast<const unsigned long long*>(&gp->aux)));
        for (int k = tid; k < (int)(sizeof(StageArgs) / 4); k += kBatchThreads)
            reinterpret_cast<int*>(&s_p)[k] = __ldg(reinterpret_cast<const int*>(gp) + k);
        for (int k = tid; k < (int)(sizeof(MixPlan) / 4); k += kBatchThreads)
            reinterpret_cast<int*>(&s_plan)[k] = __ldg(reinterpret_cast<const int*>(gplan) + k);
        const void* in_i = d.ptrs[2 * i];
        void* out_i = d.ptrs[2 * i + 1];
        void* sc = d.scratch[i];
        __syncthreads();
        StageArgs p = s_p;
        p.in = s == 0 ? in_i : (s == 1 ? sc : out_i);
        p.out = s == 0 ? sc : out_i;
        const int64_t t0 = s_tile;
        const int64_t ntile = p.ngroups * (p.group_i2 ? p.M1 : p.M2);
        const int64_t t1 = t0 + d.tiles_per_item < ntile ? t0 + d.tiles_per_item : ntile;
        C* buf = reinterpret_cast<C*>(smem_raw);
        const int ld = Mix<A, G>::pitch(p.n);
        mix_run<A, G, false>(p, s_plan, t0, 1, t1, buf, buf + G * ld, buf + 2 * G * ld, ld, kBatchThreads / G, kBatchThreads, false);
        __threadfence();                           // release this thread's stores
        __syncthreads();
        if (tid == 0) atomicAdd(&d.done[q], 1u);
    }
}

// The batched kernel for tiles of G lines and the shared memory of its tiles of lines of
// up to n points, per arithmetic (batch_df.cu, batch_f32.cu); FP32 has G = 8 and 4,
// double-float 8, 4 and 2.
size_t batch_tile_bytes_df(int G, int n);
size_t batch_tile_bytes_f32(int G, int n);
const void* batch_kernel_df(int G);
const void* batch_kernel_f32(int G);

template <class A, int G>
size_t batch_tile_bytes(int n) { return (2 * (size_t)G * Mix<A, G>::pitch(n) + n) * sizeof(typename A::C); }

}  // namespace ofg
