// batch.cu -- many 3-D transforms of uneven sizes in one persistent launch,
// replayed from a captured CUDA graph.
//
// Work items are runs of tiles (of G lines each) of one stage of
// one transform, handed out in stage-major order (every stage-1 tile of every transform, then every
// stage-2 tile, then every stage-3 tile) through one atomic queue head.  A
// stage-s item of transform i first waits until all stage-(s-1) tiles of
// transform i are done (a per-(stage, transform) counter).  Those items have
// lower queue indices, so they were handed to CTAs that were already running
// and that never wait on anything later: the waits always end.  Each wait is
// still bounded (clock64 budget); on expiry the kernel records
// OPENFFT_ERR_TIMEOUT in a status word, every CTA stops taking items, and the
// host reads the status at openfft_sync.
//
// Per item the CTA runs the any-length stage computation (fft_mix.cuh) with the
// length's radix plan.  Data written by one CTA and read by another in a later stage
// is loaded with cp.async after an acquire on the counter (a device-scope fence, which
// also covers the copies that go through L1); writers fence before releasing.
//
// The time is the tiles': small CTAs (128 threads, up to 8 per SM) keep copies, passes
// and stores of different items in flight.  64 uneven complex64 transforms (48^3 to
// 100x108x120) take 461 us, 797 with 256-thread CTAs and the specialised tile bodies
// (272 would be three reads and writes at the measured copy rate); the same in
// double-float 1534, 3253 before.
//
// A batch with a long axis (over 564 points in FP32, 282 in double-float), or with so many
// transforms that the queue tables fill the shared memory, holds one or two such CTAs on
// an SM.  It runs on one CTA of 512 threads instead, where each stage has its own tile
// width and the CTA's threads split into groups with a tile each, so that the short
// axes beside a long one keep wide tiles and all of the threads.  One 2048x48x48 beside 63 48^3:
// complex64 321 us (with 128-thread CTAs and one width for all stages 1282; generic body of
// 256 threads, which it replaced, 705), complex128 567 (4279, 1882); 40 60^3 beside four
// 1200x200x40 851 and 2393 (1904 and 7491); 4000 8^3 2099 and 2143 (2323 and 4273).  With
// 64 registers and two CTAs an SM instead of 128 and one, complex128 took 1.2 to 2.1
// times as long (spills), with 256 threads and three CTAs 1.1 to 2.5 times.
//
// A CTA claims its next
// item before it starts on the current one, so the queue's atomic and the search are
// not waited for.  A claimed item may stay behind one that waits for earlier items;
// waits still end: the unfinished item with the lowest index is never behind another,
// and everything it waits for has lower indices.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstring>
#include <vector>

#include "../../include/openfft_gb.h"
#include "batch.h"
#include "fft_stage.h"
#include "batch_kernel.cuh"
#include "fft_mix_launch.cuh"

namespace ofg {

// Tiles of one (stage, transform) per work item: enough that an item's queue and
// descriptor work is small beside them, few enough that a stage of the batch is about
// kItemsPerCta items for every CTA: eight 128^3 complex64 transforms take 182 us (245
// with 16 tiles an item), 64 uneven ones 461 (472 with four items per CTA, 495 six).
constexpr int kMaxTilesPerItem = 16;
constexpr int kItemsPerCta = 2;
// Shared memory of a CTA at most: tile buffers and queue tables.
constexpr size_t kMaxBatchSmem = 201 * 1024;

// --------------------------------------------------------------- host ----

namespace {

size_t tile_bytes_of(bool f32, int G, int n) { return f32 ? batch_tile_bytes_f32(G, n) : batch_tile_bytes_df(G, n); }
const void* kernel_of(bool f32, bool wide) { return f32 ? batch_kernel_f32(wide) : batch_kernel_df(wide); }
int threads_of(bool wide) { return wide ? kBatchWideThreads : kBatchThreads; }

// Tile width of a stage of lines of n points, Mg of them side by side in the output: at
// most 8 lines, no more than there are, and what `budget` bytes of shared memory hold.
int tile_width(bool f32, int n, int64_t Mg, size_t budget)
{
    int G = 8;
    while (G > 1 && (G / 2 >= Mg || tile_bytes_of(f32, G, n) > budget)) G /= 2;
    return G;
}

int64_t grouped_lines(const StageArgs& a) { return a.group_i2 ? a.M2 : a.M1; }
int64_t tiles_of(const StageArgs& a) { return a.ngroups * (a.group_i2 ? a.M1 : a.M2); }

}  // namespace

struct BatchPlan {
    int count = 0, dtype = 0, arith = 0;
    bool wide = false;                         // the kernel of 512-thread CTAs
    std::vector<int> dims;                     // 3 * count
    std::vector<int64_t> N;                    // per transform
    size_t smem = 0;
    int grid = 0;
    // device memory
    BatchStage* d_stages = nullptr;            // and the radix plans after them
    int64_t* d_item_base = nullptr;
    unsigned* d_need = nullptr;
    void** d_ptrs = nullptr;
    void** d_scratch = nullptr;
    unsigned char* d_ctr = nullptr;            // BatchCounters + done[3*count]
    size_t ctr_bytes = 0;
    std::vector<void*> scratch;
    std::vector<void*> twiddles;
    // host staging of the pointer table (page-locked, read by the graph's copy node)
    void** h_ptrs = nullptr;
    std::vector<void*> cur_ptrs;
    // graph
    cudaStream_t own = nullptr;
    cudaEvent_t ev_in = nullptr, ev_out = nullptr;
    cudaGraphExec_t exec[2] = {nullptr, nullptr};
    long long wait_budget = 2000000000LL;      // about one second of clock64 cycles
    unsigned need_extra = 0;                   // test hook: extra tiles the first wait expects
    int64_t items_per_stage[3] = {0, 0, 0};
};

static void free_batch(BatchPlan* b)
{
    if (!b) return;
    for (auto& e : b->exec) if (e) cudaGraphExecDestroy(e);
    if (b->own) cudaStreamDestroy(b->own);
    if (b->ev_in) cudaEventDestroy(b->ev_in);
    if (b->ev_out) cudaEventDestroy(b->ev_out);
    cudaFree(b->d_stages); cudaFree(b->d_item_base); cudaFree(b->d_need);
    cudaFree(b->d_ptrs); cudaFree(b->d_scratch); cudaFree(b->d_ctr);
    for (void* p : b->scratch) cudaFree(p);
    for (void* p : b->twiddles) cudaFree(p);
    if (b->h_ptrs) cudaFreeHost(b->h_ptrs);
    delete b;
}

void batch_destroy(BatchPlan* b) { free_batch(b); }

int batch_create(int count, const int* dims, const int* P, int dtype, int sms, BatchPlan** out,
                 int (*fail)(int, const char*))
{
    if (count < 1 || !dims || !P) return fail(OPENFFT_ERR_INVALID_ARG, "count >= 1 and non-null arrays required");
    if (dtype != OPENFFT_C2C_F64 && dtype != OPENFFT_C2C_F32) return fail(OPENFFT_ERR_UNSUPPORTED, "batched plans take F64 or F32");
    BatchPlan* b = new BatchPlan();
    b->count = count;
    b->dtype = dtype;
    b->arith = dtype == OPENFFT_C2C_F32 ? ARITH_F32 : ARITH_DF;
    b->dims.assign(dims, dims + 3 * count);
    const int E = dtype == OPENFFT_C2C_F32 ? 8 : 16;
    const int ext = dtype == OPENFFT_C2C_F32 ? FMT_C64 : FMT_C128;
    const int mid = dtype == OPENFFT_C2C_F32 ? FMT_C64 : FMT_DF;
    const int twf = dtype == OPENFFT_C2C_F32 ? FMT_C64 : FMT_DF;
    std::vector<BatchStage> st((size_t)2 * 3 * count);
    cudaError_t e;
    const bool f32 = dtype == OPENFFT_C2C_F32;
    // twiddle table and radix plan per distinct length
    std::vector<int> lens;
    std::vector<MixPlan> plans;
    auto tables_for = [&](int n, StageArgs& a) -> int {
        size_t k = 0;
        while (k < lens.size() && lens[k] != n) ++k;
        if (k == lens.size()) {
            const MixPlan pl = n <= kMaxLen ? mix_radix_plan(n, !f32) : MixPlan{};
            if (pl.npass == 0) return fail(OPENFFT_ERR_UNSUPPORTED_RADIX, "axis length must factor into 2, 3, 5, 7 and be <= 2048");
            void* t = nullptr;
            if (dev_malloc((void**)&t, twiddle_bytes(n, twf))) { cudaGetLastError(); return fail(OPENFFT_ERR_NOMEM, "twiddle tables"); }
            b->twiddles.push_back(t);
            if (launch_twiddles(n, twf, t, nullptr)) { cudaGetLastError(); return fail(OPENFFT_ERR_NOMEM, "twiddle tables"); }
            lens.push_back(n);
            plans.push_back(pl);
        }
        a.tw = b->twiddles[k];
        a.aux = reinterpret_cast<const void*>(k);        // its plan's index until the table has an address
        return OPENFFT_OK;
    };
    for (int i = 0; i < count; ++i) {
        const int64_t Na = dims[3 * i], Nb = dims[3 * i + 1], Nc = dims[3 * i + 2];
        if (Na < 1 || Nb < 1 || Nc < 1 || P[i] < 1) { free_batch(b); return fail(OPENFFT_ERR_INVALID_ARG, "sizes and P must be >= 1"); }
        if (P[i] > Na * Nb || P[i] > Nc * Na || P[i] > Nc * Nb) { free_batch(b); return fail(OPENFFT_ERR_P_TOO_LARGE, "P exceeds N1*N2 of an ordering (Eq. 2 undefined)"); }
        const int64_t N = Na * Nb * Nc;
        b->N.push_back(N);
        void* sc = nullptr;
        if (dev_malloc((void**)&sc, (size_t)N * E)) { cudaGetLastError(); free_batch(b); return fail(OPENFFT_ERR_NOMEM, "batched workspace"); }
        b->scratch.push_back(sc);
        // forward / backward stage geometry, as in the fused single-transform path
        struct Geo { int64_t n, M1, M2, S1, S2, Sk; int g2, contig, in_fmt, out_fmt, cin, cout; double scale; };
        const double invN = 1.0 / (double)N;
        const Geo geo[2][3] = {
            {{Nc, Na * Nb, 1, 1, 0, Na * Nb, 0, 0, ext, mid, 0, 0, 1.0},
             {Nb, Na, Nc, 1, Nb * Na, Na, 0, 0, mid, mid, 0, 0, 1.0},
             {Na, Nc * Nb, 1, Na, 0, 1, 0, 1, mid, ext, 0, 0, 1.0}},
            {{Na, Nb, Nc, 1, Na * Nb, Nb, 0, 0, ext, mid, 1, 0, 1.0},
             {Nb, Na, Nc, Nb * Nc, 1, Nc, 1, 0, mid, mid, 0, 0, 1.0},
             {Nc, Na * Nb, 1, Nc, 0, 1, 0, 1, mid, ext, 0, 1, invN}}};
        for (int dir = 0; dir < 2; ++dir)
            for (int s = 0; s < 3; ++s) {
                const Geo& g = geo[dir][s];
                BatchStage& bs = st[(size_t)dir * 3 * count + (size_t)s * count + i];
                std::memset(&bs, 0, sizeof(bs));
                StageArgs& a = bs.args;
                const int n = (int)g.n;
                if (const int status = tables_for(n, a)) { free_batch(b); return status; }
                a.M1 = g.M1; a.M2 = g.M2; a.S1 = g.S1; a.S2 = g.S2; a.Sk = g.Sk;
                a.scale = g.scale;
                split_scale(a);
                a.n = n;
                a.group_i2 = g.g2; a.contig_store = g.contig;
                a.conj_in = g.cin; a.conj_out = g.cout; a.do_fft = 1;
                a.in_fmt = g.in_fmt; a.out_fmt = g.out_fmt;
                a.in_elems = a.out_elems = N;          // read by the checked build
                a.chk = fallback_status_word();
            }
    }
    // Kernel and tile widths.  CTAs of 128 threads and tiles of 8 lines for every stage, while
    // an SM holds three CTAs with such tiles of the longest axis (and the queue tables).
    // Otherwise one CTA of 512 threads an SM, whose shared memory every stage has to
    // itself: the width is the most that fits, and the threads split into groups with a
    // tile each, as many as fit beside each other.
    const size_t tables = sizeof(int64_t) * (size_t)(3 * count + 1) + sizeof(unsigned) * (size_t)(3 * count);
    int nmax = 1;
    for (int v : b->dims) nmax = std::max(nmax, v);
    b->wide = tile_bytes_of(f32, 8, nmax) + tables > 75 * 1024;
    const size_t budget = tables < kMaxBatchSmem ? kMaxBatchSmem - tables : 0;
    for (BatchStage& bs : st) {
        StageArgs& a = bs.args;
        a.G = b->wide ? tile_width(f32, a.n, grouped_lines(a), budget) : 8;
        a.ngroups = (grouped_lines(a) + a.G - 1) / a.G;
        const size_t bytes = tile_bytes_of(f32, a.G, a.n);
        bs.groups = 1;
        while (b->wide && bs.groups < kBatchWideGroups && 2 * bs.groups * bytes <= budget) bs.groups *= 2;
        bs.group_elems = (int)(bytes / E);
        b->smem = std::max(b->smem, bs.groups * bytes);
    }
    b->ctr_bytes = sizeof(BatchCounters) + sizeof(unsigned) * (size_t)3 * count;
    const size_t stage_bytes = st.size() * sizeof(BatchStage), plan_bytes = plans.size() * sizeof(MixPlan);
    if (dev_malloc((void**)&b->d_stages, stage_bytes + plan_bytes) ||
        dev_malloc((void**)&b->d_item_base, sizeof(int64_t) * (size_t)(2 * (3 * count + 1))) ||
        dev_malloc((void**)&b->d_need, sizeof(unsigned) * (size_t)(2 * 3 * count)) ||
        dev_malloc((void**)&b->d_ptrs, sizeof(void*) * (size_t)(2 * count)) ||
        dev_malloc((void**)&b->d_scratch, sizeof(void*) * (size_t)count) ||
        dev_malloc((void**)&b->d_ctr, b->ctr_bytes) ||
        cudaMallocHost(&b->h_ptrs, sizeof(void*) * (size_t)(2 * count))) {
        cudaGetLastError();
        free_batch(b);
        return fail(OPENFFT_ERR_NOMEM, "batched plan tables");
    }
    // launch shape: persistent, as many CTAs as fit (tile buffer + queue tables)
    if (b->smem + tables > kMaxBatchSmem) { free_batch(b); return fail(OPENFFT_ERR_UNSUPPORTED, "batch too large for the queue tables in shared memory"); }
    // The kernel's shared-memory limit is the same for every plan: plans of other sizes share
    // the kernel, and this one's launches are captured at its first calls.
    int per_sm = 1;
    e = prepare_kernel(kernel_of(f32, b->wide), nullptr, (int)kMaxBatchSmem);
    if (!e) e = resident_ctas_per_sm(kernel_of(f32, b->wide), threads_of(b->wide), b->smem + tables, &per_sm);
    if (e) { free_batch(b); return fail(OPENFFT_ERR_CUDA, cudaGetErrorString(e)); }
    b->grid = sms * (per_sm > 0 ? per_sm : 1);
    {
        int64_t rounds = 0;                      // of one direction's three stages: a tile for each group
        for (int q = 0; q < 3 * count; ++q) rounds += (tiles_of(st[q].args) + st[q].groups - 1) / st[q].groups;
        const int64_t per = rounds / 3 / ((int64_t)b->grid * kItemsPerCta);
        for (BatchStage& bs : st)
            bs.tiles_per_item = bs.groups * (int)(per < 1 ? 1 : (per > kMaxTilesPerItem ? kMaxTilesPerItem : per));
    }
    // per direction (the two traverse the axes in opposite orders): tiles per
    // (stage, transform) and the stage-major queue prefix
    std::vector<int64_t> bases((size_t)2 * (3 * count + 1));
    std::vector<unsigned> needs((size_t)2 * 3 * count);
    for (int dir = 0; dir < 2; ++dir) {
        int64_t acc = 0;
        for (int q = 0; q < 3 * count; ++q) {
            const BatchStage& bs = st[(size_t)dir * 3 * count + q];
            const int64_t items = (tiles_of(bs.args) + bs.tiles_per_item - 1) / bs.tiles_per_item;
            bases[(size_t)dir * (3 * count + 1) + q] = acc;
            needs[(size_t)dir * 3 * count + q] = (unsigned)items;
            acc += items;
            if (dir == 0) b->items_per_stage[q / count] += items;
        }
        bases[(size_t)dir * (3 * count + 1) + 3 * count] = acc;
    }
    // the stage descriptors, then the radix plans they point to
    std::vector<unsigned char> up(stage_bytes + plan_bytes);
    const MixPlan* d_plans = reinterpret_cast<const MixPlan*>(reinterpret_cast<unsigned char*>(b->d_stages) + stage_bytes);
    for (BatchStage& bs : st) bs.args.aux = d_plans + reinterpret_cast<size_t>(bs.args.aux);
    std::memcpy(up.data(), st.data(), stage_bytes);
    std::memcpy(up.data() + stage_bytes, plans.data(), plan_bytes);
    e = cudaMemcpy(b->d_stages, up.data(), up.size(), cudaMemcpyHostToDevice);
    if (!e) e = cudaMemcpy(b->d_item_base, bases.data(), bases.size() * sizeof(int64_t), cudaMemcpyHostToDevice);
    if (!e) e = cudaMemcpy(b->d_need, needs.data(), needs.size() * sizeof(unsigned), cudaMemcpyHostToDevice);
    if (!e) e = cudaMemcpy(b->d_scratch, b->scratch.data(), sizeof(void*) * (size_t)count, cudaMemcpyHostToDevice);
    if (!e) e = cudaStreamCreateWithFlags(&b->own, cudaStreamNonBlocking);
    if (!e) e = cudaEventCreateWithFlags(&b->ev_in, cudaEventDisableTiming);
    if (!e) e = cudaEventCreateWithFlags(&b->ev_out, cudaEventDisableTiming);
    if (e) { free_batch(b); return fail(OPENFFT_ERR_CUDA, cudaGetErrorString(e)); }
    e = cudaDeviceSynchronize();
    if (e) { free_batch(b); return fail(OPENFFT_ERR_CUDA, cudaGetErrorString(e)); }
    *out = b;
    return OPENFFT_OK;
}

static cudaError_t launch_batch(BatchPlan* b, int dir_index, cudaStream_t s)
{
    BatchDev d;
    d.stages = b->d_stages;
    d.item_base = b->d_item_base + (size_t)dir_index * (3 * b->count + 1);
    d.need = b->d_need + (size_t)dir_index * 3 * b->count;
    d.ptrs = b->d_ptrs;
    d.scratch = b->d_scratch;
    d.ctr = reinterpret_cast<BatchCounters*>(b->d_ctr);
    d.done = reinterpret_cast<unsigned*>(b->d_ctr + sizeof(BatchCounters));
    d.count = b->count;
    d.dir_index = dir_index;
    d.wait_budget = b->wait_budget;
    cudaError_t e = cudaMemsetAsync(b->d_ctr, 0, b->ctr_bytes, s);
    if (e) return e;
    e = cudaMemcpyAsync(b->d_ptrs, b->h_ptrs, sizeof(void*) * (size_t)(2 * b->count), cudaMemcpyHostToDevice, s);
    if (e) return e;
    const size_t tables = sizeof(int64_t) * (size_t)(3 * b->count + 1) + sizeof(unsigned) * (size_t)(3 * b->count);
    const size_t sm = b->smem + tables;
    void* args[] = {&d, &b->smem};
    return cudaLaunchKernel(kernel_of(b->arith == ARITH_F32, b->wide), dim3((unsigned)b->grid), dim3(threads_of(b->wide)), args, sm, s);
}

int batch_exec(BatchPlan* b, const void* const* in, void* const* out, int dir, cudaStream_t user,
               int (*fail)(int, const char*))
{
    if (!b || !in || !out) return fail(OPENFFT_ERR_INVALID_ARG, "null plan or pointer arrays");
    if (dir != OPENFFT_FORWARD && dir != OPENFFT_BACKWARD) return fail(OPENFFT_ERR_INVALID_ARG, "dir must be -1 or +1");
    std::vector<void*> ptrs((size_t)2 * b->count);
    for (int i = 0; i < b->count; ++i) {
        if (!in[i] || !out[i]) return fail(OPENFFT_ERR_INVALID_ARG, "null transform buffer");
        if (in[i] == out[i]) return fail(OPENFFT_ERR_ALIAS, "in and out must differ (out-of-place only)");
        ptrs[(size_t)2 * i] = const_cast<void*>(in[i]);
        ptrs[(size_t)2 * i + 1] = out[i];
    }
    cudaError_t e;
    if (ptrs != b->cur_ptrs) {
        // the graph's copy node reads h_ptrs when it runs: wait for earlier replays first
        if ((e = cudaStreamSynchronize(b->own))) return fail(OPENFFT_ERR_CUDA, cudaGetErrorString(e));
        std::memcpy(b->h_ptrs, ptrs.data(), sizeof(void*) * ptrs.size());
        b->cur_ptrs = ptrs;
    }
    const int di = dir == OPENFFT_FORWARD ? 0 : 1;
    if (!b->exec[di]) {
        cudaGraph_t g = nullptr;
        if ((e = cudaStreamBeginCapture(b->own, cudaStreamCaptureModeThreadLocal))) return fail(OPENFFT_ERR_CUDA, cudaGetErrorString(e));
        cudaError_t le = launch_batch(b, di, b->own);
        e = cudaStreamEndCapture(b->own, &g);
        if (le || e) { if (g) cudaGraphDestroy(g); return fail(OPENFFT_ERR_CUDA, cudaGetErrorString(le ? le : e)); }
        e = cudaGraphInstantiate(&b->exec[di], g, 0);
        cudaGraphDestroy(g);
        if (e) { b->exec[di] = nullptr; return fail(OPENFFT_ERR_CUDA, cudaGetErrorString(e)); }
    }
    // order the replay after the caller's stream and the caller's stream after the replay
    if ((e = cudaEventRecord(b->ev_in, user))) return fail(OPENFFT_ERR_CUDA, cudaGetErrorString(e));
    if ((e = cudaStreamWaitEvent(b->own, b->ev_in, 0))) return fail(OPENFFT_ERR_CUDA, cudaGetErrorString(e));
    if ((e = cudaGraphLaunch(b->exec[di], b->own))) return fail(OPENFFT_ERR_CUDA, cudaGetErrorString(e));
    if ((e = cudaEventRecord(b->ev_out, b->own))) return fail(OPENFFT_ERR_CUDA, cudaGetErrorString(e));
    if ((e = cudaStreamWaitEvent(user, b->ev_out, 0))) return fail(OPENFFT_ERR_CUDA, cudaGetErrorString(e));
    return OPENFFT_OK;
}

int batch_status(BatchPlan* b, int (*fail)(int, const char*))
{
    cudaError_t e = cudaStreamSynchronize(b->own);
    if (e) return fail(OPENFFT_ERR_CUDA, cudaGetErrorString(e));
    BatchCounters c;
    e = cudaMemcpy(&c, b->d_ctr, sizeof(c), cudaMemcpyDeviceToHost);
    if (e) return fail(OPENFFT_ERR_CUDA, cudaGetErrorString(e));
    if (c.status != OPENFFT_OK) return fail(c.status, "a bounded dependency wait of the batched kernel ran out");
    return OPENFFT_OK;
}

int batch_set_wait_budget(BatchPlan* b, long long cycles)
{
    b->wait_budget = cycles;
    return OPENFFT_OK;
}

int batch_inject_stall(BatchPlan* b, int enable)
{
    // test hook (forward direction, stage 1 of transform 0): its stage-2 items
    // wait for one more stage-1 tile than exists, so the bounded wait runs out
    const size_t off = 0;
    unsigned v = 0;
    cudaError_t e = cudaMemcpy(&v, b->d_need + off, sizeof(unsigned), cudaMemcpyDeviceToHost);
    if (e) return OPENFFT_ERR_CUDA;
    const unsigned base = v - b->need_extra;
    b->need_extra = enable ? 1u : 0u;
    v = base + b->need_extra;
    e = cudaMemcpy(b->d_need + off, &v, sizeof(unsigned), cudaMemcpyHostToDevice);
    return e ? OPENFFT_ERR_CUDA : OPENFFT_OK;
}

int64_t batch_items(BatchPlan* b) { return b->items_per_stage[0] + b->items_per_stage[1] + b->items_per_stage[2]; }
int batch_count(BatchPlan* b) { return b->count; }
int64_t batch_points(BatchPlan* b, int i) { return b->N[(size_t)i]; }

}  // namespace ofg
