// fft_stage.h -- host-visible description of one FFT stage launch.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>
#include "checked.h"

namespace ofg {

constexpr int kStageThreads = 256;     // threads per CTA of the stage kernel
constexpr int kMaxLinesPerCta = 32;    // G <= 32
constexpr int kMaxPasses = 16;
constexpr int kMaxLen = 2048;          // longest supported axis (two tiles of one line fit in smem)

// element formats in global memory (real arrays of the real transform: R64 / R32)
enum { FMT_C128 = 0, FMT_C64 = 1, FMT_DF = 2, FMT_R64 = 3, FMT_R32 = 4 };
// arithmetic: FP64, FP32, double-float, and the split-precision tensor-core
// DFT-GEMM forms (complex64 data)
enum { ARITH_F64 = 0, ARITH_F32 = 1, ARITH_DF = 2, ARITH_TC_TF32 = 3, ARITH_TC_BF16 = 4 };

// Lines of a stage are l = i1 + i2 * M1 (i1 < M1, i2 < M2), each contiguous
// of length n at in + l * n.  Output element (l, k) goes to
// out[i1 * S1 + i2 * S2 + k * Sk].  A CTA takes G consecutive values of i1
// (group_i2 = 0) or of i2 (group_i2 = 1), the coordinate whose output stride
// is 1, so a store at fixed k writes G consecutive elements.  With M3 > 1 that
// geometry repeats: line l + i3 M1 M2, out + i3 S3, for i3 < M3 (0 stands for 1).
struct StageArgs {
    const void* in;
    void* out;
    const void* tw;            // twiddle table of length n (W[e] = exp(-2 pi i e / n))
    const void* aux;           // DFT-GEMM stages: operand image of the DFT matrices
    int64_t M1, M2, S1, S2, Sk;
    int64_t M3, S3;
    int64_t ngroups;           // ceil(M_grouped / G)
    double scale;              // applied at store (1.0 = none)
    float scale_hi, scale_lo;  // the same as an FP32 pair (split_scale)
    int n, G, log2G;
    int group_i2, contig_store;
    int npass;
    int radix[kMaxPasses];
    int conj_in, conj_out, do_fft;
    int in_fmt, out_fmt;
    // elements of the arrays that in and out point into, counted from those
    // pointers (launch_stage fills in M1 M2 n when left 0), and the status
    // word of the bounds checks; read only by the checked build (checked.h)
    int64_t in_elems, out_elems;
    int* chk;
};


// A positive output factor as an FP32 pair with hi + lo = scale: hi does not exceed
// it and lo is positive, so that v hi + v lo of an infinite v is infinite.  Split
// here and not by every thread (64x48x100 complex64 backward, three stages:
// 13.2 -> 12.3 us).
inline void split_scale(StageArgs& a)
{
    a.scale_hi = (float)(a.scale * (1.0 - 0x1p-24));
    a.scale_lo = (float)(a.scale - (double)a.scale_hi);
}

struct StageLaunch {
    StageArgs args;
    int arith;
    int64_t grid;              // CTAs of the generic kernel = tiles of G lines
    size_t smem;               // dynamic shared memory of the generic kernel
    int sms;                   // multiprocessors of the device (persistent grids)
    int family;                // KERNEL_*: which stage kernel runs this launch
    int* status;               // device status word (DFT-GEMM stages)
    // lines of the stage that this launch is a range of (0: it is the whole stage)
    int64_t stage_lines = 0;
    // 1: the launch waits until the kernel before it has ended.  For a stage whose twiddle
    // table that kernel writes: the stage kernels read tables through the read-only path,
    // which wants them complete before the kernel is resident.
    int apart = 0;
};

// Lines that the choice of a stage's kernel goes by.  A range of lines takes the kernel
// of its whole stage: the kernels round differently, and openfft_exec_c2c_host, which
// runs the first and the last stage range by range, gives openfft_exec_c2c's bits.
inline int64_t choice_lines(const StageLaunch& L) { return L.stage_lines ? L.stage_lines : L.args.M1 * L.args.M2; }

// stage kernel families: warp-per-line (power-of-two n), tile (specialised n), generic
// (any n).  AUTO takes the any-length kernel (fft_mix.cuh), or on power-of-two lengths the
// warp kernels where they are faster (fft_tile_df.cu, fft_tile_f32.cu), and what neither
// takes goes to the tile or the generic kernel
enum { KERNEL_AUTO = 0, KERNEL_WARP = 1, KERNEL_TILE = 2, KERNEL_GENERIC = 3 };
// the real stages of the real transform (r2c.cu): the forward stage 1 and the
// inverse's last stage; M1 = number of real lines, G = complex lines per CTA
enum { KERNEL_R2C = 4, KERNEL_C2R = 5 };
cudaError_t launch_real_stage(const StageLaunch& L, cudaStream_t st);
// its any-length kernel (r2c_mix.cu); *handled = false when the stage has none
cudaError_t launch_real_mix(const StageLaunch& L, cudaStream_t st, bool* handled);

// Stage kernels are launched with programmatic stream serialisation: a stage's CTAs
// may become resident while the stage before it drains, and wait there
// (grid_wait, which every stage kernel passes before it touches global memory)
// until that grid has completed and its writes are visible.  It takes the launch
// gap, about 2 us, out of the chain of stages: 32^3 complex128 went from 16.4 to
// 11.8 us a transform.  The next stage may start when every CTA of this one has
// ended, and only the asynchronous-output kernels say so earlier (grid_release), when
// they wait for nothing but the copy engine (256^3 complex128 373 us without, 364
// with).  The earlier a CTA says it, the sooner the next stage's CTAs gather on the SMs that
// have room first: said at the start of a CTA's last tile, 64x48x100 complex64
// backward took 12.2 us instead of 10.2, 72^3 complex128 28 instead of 21, 180x200x225
// real inverse in float 61 instead of 56, 512^3 complex128 3220 instead of 3150; at
// the start of the kernel, 240x288x320 complex64 316 instead of 227.
#ifdef __CUDACC__
__device__ __forceinline__ void grid_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_release() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
template <class... P, class... Args>
cudaError_t launch_chained(const StageLaunch& L, void (*kern)(P...), unsigned grid, int threads, size_t smem, cudaStream_t st,
                           const Args&... args)
{
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = L.apart ? 0 : 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, P(args)...);
}
#endif

cudaError_t stage_kernels_init(int max_dyn_smem);
// Device allocation of the library's workspaces (capi.cu): cudaMalloc, except
// that a test control (openfft_debug_alloc_fail) can make the n-th call fail
// as if the device were out of memory.
cudaError_t dev_malloc(void** ptr, size_t bytes);
// Resident CTAs per SM of a persistent kernel with `threads` threads and
// `dyn_smem` bytes of dynamic shared memory, from the kernel's own limits
// (shared memory with the whole carveout as shared memory, registers,
// threads); *carveout (if given) is the percentage that these CTAs need.
cudaError_t resident_ctas_per_sm(const void* func, int threads, size_t dyn_smem, int* per_sm, int* carveout = nullptr);
// The same for a kernel that is always launched with `dyn_smem` bytes; sets the kernel's
// dynamic shared memory limit and carveout.
cudaError_t persistent_ctas_per_sm(const void* func, int threads, size_t dyn_smem, int* per_sm);
// Launch properties are cached per device (kernel attributes are per device):
// the current device's slot of `slots`, or nullptr beyond kMaxDevices (then
// the caller recomputes on every launch).
constexpr int kMaxDevices = 64;
inline int* device_slot(int (&slots)[kMaxDevices])
{
    int d = 0;
    if (cudaGetDevice(&d) != cudaSuccess || d < 0 || d >= kMaxDevices) return nullptr;
    return &slots[d];
}
// specialised kernels (fft_tile_*.cu); *handled = false when (n, G) has none
cudaError_t launch_tile_f64(const StageLaunch& L, cudaStream_t st, bool* handled);
cudaError_t launch_tile_f32(const StageLaunch& L, cudaStream_t st, bool* handled);
cudaError_t launch_tile_df(const StageLaunch& L, cudaStream_t st, bool* handled);
// the asynchronous-output double-float kernels (fft_tma_256.cu, fft_tma_512.cu)
cudaError_t launch_warp_tma_256(const StageLaunch& L, cudaStream_t st, bool* handled);
cudaError_t launch_warp_tma_512(const StageLaunch& L, cudaStream_t st, bool* handled);
// any length (fft_mix_df.cu, fft_mix_f32.cu)
cudaError_t launch_mix_df(const StageLaunch& L, cudaStream_t st, bool* handled);
cudaError_t launch_mix_f32(const StageLaunch& L, cudaStream_t st, bool* handled);
cudaError_t launch_stage(const StageLaunch& L, cudaStream_t st);
// Twiddle table of length n in format fmt (FMT_C128, FMT_C64 or FMT_DF);
// twiddle_bytes(n, fmt) bytes at out.
cudaError_t launch_twiddles(int n, int fmt, void* out, cudaStream_t st);
inline size_t twiddle_bytes(int n, int fmt) { return (size_t)n * (fmt == FMT_C64 ? 8 : (fmt == FMT_DF ? 32 : 16)); }

// DFT-GEMM stages (dftgemm.cu): n = R S with 2 <= R, S <= 32 (radix[0] = R,
// radix[1] = S); status receives OPENFFT_ERR_TIMEOUT if an MMA wait runs out.
// The stage reads the split operand image of its two DFT matrices from
// args.aux (dftgemm_image_bytes bytes, built once by launch_dftgemm_image from
// the complex64 twiddle table of length n).
bool dftgemm_factor(int n, int tf32, int* R, int* S);
int dftgemm_lines(int n, int R, int S, bool tf32, int Gt);
size_t dftgemm_image_bytes(int n, int R, int S, bool tf32);
cudaError_t launch_dftgemm_image(int n, int R, int S, bool tf32, const void* tw, void* out, cudaStream_t st);
cudaError_t launch_dftgemm(const StageLaunch& L, cudaStream_t st, int* status);

}  // namespace ofg
