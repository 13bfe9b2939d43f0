// batch_f32.cu -- the batched kernels in FP32.
#include "batch_kernel.cuh"

namespace ofg {

size_t batch_tile_bytes_f32(int G, int n) { return batch_tile_bytes<ArF32>(G, n); }
const void* batch_kernel_f32(bool wide)
{
    return wide ? (const void*)batch_kernel<ArF32, true> : (const void*)batch_kernel<ArF32, false>;
}

}  // namespace ofg
