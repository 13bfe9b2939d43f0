// batch_f32.cu -- the batched kernel in FP32.
#include "batch_kernel.cuh"

namespace ofg {

size_t batch_tile_bytes_f32(int G, int n) { return G == 8 ? batch_tile_bytes<ArF32, 8>(n) : batch_tile_bytes<ArF32, 4>(n); }
const void* batch_kernel_f32(int G) { return G == 8 ? (const void*)batch_kernel<ArF32, 8> : (const void*)batch_kernel<ArF32, 4>; }

}  // namespace ofg
