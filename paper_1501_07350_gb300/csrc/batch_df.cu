// batch_df.cu -- the batched kernels in packed double-float.
#include "batch_kernel.cuh"

namespace ofg {

size_t batch_tile_bytes_df(int G, int n) { return batch_tile_bytes<ArDP>(G, n); }
const void* batch_kernel_df(bool wide)
{
    return wide ? (const void*)batch_kernel<ArDP, true> : (const void*)batch_kernel<ArDP, false>;
}

}  // namespace ofg
