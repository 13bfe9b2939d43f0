// batch_df.cu -- the batched kernel in packed double-float.
#include "batch_kernel.cuh"

namespace ofg {

size_t batch_tile_bytes_df(int G, int n)
{
    return G == 8 ? batch_tile_bytes<ArDP, 8>(n) : (G == 4 ? batch_tile_bytes<ArDP, 4>(n) : batch_tile_bytes<ArDP, 2>(n));
}
const void* batch_kernel_df(int G)
{
    return G == 8 ? (const void*)batch_kernel<ArDP, 8>
                  : (G == 4 ? (const void*)batch_kernel<ArDP, 4> : (const void*)batch_kernel<ArDP, 2>);
}

}  // namespace ofg
