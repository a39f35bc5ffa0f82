// Translation unit of the sparse shuffle (mask first, only selected coordinates touched).
#include "wash_shuffle_sparse.cuh"

namespace wash {

cudaError_t launch_shuffle_sparse(const ShuffleArgs &args, int a_dtype, int b_dtype, const LaunchShape &shape,
                                  cudaStream_t stream, bool *supported)
{
    return launch_shuffle_sparse_tiles(args, a_dtype, b_dtype, shape, stream, supported);
}

}  // namespace wash
