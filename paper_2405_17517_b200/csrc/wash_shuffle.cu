// Translation unit of the streaming shuffle (stack staged through shared memory by cp.async).
#include "wash_shuffle_async.cuh"

namespace wash {

cudaError_t launch_shuffle_stream(const ShuffleArgs &args, int a_dtype, int b_dtype, const LaunchShape &shape,
                                  cudaStream_t stream, bool *supported)
{
    return launch_shuffle_async(args, a_dtype, b_dtype, shape, stream, supported);
}

}  // namespace wash
