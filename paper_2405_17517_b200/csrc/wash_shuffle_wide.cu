// Translation unit of the streaming shuffle for populations of more than 16 models.
#include "wash_shuffle_wide.cuh"

namespace wash {

cudaError_t launch_shuffle_stream_wide(const ShuffleArgs &args, int a_dtype, int b_dtype, const LaunchShape &shape,
                                       cudaStream_t stream, bool *supported)
{
    return launch_shuffle_wide(args, a_dtype, b_dtype, shape, stream, supported);
}

}  // namespace wash
