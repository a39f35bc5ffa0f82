// Translation unit of the dense operators (EMA, average, PAPA-all) on bf16 stacks.
#include "wash_reduce.cuh"

namespace wash {

cudaError_t launch_reduce_bf16(const ReduceArgs &args, int op, int out_dtype, const LaunchShape &shape, cudaStream_t stream)
{
    switch (op) {
    case kOpEma:
        return launch_reduce_typed<BF16, BF16, kOpEma>(args, shape, stream);
    case kOpPapaAll:
        return launch_reduce_typed<BF16, BF16, kOpPapaAll>(args, shape, stream);
    default:
        if (out_dtype == kDtypeF32) return launch_reduce_typed<BF16, F32, kOpAverage>(args, shape, stream);
        return launch_reduce_typed<BF16, BF16, kOpAverage>(args, shape, stream);
    }
}

}  // namespace wash
