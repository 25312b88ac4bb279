// npm_tc_fwd_fp16.cu -- the tensor-core forward kernel (npm_tc_forward.cuh) in the
// FP16 operand format.
#include "npm_tc_forward.cuh"

namespace npm {
namespace tc {
template cudaError_t launch_fwd_ops<kOneFp16>(const TcCfg&, const void*, const uint4*, const uint8_t*, QueryBatch&, int64_t, int*,
                                        long long, bool, cudaStream_t);
}  // namespace tc
}  // namespace npm
