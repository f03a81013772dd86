// The encoder's kernels for bf16 gradients and 32-bit draws (see uq_encode.cuh).
#include "uq_encode.cuh"

namespace uq {

cudaError_t launch_encode_bf16_r32(const EncodeParams &p, int fmt, cudaStream_t st)
{
    return dispatch_fmt<UQ_BF16, 32>(p, fmt, st);
}

}  // namespace uq
