// The encoder's kernels for binary32 gradients and 16-bit draws (see uq_encode.cuh).
#include "uq_encode.cuh"

namespace uq {

cudaError_t launch_encode_f32_r16(const EncodeParams &p, int fmt, cudaStream_t st)
{
    return dispatch_fmt<UQ_F32, 16>(p, fmt, st);
}

}  // namespace uq
