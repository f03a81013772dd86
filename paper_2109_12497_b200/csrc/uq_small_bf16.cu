// The one-kernel step for bfloat16 gradients (see uq_small.cuh).
#include "uq_small.cuh"

namespace uq {

cudaError_t launch_small_bf16(const SmallParams &p, int norm, int rng_bits, cudaStream_t st)
{
    return norm == UQ_NORM_L2 ? launch_small_mode<UQ_BF16, UQ_NORM_L2>(p, rng_bits, st)
                              : launch_small_mode<UQ_BF16, UQ_NORM_LINF>(p, rng_bits, st);
}

}  // namespace uq
