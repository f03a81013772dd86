// Host side of the encoders: fills the kernel parameters and picks the translation unit that holds
// the kernels of the element type and draw width (uq_encode.cuh has the kernels).
#include "uq_encode.cuh"

namespace uq {

// idx_bits == 0 selects the single-scale quantizer (scales = {s}).  select: find and store the shared
// indices first instead of reading them.  out / S (may be NULL; S only with out): also add the workers'
// levels up and write the reconstructed average / the integer sums.
cudaError_t launch_encode(const uq_layout &L, const void *g, const float *W, const ScaleSet &scales,
                          uint8_t *idx, int idx_bits, bool select, uint64_t seed, int rng_bits, int fmt,
                          void *lev, float *out, int32_t *S, uint32_t *status, cudaStream_t st)
{
    EncodeParams p;
    p.v.g = g; p.v.W = W; p.v.seg_off = L.seg_off; p.v.d = L.d; p.v.stride = L.worker_stride; p.v.nseg = L.nseg; p.v.M = L.M;
    p.v.s_hat = (float)scales.s[0];
    p.v.scales = scales;
    p.lev = lev; p.out = out; p.S = S; p.idx = idx; p.status = status;
    p.select = select ? 1 : 0; p.idx_bits = idx_bits;
    p.worker0 = L.worker0; p.coord0 = L.coord0;
    p.key = philox_key(seed);
    if (L.dtype == UQ_F32) return rng_bits == 32 ? launch_encode_f32_r32(p, fmt, st) : launch_encode_f32_r16(p, fmt, st);
    return rng_bits == 32 ? launch_encode_bf16_r32(p, fmt, st) : launch_encode_bf16_r16(p, fmt, st);
}

}  // namespace uq
