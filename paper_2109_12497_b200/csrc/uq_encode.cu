// Host side of the encoders: fills the kernel parameters and picks the translation unit that holds
// the kernels of the element type and draw width (uq_encode.cuh has the kernels).
#include "uq_encode.cuh"

namespace uq {

cudaError_t launch_select(const uq_layout &L, const void *g, const float *W, const ScaleSet &scales,
                          int idx_bits, uint8_t *idx, uint32_t *status, cudaStream_t st);
cudaError_t launch_aggregate_decode(const uq_layout &L, const void *lev, int fmt, const float *W,
                                    const ScaleSet &scales, const uint8_t *idx, int idx_bits, float *out,
                                    int32_t *S, cudaStream_t st, float *theta = nullptr, float *mom = nullptr,
                                    float lr = 0.0f, float mu = 0.0f, float wd = 0.0f);

// Whether quantization, sum and reconstruction run faster as kernels of their own: with so few rows that a
// warp scheduler does not even get one, and so many workers that a warp's way through all of them takes
// longer than the launches (M = 32, d = 5674, two scales: 39.3 us for the step in one kernel, 35.4 us in three).
static bool better_separate(const uq_layout &L) { return L.M > 3 * kGroup && L.d <= (int64_t)148 * 4 * 256; }

// idx_bits == 0 selects the single-scale quantizer (scales = {s}).  select: find and store the shared
// indices first instead of reading them.  out / S (may be NULL; S only with out): also add the workers'
// levels up and write the reconstructed average / the integer sums.
cudaError_t launch_encode(const uq_layout &L, const void *g, const float *W, const ScaleSet &scales,
                          uint8_t *idx, int idx_bits, bool select, uint64_t seed, int rng_bits, int fmt,
                          void *lev, float *out, int32_t *S, uint32_t *status, cudaStream_t st)
{
    if (out != nullptr && better_separate(L)) {
        cudaError_t e = select ? launch_select(L, g, W, scales, idx_bits, idx, status, st) : cudaSuccess;
        if (e == cudaSuccess)
            e = launch_encode(L, g, W, scales, idx, idx_bits, false, seed, rng_bits, fmt, lev, nullptr, nullptr, status, st);
        return e != cudaSuccess ? e : launch_aggregate_decode(L, lev, fmt, W, scales, idx, idx_bits, out, S, st);
    }
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
