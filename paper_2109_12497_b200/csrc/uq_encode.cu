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

// Whether selection, quantization, and sum with reconstruction run faster as kernels of their own.  In one kernel a warp
// takes its row through all workers, so few rows of many workers leave most of the GPU idle, and the row that holds d, in
// its slow form, is what the kernel ends up waiting for (0.55 to 0.7 us per worker; steps of 2, 4 and 8 binary32 workers,
// which no line below concerns, have no slow form there); the kernels of their own deal the
// workers out in groups of eight and cost a launch each.  One kernel / separate ones, launches without gaps, binary32,
// 4 scales, 32-bit draws (without selection; with it; selection and levels alone): 4 001 coordinates, M = 8: 0.84 / 1.00 /
// 1.18, M = 16: 1.18 / 1.26 / 1.56, M = 64: 2.6 / 2.2 / 3.1 times; 399 999 coordinates, M = 16: 1.05 / 0.77 / 1.29, M = 32:
// 1.51 / 1.04 / 1.25, M = 64: 1.59 / 1.35 / 1.70; 1 000 003, M = 32: 1.06 / 1.10 / 1.24.  Whole rows (d a multiple of 256),
// 4 096 coordinates, M = 16: 1.00 / 0.78 / 1.10, M = 64: 1.88 / 1.45 / 2.10; 401 408, M = 32: 1.07 / 0.75 / 0.89.  With a
// layer table the kernels of their own lose more in the rows that boundaries cross, where they walk along the table (161
// layers; 120 003 coordinates, M = 16: 0.91 / 0.81 / 1.08, M = 24: 1.12 / 0.90 / 1.25, M = 32: 1.29 / 0.91 / 1.54, M = 64: 1.74 /
// 1.33 / 1.83; 400 001, M = 24: 0.91 / 0.80 / 0.99, M = 32: 1.20 / 0.84 / 1.11, M = 64: 1.51 / 1.19 / 1.48).  The lines below are straight ones through where the two are even, over both element types
// and draw widths.
static bool better_separate(const uq_layout &L, bool reconstruct)
{
    const bool whole_rows = L.d % 256 == 0, layers = L.nseg > 1;
    if (reconstruct) {
        if (whole_rows) return L.M > 28 && L.d <= (int64_t)6000 * (L.M - 28);
        return layers ? L.M > 24 && L.d <= (int64_t)5000 * L.M : L.M >= 20 && L.d <= (int64_t)12000 * L.M;
    }
    return whole_rows ? L.M > 24 && L.d <= (int64_t)10000 * (L.M - 16) : L.M >= (layers ? 16 : 8) && L.d <= (int64_t)30000 * L.M;
}

// Kernels that launch_encode starts.
int encode_launches(const uq_layout &L, bool select, bool reconstruct)
{
    if (L.d == 0) return 0;
    return (select || reconstruct) && better_separate(L, reconstruct) ? 1 + select + reconstruct : 1;
}

// idx_bits == 0 selects the single-scale quantizer (scales = {s}).  select: find and store the shared
// indices first instead of reading them.  out / S (may be NULL; S only with out): also add the workers'
// levels up and write the reconstructed average / the integer sums.
cudaError_t launch_encode(const uq_layout &L, const void *g, const float *W, const ScaleSet &scales,
                          uint8_t *idx, int idx_bits, bool select, uint64_t seed, int rng_bits, int fmt,
                          void *lev, float *out, int32_t *S, uint32_t *status, cudaStream_t st)
{
    const bool reconstruct = out != nullptr;
    if (encode_launches(L, select, reconstruct) > 1) {
        cudaError_t e = select ? launch_select(L, g, W, scales, idx_bits, idx, status, st) : cudaSuccess;
        if (e == cudaSuccess)
            e = launch_encode(L, g, W, scales, idx, idx_bits, false, seed, rng_bits, fmt, lev, nullptr, nullptr, status, st);
        return e != cudaSuccess || !reconstruct ? e : launch_aggregate_decode(L, lev, fmt, W, scales, idx, idx_bits, out, S, st);
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
