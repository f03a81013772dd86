// Host side of the one-kernel step (uq_small.cuh has the kernel, uq_small_{f32,bf16}.cu its instances).
#include "uq_small.cuh"

namespace uq {

size_t small_workspace_bytes() { return kSmallHeader + (size_t)kSmallMaxCtas * kSmallMaxWorkers * sizeof(double); }

bool small_step_supported(const uq_layout &L, int fmt)
{
    return L.nseg == 1 && L.M <= kSmallMaxWorkers && (fmt == UQ_FMT_I8 || fmt == UQ_FMT_I4X2 || fmt == UQ_FMT_I2X4);
}

// idx_bits == 0 selects the single-scale quantizer (scales = {s}).
cudaError_t launch_small_step(const uq_layout &L, const void *g, int norm, const ScaleSet &scales, int idx_bits,
                              uint64_t seed, int rng_bits, int fmt, float *W, uint8_t *idx, void *lev, float *out,
                              int32_t *S, uint32_t *status, void *workspace, cudaStream_t st)
{
    SmallParams p;
    p.g = g; p.lev = lev; p.idx = idx; p.W = W; p.out = out; p.S = S; p.status = status;
    p.counter = (uint32_t *)workspace;
    p.part = (double *)((char *)workspace + kSmallHeader);
    p.d = L.d; p.stride = L.worker_stride; p.coord0 = L.coord0; p.M = L.M; p.worker0 = L.worker0;
    p.fmt = fmt; p.idx_bits = idx_bits; p.rounds = 1; p.scales = scales;
    p.key = philox_key(seed);
    return L.dtype == UQ_F32 ? launch_small_f32(p, norm, rng_bits, st) : launch_small_bf16(p, norm, rng_bits, st);
}

}  // namespace uq
