// One whole step of either quantizer in ONE kernel, for gradients so small that the launches of the regular
// step cost more than its arithmetic (Algorithm 1 / 2, lines "MaxAllReduce Norm" to "Reconstruct gradient";
// one segment, at most 8 workers).
//
// A thread owns units of 8 coordinates of all workers, loads them once and keeps them in registers (8
// unit-rows: UPT units of MW workers) across the scale agreement:
//   phase 1  the norm accumulators of the workers, reduced over the CTA
//   exchange the CTAs' partials: CLUSTER (8 or 16 CTAs): through distributed shared memory, behind the
//            cluster barrier; otherwise through the scratch, behind an arrival counter (zero when the kernel
//            starts: the caller zeroes the scratch once, the last CTA to go zeroes it again).  Nothing is assumed
//            about which CTAs are resident: a CTA marks its share as taken before it begins, and one that has
//            waited for long takes a share that nobody has, so the grid gets on with whatever part of it runs (a
//            CTA whose share was taken returns; W and the status flags are written by whoever holds share 0).
//            The wait is bounded all the same: a CTA that gives up sets UQ_STATUS_TIMEOUT and returns.  All
//            warps add up the partials in the same fixed order, so all of them hold the same bits of W
//   phase 2  [the shared indices from the maxima over the workers,] quantization of the workers' units, level
//            rows, sums in packed lanes, average
// Only a gradient with more units than the grid holds, and shares taken from others, are read again in phase 2.  Levels,
// indices, sums and the reconstruction are bit for bit those of the separate calls given the same W; W itself is summed in
// another fixed order (L2: within one unit in the last place of the regular kernel's).
//
// What bounds it is latency: one trip to memory, the barrier, the chains of the Philox rounds.  Measured on a
// B200, launches back to back (a grid with a counter in memory, every value loaded twice -> this form):
// 4 x 4099 bf16, 8 scales 8.8 -> 5.2 us, 8 x 10^4 fp32 10.1 -> 6.8 us (one cluster).  A step of 2 x 2^20 binary32 took
// 12.3 us as a cooperative launch, which is what such launches take one after the other in a stream whatever the kernel
// does (11.0 in a replayed graph); as an ordinary one, whose launch overlaps the kernel in front, 10.1, and with one fence
// at the barrier instead of three 9.8.  (The draws of the first units made while their loads are on their way, kept in
// shared memory: no gain on the grid, one cluster 5.5 -> 6.0 us.)
#pragma once
#include "uq_device.cuh"
#include "uq_norm.cuh"
#include "uq_select.cuh"
#include "uq_unit.cuh"

namespace uq {

constexpr int kSmallMaxWorkers = 8;
constexpr int kSmallHeader = 64;                  // bytes in front of the partials: arrival and departure counters, shares taken
constexpr int kSmallTaken = 2;                    // the header's first word of the bits of shares taken
constexpr int kSmallShares = (kSmallHeader / 4 - kSmallTaken) * 32;
constexpr uint32_t kSmallSpinLimit = 1u << 20;    // polls of the counter before a CTA gives up (about a second)
constexpr uint32_t kSmallPatience = 64;           // polls before it looks for a share that nobody has taken (about 50 us)
constexpr int kSmallThreads = 512;                // most threads per CTA
constexpr int kSmallMinThreads = 128;             // least threads per CTA of a grid

struct SmallParams {
    const void *g;
    void *lev;
    uint8_t *idx;             // multi-scale only
    float *W, *out;
    int32_t *S;
    uint32_t *status;
    uint32_t *counter;        // scratch: [0] arrivals, [1] departures, [kSmallTaken ..] shares taken
    double *part;             // scratch: [gridDim.x][kSmallMaxWorkers]
    int64_t d, stride, coord0;
    int32_t M, worker0, fmt, idx_bits;
    int32_t rounds;           // units per thread / UPT, rounded up; 1: everything stays in registers
    ScaleSet scales;          // single-scale: every entry is s
    PhiloxKey key;
};

__device__ __forceinline__ uint32_t ld_acquire(const uint32_t *p)
{
    uint32_t v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }

// A double of CTA `rank`'s shared memory, at the place of `p` in mine.
__device__ __forceinline__ double ld_cluster(const double *p, uint32_t rank)
{
    uint32_t a;
    double v;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank));
    asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(a) : "memory");
    return v;
}

__device__ __forceinline__ void store_unit_any(int fmt, uint32_t lo, uint32_t hi, char *row, int64_t i)
{
    if (fmt == UQ_FMT_I8) store_unit<UQ_FMT_I8>(lo, hi, row + i, nullptr);
    else if (fmt == UQ_FMT_I4X2) store_unit<UQ_FMT_I4X2>(lo, hi, row + (i >> 1), nullptr);
    else store_unit<UQ_FMT_I2X4>(lo, hi, row + (i >> 2), nullptr);
}

// One warp: the sums of partials k = first, first + step, .. < n of each of MW workers (value(k, m)); lane L
// ends with that of worker L % MW.  The order depends on the arguments only.
template <int NORM, int MW, typename F> __device__ __forceinline__ double sum_partials(int first, int step, int n, F value)
{
    const int lane = threadIdx.x & 31, m = lane & (MW - 1);
    constexpr int PARTS = 32 / MW;
    double a = 0.0;
    for (int k0 = first + step * (lane / MW); k0 < n; k0 += 4 * step * PARTS) {      // four loads in flight, added in order
        double v[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) v[k] = k0 + k * step * PARTS < n ? value(k0 + k * step * PARTS, m) : 0.0;   // 0 is neutral for both norms
#pragma unroll
        for (int k = 0; k < 4; ++k) a = combine<NORM>(a, v[k]);
    }
    __syncwarp();
#pragma unroll
    for (int o = 16; o >= MW; o >>= 1) a = combine<NORM>(a, __shfl_xor_sync(0xFFFFFFFFu, a, o));
    return a;
}

// W from the workers' sums (lane L: worker L % MW).
template <int NORM, int MW> __device__ __forceinline__ float scale_from_sums(double a, int M)
{
    const int m = threadIdx.x & (MW - 1);
    const bool nan = __any_sync(0xFFFFFFFFu, m < M && a != a);            // (fmax drops a NaN)
    double top = m < M ? a : 0.0;
#pragma unroll
    for (int o = MW / 2; o > 0; o >>= 1) top = fmax(top, __shfl_xor_sync(0xFFFFFFFFu, top, o));
    if (NORM == UQ_NORM_L2) return nan ? __uint_as_float(0x7FC00000u) : __double2float_rn(sqrt(top));
    return __uint_as_float((uint32_t)top);
}

template <int DT, int NORM, int RNG, bool MULTI, bool CLUSTER, int MW>
__global__ void __launch_bounds__(kSmallThreads, 1)
small_step_kernel(const __grid_constant__ SmallParams p)
{
    if (CLUSTER) grid_dependency_prologue();
    else grid_dependency_wait();
    using E = Elem<DT>;
    constexpr int H = 8 / E::G, UPT = kSmallMaxWorkers / MW;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarps = blockDim.x >> 5;
    const int M = p.M, ib = p.idx_bits;
    const int64_t d = p.d, nunits = (d + 7) >> 3;
    int64_t t = (int64_t)blockIdx.x * blockDim.x + tid;                 // of the share that I am at
    const int64_t T = (int64_t)gridDim.x * blockDim.x;
    __shared__ double sh[kSmallThreads / 32][MW], sh2[kSmallThreads / 32][MW];
    __shared__ double sh_part[MW];
    __shared__ int sh_next;                                              // after the wait: -1 go on, below: return, else a share to take
    __shared__ uint16_t sh_taken[kSmallShares];                        // shares that I took from others

    uint4 q[UPT][MW][H];
    auto load = [&](int round) {
#pragma unroll
        for (int k = 0; k < UPT; ++k) {
            const int64_t u = (int64_t)(round * UPT + k) * T + t, i = u << 3;
#pragma unroll
            for (int m = 0; m < MW; ++m)
#pragma unroll
                for (int h = 0; h < H; ++h)
                    q[k][m][h] = u < nunits && m < M
                        ? ld_stream((const char *)p.g + ((size_t)m * (size_t)p.stride + (size_t)i + h * E::G) * E::BYTES) : make_uint4(0u, 0u, 0u, 0u);
            if (u < nunits && i + 8 > d) {                             // the row's padding counts as zeros
#pragma unroll
                for (int m = 0; m < MW; ++m)
#pragma unroll
                    for (int h = 0; h < H; ++h) {
                        uint32_t w[4] = {q[k][m][h].x, q[k][m][h].y, q[k][m][h].z, q[k][m][h].w};
#pragma unroll
                        for (int c = 0; c < 4; ++c) {
                            const int64_t e = i + h * E::G + c * (4 / E::BYTES);      // first coordinate of the word
                            if (e >= d) w[c] = 0u;
                            else if (DT == UQ_BF16 && e + 1 >= d) w[c] &= 0xFFFFu;
                        }
                        q[k][m][h] = make_uint4(w[0], w[1], w[2], w[3]);
                    }
            }
        }
    };

    // ---- phase 1: per-worker norm partials of a share's units.  mine (thread 0's counts): nobody else has the share.  A CTA
    // that came late for its own reads it all the same, since the answer takes as long as the loads, but stores nothing:
    // others may be reading.
    auto norms = [&](int share, uint32_t mine) {
        Acc<NORM> acc[MW];
        for (int round = 0; round < p.rounds; ++round) {
            load(round);
#pragma unroll
            for (int m = 0; m < MW; ++m)
#pragma unroll
                for (int k = 0; k < UPT; ++k)
#pragma unroll
                    for (int h = 0; h < H; ++h) {
                        float v[E::G];
                        E::unpack(q[k][m][h], v);
#pragma unroll
                        for (int e = 0; e < E::G; ++e) acc[m].add(v[e]);
                    }
        }
#pragma unroll
        for (int m = 0; m < MW; ++m) {
            const double w = m < M ? warp_reduce<NORM>(acc[m].value()) : 0.0;
            if (lane == 0) sh[warp][m] = w;
        }
        __syncthreads();
        if (!CLUSTER && warp == 0) mine = __shfl_sync(0xFFFFFFFFu, mine, 0);
        if (tid < MW) {
            double tot = sh[0][tid];
            for (int k = 1; k < nwarps; ++k) tot = combine<NORM>(tot, sh[k][tid]);
            if (CLUSTER) sh_part[tid] = tot;
            else if (mine) __stcg(p.part + (size_t)share * kSmallMaxWorkers + tid, tot);
        }
    };
    uint32_t mine = 1;                                                  // whether my share is still mine
    if (!CLUSTER && tid == 0) mine = !(atomicOr(p.counter + kSmallTaken + (blockIdx.x >> 5), 1u << (blockIdx.x & 31)) >> (blockIdx.x & 31) & 1u);

    // ---- the exchange, and W
    int taken = 0;
    bool holds_first = blockIdx.x == 0;                                 // share 0 is mine, from the start or taken
    float W;
    if (CLUSTER) {
        norms(0, 1u);
        __syncwarp();
        cluster_arrive();
        cluster_wait();
        W = scale_from_sums<NORM, MW>(sum_partials<NORM, MW>(0, 1, (int)gridDim.x, [&](int c, int m) { return ld_cluster(sh_part + m, c); }), M);
        cluster_arrive();                          // waited for at the end: my shared memory may be read until then
    } else {
        int share = blockIdx.x;
        while (true) {
            norms(share, mine);
            __syncwarp();                     // (the partials are this warp's)
            if (tid == 0) {
                if (mine) {
                    __threadfence();          // release: this share's partials before its arrival
                    atomicAdd(p.counter, 1u);
                }
                int next = mine ? -1 : -3;
                for (uint32_t polls = 0; mine && ld_acquire(p.counter) < gridDim.x; ++polls) {
                    if (polls > kSmallSpinLimit) { next = -2; break; }
                    if (polls % kSmallPatience == kSmallPatience - 1) {
                        // a share that nobody has: its CTA may be waiting for an SM that I hold
                        for (int w = 0; w * 32 < (int)gridDim.x && next < 0; ++w) {
                            const uint32_t all = gridDim.x - w * 32 >= 32 ? 0xFFFFFFFFu : (1u << (gridDim.x - w * 32)) - 1u;
                            const uint32_t open = all & ~ld_acquire(p.counter + kSmallTaken + w);
                            if (open == 0u) continue;
                            const uint32_t bit = open & (0u - open);
                            if (!(atomicOr(p.counter + kSmallTaken + w, bit) & bit)) next = w * 32 + __ffs((int)bit) - 1;
                        }
                        if (next >= 0) break;
                    }
                    __nanosleep(32);
                }
                if (next == -2) atomicOr(p.status, (uint32_t)UQ_STATUS_TIMEOUT);
                sh_next = next;
                // the last CTA to go puts the counters and the marks back to zero for the next call (every CTA has
                // looked at its mark and read its last value of the arrival counter by then)
                if ((next == -1 || next == -3) && atomicAdd(p.counter + 1, 1u) == gridDim.x - 1) {
                    for (int w = kSmallHeader / 4 - 1; w >= 0; --w) p.counter[w] = 0u;
                }
            }
            __syncthreads();
            share = sh_next;
            if (share < -1) return;
            if (share == -1) break;
            if (tid == 0) sh_taken[taken] = (uint16_t)share;
            ++taken;
            holds_first |= share == 0;
            t = (int64_t)share * blockDim.x + tid;
        }
        // The next kernel's CTAs may come now and no sooner: where two fit an SM (up to 256 threads), those that came while
        // the grid was starting piled up on the SMs that it left free, and the next step ran at the pace of these.  8
        // binary32 workers of 122 880 / 262 144 coordinates, steps without gaps: 11.4 / 12.7 us with the kernel's first
        // instruction, 9.1 / 10.0 from here; 1 worker of 262 144 6.6 / 6.1, of 2^20 (512 threads) 7.8 / 7.9.
        grid_dependency_trigger();
        // each warp every nwarps-th CTA's partials, then every warp all warps' sums
        const double a = sum_partials<NORM, MW>(warp, nwarps, (int)gridDim.x,
                                                [&](int c, int m) { return __ldcg(p.part + (size_t)c * kSmallMaxWorkers + m); });
        if (lane < MW) sh2[warp][lane] = a;
        __syncthreads();
        W = scale_from_sums<NORM, MW>(sum_partials<NORM, MW>(0, 1, nwarps, [&](int w, int m) { return sh2[w][m]; }), M);
    }

    // ---- phase 2.  Lane k holds the factor s_k / W, the reconstruction factor W / (s_k * M) and the pass
    // threshold of scale k (single-scale: every lane the same factors)
    const float cap = (float)p.scales.s[0];
    const int32_t s_lane = p.scales.s[lane & (UQ_MAX_SCALES - 1)];
    const float inv_lane = inv_scale(s_lane, W), c_lane = decode_factor(W, s_lane, M);
    if (holds_first && warp == 0) {
        const bool overflow = __any_sync(0xFFFFFFFFu, lane < p.scales.N && not_finite(inv_lane));
        if (lane == 0) {
            p.W[0] = W;
            const uint32_t flags = (not_finite(W) ? UQ_STATUS_NONFINITE : 0u) | (overflow ? UQ_STATUS_SCALE_OVERFLOW : 0u);
            if (flags && p.status) atomicOr(p.status, flags);
        }
        __syncwarp();
    }
    int32_t thr = -1;
    int top = 0;                                                        // the bisection's first step
    if (MULTI) {
        if (lane < p.scales.N) thr = pass_threshold(inv_lane, cap);
        top = p.scales.N > 1 ? 1 << (31 - __clz(p.scales.N - 1)) : 0;
        __syncwarp();
    }
    const size_t row_bytes = (size_t)(p.stride >> p.fmt);
    const bool again = p.rounds > 1 || taken > 0;                       // the values have left the registers
    for (int share = 0; share <= taken; ++share) {
    t = (int64_t)(share == 0 ? blockIdx.x : sh_taken[share - 1]) * blockDim.x + tid;
    for (int round = 0; round < p.rounds; ++round) {
        if (again) load(round);
#pragma unroll
        for (int k = 0; k < UPT; ++k) {
            const int64_t u = (int64_t)(round * UPT + k) * T + t, i = u << 3;
            const bool active = u < nunits;
            if (!__any_sync(0xFFFFFFFFu, active)) break;                // the same for all lanes
            float inv[8], c[8];
            if (MULTI) {
                // the shared indices from the maxima over the workers (see uq_select.cuh)
                uint32_t amag[8];
#pragma unroll
                for (int e = 0; e < 8; ++e) amag[e] = 0u;
#pragma unroll
                for (int m = 0; m < MW; ++m)
#pragma unroll
                    for (int h = 0; h < H; ++h) {
                        const uint32_t w[4] = {q[k][m][h].x, q[k][m][h].y, q[k][m][h].z, q[k][m][h].w};
#pragma unroll
                        for (int x = 0; x < 4; ++x) {
                            if (DT == UQ_F32) amag[(4 * h + x) & 7] = max(amag[(4 * h + x) & 7], w[x] & 0x7FFFFFFFu);
                            else {
                                amag[(2 * x) & 7] = max(amag[(2 * x) & 7], (w[x] << 16) & 0x7FFFFFFFu);
                                amag[(2 * x + 1) & 7] = max(amag[(2 * x + 1) & 7], w[x] & 0x7FFF0000u);
                            }
                        }
                    }
                uint64_t packed = 0;
                int ks[8];
#pragma unroll
                for (int e = 0; e < 8; ++e) ks[e] = 0;
                for (int step = top; step >= 1; step >>= 1)
#pragma unroll
                    for (int e = 0; e < 8; ++e)
                        if ((int32_t)amag[e] <= __shfl_sync(0xFFFFFFFFu, thr, ks[e] + step)) ks[e] += step;
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    if (!active || i + e >= d) ks[e] = 0;                // padding keeps index 0
                    packed |= (uint64_t)ks[e] << (e * ib);
                    inv[e] = __shfl_sync(0xFFFFFFFFu, inv_lane, ks[e]);
                    c[e] = __shfl_sync(0xFFFFFFFFu, c_lane, ks[e]);
                }
                if (active) {
                    if (ib == 1) p.idx[i >> 3] = (uint8_t)packed;
                    else if (ib == 2) *(uint16_t *)(p.idx + (i >> 2)) = (uint16_t)packed;
                    else if (ib == 4) *(uint32_t *)(p.idx + (i >> 1)) = (uint32_t)packed;
                    else *(uint64_t *)(p.idx + i) = packed;
                }
            } else {
#pragma unroll
                for (int e = 0; e < 8; ++e) { inv[e] = inv_lane; c[e] = c_lane; }
            }
            if (active) {                                               // no warp-wide operation in here
                const uint64_t blk = RNG == 32 ? (uint64_t)((p.coord0 + i) >> 2) : (uint64_t)((p.coord0 + i) >> 3);
                int sum[2][2] = {{0, 0}, {0, 0}};                       // two levels share a word (see the encoder)
#pragma unroll
                for (int m = 0; m < MW; ++m) {
                    if (m < M) {
                        float v[8];
#pragma unroll
                        for (int h = 0; h < H; ++h) E::unpack(q[k][m][h], *(float(*)[E::G])(v + h * E::G));
                        uint32_t neg_lo, neg_hi, w[2];
                        unit_signs<DT>(q[k][m], neg_lo, neg_hi);
                        quantize_unit_bytes<RNG>(v, inv, cap, neg_lo, neg_hi,
                                                 unit_words<RNG>(p.key, (uint32_t)blk, (uint32_t)(blk >> 32), (uint32_t)(m + p.worker0)), w[0], w[1]);
                        store_unit_any(p.fmt, w[0], w[1], (char *)p.lev + (size_t)m * row_bytes, i);
#pragma unroll
                        for (int x = 0; x < 2; ++x) {
                            sum[x][0] = __dp2a_lo(0x40000001, (int)w[x], sum[x][0]);
                            sum[x][1] = __dp2a_hi(0x40000001, (int)w[x], sum[x][1]);
                        }
                    }
                }
                uint32_t s[8], r[8];
#pragma unroll
                for (int x = 0; x < 2; ++x)
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const int hi = (sum[x][h] + 0x2000) >> 14;
                        s[4 * x + 2 * h + 1] = (uint32_t)hi;
                        s[4 * x + 2 * h] = (uint32_t)(sum[x][h] - (hi << 14));
                    }
#pragma unroll
                for (int e = 0; e < 8; ++e) r[e] = __float_as_uint(__fmul_rn((float)(int)s[e], c[e]));
                if (i + 8 <= d) {
                    st_stream256(p.out + i, r);
                    if (p.S != nullptr) st_stream256(p.S + i, s);
                } else {
#pragma unroll
                    for (int e = 0; e < 8; ++e)
                        if (i + e < d) {
                            p.out[i + e] = __uint_as_float(r[e]);
                            if (p.S != nullptr) p.S[i + e] = (int32_t)s[e];
                        }
                }
            }
            __syncwarp();
        }
    }
    }
    if (CLUSTER) {
        __syncwarp();
        cluster_wait();
    }
}

// ---------------------------------------------------------------------------------------------
// launch
// ---------------------------------------------------------------------------------------------
constexpr int kSmallMaxCtas = 148 * 8 * 2;            // what callers size the scratch for; a grid has at most kSmallShares
static_assert(kSmallShares <= kSmallMaxCtas, "the scratch holds a partial per share and worker");

// CTAs of one instantiation that fit the device at once (with more, shares would wait for one another); looked up once
// per device and instantiation.
template <typename K> static int resident_ctas(K kernel, int *cache)
{
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
    if (cache[dev] == 0) {
        int sms = 0, per_sm = 0;
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, kSmallThreads, 0);
        cache[dev] = sms > 0 && per_sm > 0 ? sms * per_sm : -1;
    }
    return cache[dev] > 0 ? cache[dev] : 0;
}

// The largest cluster that the device schedules: 16 CTAs (an opt-in) or the portable 8; once per device and
// instantiation.
template <typename K> static int cluster_ctas(K kernel, int *cache)
{
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 8;
    if (cache[dev] == 0) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(16);
        cfg.blockDim = dim3(kSmallThreads);
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = 16; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        int clusters = 0;
        const bool ok = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
                        cudaOccupancyMaxActiveClusters(&clusters, kernel, &cfg) == cudaSuccess && clusters > 0;
        if (!ok) cudaGetLastError();
        cache[dev] = ok ? 16 : 8;
    }
    return cache[dev];
}

template <int DT, int NORM, int RNG, bool MULTI, int MW>
static cudaError_t launch_small_one(SmallParams p, cudaStream_t st)
{
    constexpr int UPT = kSmallMaxWorkers / MW;
    const int64_t nunits = (p.d + 7) / 8;
    cudaLaunchConfig_t cfg = {};
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    cfg.attrs = attr;
    // One cluster, a unit per thread, up to 4096 units: its few SMs then take no longer than a grid over all of them
    // loses in its barrier.  Grid / cluster, replayed graph, us, 1, 2, 4 and 8 binary32 workers: 32 768 coordinates 5.7 / 4.2,
    // 6.0 / 4.8, 6.6 / 5.6, 8.2 / 7.8; 40 000 5.8 / 4.8, 6.0 / 5.4, 6.6 / 6.6, 8.2 / 9.4; 50 000 5.8 / 5.5, 6.0 / 6.3,
    // 6.7 / 7.9, 8.1 / 11.4.
    if (nunits <= 8 * kSmallThreads) {
        static int ccache[64] = {};
        // one warp per scheduler of 8 SMs is not worth spreading further
        const int ctas = nunits <= 8 * 128 ? 8 : cluster_ctas(small_step_kernel<DT, NORM, RNG, MULTI, true, MW>, ccache);
        const int64_t want = (nunits + ctas - 1) / ctas;
        cfg.gridDim = dim3((unsigned)ctas);
        cfg.blockDim = dim3((unsigned)max((want + 31) / 32 * 32, (int64_t)32));
        p.rounds = 1;
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = (unsigned)ctas; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
        cfg.numAttrs = 1 + grid_dependency_attribute(attr + 1);
        return cudaLaunchKernelEx(&cfg, small_step_kernel<DT, NORM, RNG, MULTI, true, MW>, p);
    }
    static int cache[64] = {};
    const int resident = min(resident_ctas(small_step_kernel<DT, NORM, RNG, MULTI, false, MW>, cache), kSmallShares);
    if (resident <= 0) return cudaErrorNotSupported;
    // As many CTAs as the GPU takes before any has more than kSmallMinThreads threads: with 512 threads in each, a
    // gradient of 60 000 coordinates was left to a tenth of the SMs.  At least 256 / 128 / 64 threads, replayed graph, us: 1
    // binary32 worker of 60 000 coordinates 5.9 / 5.8 / 5.8, 4 workers 7.2 / 6.8 / 7.1, 8 workers 8.9 / 8.4 / 8.8, 8 of 120 000
    // 9.0 / 8.8 / 8.8, of 200 000 9.2 / 9.5 / 9.5.
    const int64_t threads = max((int64_t)kSmallMinThreads, min((int64_t)kSmallThreads, ((nunits + resident - 1) / resident + 31) / 32 * 32));
    const int64_t per = (nunits + threads - 1) / threads;                 // CTAs at one unit per thread
    p.rounds = (int)((per + (int64_t)resident * UPT - 1) / ((int64_t)resident * UPT));
    const int64_t units = (per + resident - 1) / resident;                // units per thread that the grid needs
    cfg.gridDim = dim3((unsigned)min((int64_t)resident, (per + units - 1) / units));
    cfg.blockDim = dim3((unsigned)threads);
    cfg.numAttrs = grid_dependency_attribute(attr);
    return cudaLaunchKernelEx(&cfg, small_step_kernel<DT, NORM, RNG, MULTI, false, MW>, p);
}

template <int DT, int NORM, int RNG, bool MULTI> static cudaError_t launch_small_workers(const SmallParams &p, cudaStream_t st)
{
    if (p.M <= 2) return launch_small_one<DT, NORM, RNG, MULTI, 2>(p, st);
    if (p.M <= 4) return launch_small_one<DT, NORM, RNG, MULTI, 4>(p, st);
    return launch_small_one<DT, NORM, RNG, MULTI, 8>(p, st);
}

template <int DT, int NORM> static cudaError_t launch_small_mode(const SmallParams &p, int rng_bits, cudaStream_t st)
{
    if (p.idx_bits != 0)
        return rng_bits == 32 ? launch_small_workers<DT, NORM, 32, true>(p, st) : launch_small_workers<DT, NORM, 16, true>(p, st);
    return rng_bits == 32 ? launch_small_workers<DT, NORM, 32, false>(p, st) : launch_small_workers<DT, NORM, 16, false>(p, st);
}

cudaError_t launch_small_f32(const SmallParams &p, int norm, int rng_bits, cudaStream_t st);
cudaError_t launch_small_bf16(const SmallParams &p, int norm, int rng_bits, cudaStream_t st);

}  // namespace uq
