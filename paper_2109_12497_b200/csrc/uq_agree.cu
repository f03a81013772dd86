// Shared scale W[j] = max_m || g^m on segment j ||   (Algorithm 1, line "MaxAllReduce Norm").
//
// Two launches.  (1) norm_partials, norm_rows (large binary32 gradients: a CTA takes a tile of four workers) or
// norm_staged (small gradients in segments): the coordinate axis is cut into fixed tiles of kNormTile coordinates; the
// CTA of (tile t, worker m) reduces every segment that crosses its tile and
// stores one partial per (tile, segment) pair in slot t + j of worker m's scratch row.  Tiles and
// segments are both ordered, so t + j is unique for every pair and the row needs
// ntiles + nseg slots.  (2) norm_finalize: one CTA per segment adds that segment's slots in a
// fixed order, takes the max over workers, and writes W[j].  The summation tree depends only on
// (d, seg_off), never on the grid or on timing, so W is reproducible bit for bit.
#include <type_traits>

#include "uq_device.cuh"
#include "uq_norm.cuh"

namespace uq {

constexpr int kNormItems = 4;      // rows of a tile that a CTA takes
constexpr int kStagedTiles = 512;  // most tiles of all workers that norm_staged_kernel takes (where few boundaries cross many tiles it
                                   // loses: 1.5 M coordinates in 3 segments, 8 workers 10.9 -> 11.6 us)
constexpr int kDealtTiles = 256;   // and that it gives two warps per chunk: more CTAs than that fill the GPU (100 003 coordinates, 16 workers: 9.1 us with two, 9.0 with one)
constexpr int kSlab = 32768;       // tiles per grid.y step (keeps grid.x below 2^31)

template <int DT, int NORM>
__global__ void __launch_bounds__(kThreads, 8)     // 32 registers: eight CTAs per SM keep HBM busy
norm_partials_kernel(const void *__restrict__ g, int64_t d, int64_t stride, int nseg,
                     const int64_t *__restrict__ seg_off, int64_t ntiles, double *__restrict__ part)
{
    grid_dependency_prologue();
    using E = Elem<DT>;
    constexpr int UNITS = kNormTile / (kThreads * E::G);
    constexpr bool TILE_MAJOR = DT == UQ_F32;
    // CTA order, as measured on B200 (see launch): fp32 walks the tiles front to back with the worker
    // varying fastest (grid.x = M * tiles of one slab of kSlab tiles, grid.y = slab); bf16 streams
    // one worker's row front to back before the next worker's (grid.x = tile, grid.y = worker).
    int m;
    int64_t tile;
    if (TILE_MAJOR) {
        const uint32_t M = gridDim.x / (uint32_t)min(ntiles, (int64_t)kSlab);
        m = (int)(blockIdx.x % M);
        tile = (int64_t)blockIdx.y * kSlab + blockIdx.x / M;
        if (tile >= ntiles) return;                              // the last slab may be ragged
    } else {
        tile = blockIdx.x;
        m = blockIdx.y;
    }
    const int64_t t0 = tile * kNormTile;
    const int64_t t1 = min(t0 + (int64_t)kNormTile, d);
    const char *row = (const char *)g + (size_t)m * (size_t)stride * E::BYTES;
    double *prow = part + (size_t)m * (size_t)(ntiles + nseg);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;

    // The tile's vector loads (the row is padded, so a 16-byte load that starts before d is
    // legal) are issued before the segment lookup when they fit few registers (bf16: 4 loads),
    // after it otherwise (fp32: 8 loads; the lookup is two dependent loads for up to 1024
    // segments, hidden by the other resident CTAs).
    constexpr bool LOADS_FIRST = UNITS <= 4;
    uint4 q[UNITS];
    if (LOADS_FIRST) {
#pragma unroll
        for (int u = 0; u < UNITS; ++u) {
            const int64_t i = t0 + (int64_t)(u * kThreads + tid) * E::G;
            q[u] = i < t1 ? ld_stream(row + i * E::BYTES) : make_uint4(0, 0, 0, 0);
        }
    }
    const int j0 = warp_find_segment(seg_off, nseg, t0);
    if (segment_end(seg_off, nseg, j0, d) >= t1) {
        // the whole tile lies in segment j0: one block reduction in a fixed order
        if (!LOADS_FIRST) {
#pragma unroll
            for (int u = 0; u < UNITS; ++u) {
                const int64_t i = t0 + (int64_t)(u * kThreads + tid) * E::G;
                q[u] = i < t1 ? ld_stream(row + i * E::BYTES) : make_uint4(0, 0, 0, 0);
            }
        }
        Acc<NORM> acc;
        if (LOADS_FIRST && t1 - t0 == kNormTile) {    // full bf16 tile: no per-element bounds (for
                                                      // fp32 the unguarded form costs 2.5x the registers)
#pragma unroll
            for (int u = 0; u < UNITS; ++u) {
                float v[E::G];
                E::unpack(q[u], v);
#pragma unroll
                for (int e = 0; e < E::G; ++e) acc.add(v[e]);
            }
        } else {
#pragma unroll
            for (int u = 0; u < UNITS; ++u) {
                // elements of this unit that are data (the row's padding beyond d is not)
                const int valid = (int)min((int64_t)E::G, t1 - (t0 + (int64_t)(u * kThreads + tid) * E::G));
                float v[E::G];
                E::unpack(q[u], v);
#pragma unroll
                for (int e = 0; e < E::G; ++e)
                    if (e < valid) acc.add(v[e]);
            }
        }
        __shared__ double sh[kWarps];
        double w = warp_reduce<NORM>(acc.value());
        if (lane == 0) sh[warp] = w;
        __syncthreads();
        if (tid == 0) {
            double tot = sh[0];
#pragma unroll
            for (int k = 1; k < kWarps; ++k) tot = combine<NORM>(tot, sh[k]);
            prow[tile + j0] = tot;
        }
    } else {
        norm_mixed_tile<DT, NORM>(row, prow, tile, t0, t1, d, nseg, seg_off);
    }
}

// The ragged last tile of a CTA's workers, inside one segment (out of line: one tile of the grid).
template <int DT, int NORM>
__device__ __noinline__ void norm_ragged_tile(const char *__restrict__ row, int64_t row_bytes, double *__restrict__ slot, int64_t slots,
                                              int n, int64_t t0, int64_t t1)
{
    using E = Elem<DT>;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    __shared__ double sh[kNormItems][kWarps];
    for (int k = 0; k < n; ++k) {
        Acc<NORM> acc;
#pragma unroll 4
        for (int64_t i = t0 + (int64_t)tid * E::G; i < t1; i += kThreads * E::G) {
            float v[E::G];
            E::unpack(ld_stream(row + k * row_bytes + i * E::BYTES), v);      // (rows are padded to whole vectors)
#pragma unroll
            for (int e = 0; e < E::G; ++e)
                if (i + e < t1) acc.add(v[e]);
        }
        __syncwarp();
        const double w = warp_reduce<NORM>(acc.value());
        if (lane == 0) sh[k][warp] = w;
    }
    __syncthreads();
    if (tid < n) {
        double tot = sh[tid][0];
        for (int x = 1; x < kWarps; ++x) tot = combine<NORM>(tot, sh[tid][x]);
        slot[tid * slots] = tot;
    }
}

// A CTA takes up to kNormItems workers' rows of one tile.  A full tile inside one segment (the common case) has no
// bounds checks, one segment lookup and one barrier for all rows, and a vector's registers are filled again
// with the next row's as soon as it is added.  (With a CTA per row and checked elements a binary32 element
// cost 18 instructions, of which it needs 2.3: the kernel reached 0.95 of the copy peak in a burst and lost
// a tenth of it at the board's power cap.)
template <int DT, int NORM>
__global__ void __launch_bounds__(kThreads, 4)
norm_rows_kernel(const void *__restrict__ g, int64_t d, int64_t stride, int M, int nseg,
                 const int64_t *__restrict__ seg_off, int64_t ntiles, double *__restrict__ part)
{
    grid_dependency_prologue();
    using E = Elem<DT>;
    constexpr int UNITS = kNormTile / (kThreads * E::G);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // tiles front to back, a tile's groups of workers side by side (grid.x = groups * tiles of one slab of kSlab
    // tiles, grid.y = slab): the kernel ends on the high coordinates of all workers, which the encoder reads first
    const uint32_t groups = (uint32_t)(M + kNormItems - 1) / kNormItems;
    const int m = (int)(blockIdx.x % groups) * kNormItems;
    const int64_t tile = (int64_t)blockIdx.y * kSlab + blockIdx.x / groups;
    if (tile >= ntiles) return;                                       // the last slab may be ragged
    const int n = min(kNormItems, M - m);
    const int64_t t0 = tile * kNormTile, t1 = min(t0 + (int64_t)kNormTile, d);
    const int64_t row_bytes = stride * E::BYTES, slots = ntiles + nseg;
    const char *row = (const char *)g + m * row_bytes;
    double *prow = part + m * slots;
    uint4 q[UNITS];
    const char *p = row + (t0 + tid * E::G) * E::BYTES;
    if (t1 - t0 == kNormTile) {
#pragma unroll
        for (int u = 0; u < UNITS; ++u) q[u] = ld_stream(p + u * (kThreads * 16));
    }
    const int j = warp_find_segment(seg_off, nseg, t0);
    if (segment_end(seg_off, nseg, j, d) < t1) {
        for (int k = 0; k < n; ++k) {
            norm_mixed_tile<DT, NORM>(row + k * row_bytes, prow + k * slots, tile, t0, t1, d, nseg, seg_off);
            __syncthreads();                                            // its shared memory is free again
        }
        return;
    }
    if (t1 - t0 != kNormTile) {
        norm_ragged_tile<DT, NORM>(row, row_bytes, prow + tile + j, slots, n, t0, t1);
        return;
    }
    __shared__ double sh[kNormItems][kWarps];
#pragma unroll 1
    for (int k = 0; k < n; ++k) {
        p += row_bytes;
        const bool more = k + 1 < n;
        Acc<NORM> acc;
#pragma unroll
        for (int u = 0; u < UNITS; ++u) {
            float v[E::G];
            E::unpack(q[u], v);
#pragma unroll
            for (int e = 0; e < E::G; ++e) acc.add(v[e]);
            if (more) q[u] = ld_stream(p + u * (kThreads * 16));
        }
        const double w = warp_reduce<NORM>(acc.value());
        if (lane == 0) sh[k][warp] = w;
    }
    __syncthreads();
    if (tid < n) {
        double tot = sh[tid][0];
#pragma unroll
        for (int x = 1; x < kWarps; ++x) tot = combine<NORM>(tot, sh[tid][x]);
        prow[tile + j + tid * slots] = tot;
    }
}

// Small gradients in several segments.  What bounds them is latency: a layer table crosses nearly every tile, and a
// warp that walks the pieces of its chunk in memory makes a trip there for every few of them.  Here the whole tile
// is on its way to shared memory while the segment is looked up, the pieces are walked there, and the pieces of a
// chunk are dealt out to WPC warps.  The additions are those of norm_partials_kernel in the same order, so which of the
// two runs is a matter of speed alone.  Norms of 8 binary32 workers in 161 layers, both kernels, launches without gaps,
// by norm_partials_kernel / here with one / with two warps per chunk: 20 011 coordinates 15.0 / 11.1 / 9.2 us, 100 003
// 10.8 / 7.6 / 7.0 us, 400 003 14.8 / 8.9 / 8.9 us.
template <int DT, int NORM, int WPC>
__global__ void __launch_bounds__(kThreads * WPC)
norm_staged_kernel(const void *__restrict__ g, int64_t d, int64_t stride, int nseg, const int64_t *__restrict__ seg_off,
                   int64_t ntiles, double *__restrict__ part)
{
    grid_dependency_prologue();
    using E = Elem<DT>;
    using T = typename std::conditional<DT == UQ_F32, float, uint16_t>::type;
    constexpr int VECS = kNormTile / E::G, UNITS = VECS / kThreads, CHUNK = kNormTile / kWarps;
    __shared__ uint4 stage[VECS];
    __shared__ double sh_head[kWarps], sh_tail[kWarps];                  // as in norm_mixed_tile
    __shared__ int sh_head_seg[kWarps], sh_tail_seg[kWarps], sh_head_open[kWarps];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t tile = blockIdx.x, t0 = tile * kNormTile, t1 = min(t0 + (int64_t)kNormTile, d);
    const char *row = (const char *)g + (size_t)blockIdx.y * (size_t)stride * E::BYTES;
    double *prow = part + (size_t)blockIdx.y * (size_t)(ntiles + nseg);
    const uint32_t sp = (uint32_t)__cvta_generic_to_shared(stage);
#pragma unroll
    for (int v = tid; v < VECS; v += kThreads * WPC)                             // (rows are padded to whole vectors)
        if (t0 + v * E::G < t1) copy_async16(sp + v * 16, row + (t0 + v * E::G) * E::BYTES);
    if (tid < kWarps) sh_head_seg[tid] = sh_tail_seg[tid] = -1;
    const int chunk = warp / WPC, sub = warp % WPC;
    const int64_t c0 = t0 + (int64_t)chunk * CHUNK, c1 = min(c0 + CHUNK, t1);
    const int jt = warp_find_segment(seg_off, nseg, t0);
    int64_t ends = segment_end(seg_off, nseg, min(jt + lane, nseg - 1), d);                     // lane l: where segment jt + l ends
    const int64_t start = __ldg(seg_off + jt);
    const bool uniform = __shfl_sync(0xFFFFFFFFu, ends, 0) >= t1;
    int j0 = jt, base = jt;                                         // my chunk's first segment, and lane 0's
    int64_t seg_b = start;                                                                      // and where the one before it ends
    if (!uniform && c0 < c1) {
        const int before = __popc(__ballot_sync(0xFFFFFFFFu, ends <= c0 && jt + lane < nseg - 1));
        if (before == 32) {
            j0 = warp_find_segment(seg_off, nseg, c0);
            seg_b = __ldg(seg_off + j0);
        } else {
            j0 = jt + before;
            if (before > 0) seg_b = __shfl_sync(0xFFFFFFFFu, ends, before - 1);
        }
        if (j0 - jt >= 16) {
            ends = segment_end(seg_off, nseg, min(j0 + lane, nseg - 1), d);
            base = j0;
        }
    }
    copy_async_wait();
    __syncthreads();
    if (uniform) {
        Acc<NORM> acc;
        if (warp < kWarps) {
#pragma unroll
            for (int u = 0; u < UNITS; ++u) {
                const int64_t i = t0 + (int64_t)(u * kThreads + tid) * E::G;
                if (i >= t1) break;
                float v[E::G];
                E::unpack(stage[u * kThreads + tid], v);
#pragma unroll
                for (int e = 0; e < E::G; ++e)
                    if (i + e < t1) acc.add(v[e]);
            }
            __syncwarp();
            const double w = warp_reduce<NORM>(acc.value());
            if (lane == 0) sh_head[warp] = w;
        }
        __syncthreads();
        if (tid == 0) {
            double tot = sh_head[0];
#pragma unroll
            for (int k = 1; k < kWarps; ++k) tot = combine<NORM>(tot, sh_head[k]);
            prow[tile + jt] = tot;
        }
        return;
    }
    // The pieces of my chunk that are mine, four at a time: their reductions over the lanes overlap.
    int64_t a = c0;
    int j = j0, k = 0;
    bool more = a < c1;
    while (more) {
        double w[4];
        int seg[4];                                                              // -1: no piece
        bool first[4], goes_on[4];                                               // may continue one from the left; may continue to the right
#pragma unroll
        for (int n = 0; n < 4; ++n) {
            Acc<NORM> acc;
            seg[n] = -1;
            while (more && seg[n] < 0) {
                const int64_t seg_a = seg_b;
                if (j - base == 32) {
                    ends = segment_end(seg_off, nseg, min(j + lane, nseg - 1), d);
                    base = j;
                }
                seg_b = __shfl_sync(0xFFFFFFFFu, ends, j - base);
                const int64_t b = min(max(seg_b, a), c1);
                if (b > a && k++ % WPC == sub) {
                    seg[n] = j;
                    first[n] = a == c0 && seg_a < c0;
                    goes_on[n] = b == c1 && seg_b > c1;
#pragma unroll 8
                    for (int i = (int)(a - t0) + lane; i < (int)(b - t0); i += 32) {
                        const T x = *((const T *)stage + i);
                        acc.add(DT == UQ_F32 ? (float)x : __uint_as_float((uint32_t)x << 16));
                    }
                    __syncwarp();
                }
                a = b;
                more = a < c1 && j + 1 < nseg;
                ++j;
            }
            w[n] = acc.value();
        }
#pragma unroll
        for (int n = 0; n < 4; ++n) w[n] = warp_reduce<NORM>(w[n]);
        if (lane == 0) {
#pragma unroll
            for (int n = 0; n < 4; ++n) {
                if (seg[n] < 0) continue;
                if (first[n]) { sh_head[chunk] = w[n]; sh_head_seg[chunk] = seg[n]; sh_head_open[chunk] = goes_on[n]; }
                else if (goes_on[n]) { sh_tail[chunk] = w[n]; sh_tail_seg[chunk] = seg[n]; }
                else prow[tile + seg[n]] = w[n];
            }
        }
        __syncwarp();
    }
    __syncthreads();
    // What goes on to the right is added up in chunk order, a thread per piece that starts one: the tail of a chunk, or
    // the head of the tile's first.
    if (tid < 2 * kWarps) {
        int w = tid >> 1;
        const bool from_head = (tid & 1) != 0;
        const int j = from_head ? (w == 0 ? sh_head_seg[0] : -1) : sh_tail_seg[w];
        if (j >= 0) {
            double sum = from_head ? sh_head[0] : sh_tail[w];
            bool open = !from_head || sh_head_open[0];
            for (++w; open && w < kWarps && sh_head_seg[w] == j; ++w) {
                sum = combine<NORM>(sum, sh_head[w]);
                open = sh_head_open[w];
            }
            prow[tile + j] = sum;
        }
    }
}

// One CTA per segment, one warp per worker: lane l adds up the slots of the segment's tiles l, l + 32, .. one after
// the other, and then the lanes' sums are added.  That order depends on the segment's tiles alone: a worker's sum has
// the same bits whatever else is in the buffer.  What bounds it is the latency of the loads, of which a lane has K
// in flight: 8 workers of 13.1 M bf16 coordinates in one segment, the kernel 7.0 us with 8, 5.0 with 32, the step 132.2 and
// 130.9; 2 such workers 46.3 and 44.9, one binary32 worker of 25 M 69.6 and 67.3; 16 of 67 M no difference.  (With 32
// throughout, a CTA's registers do not fit beside the kernel in front of it: a step of 64 workers of 114 688 coordinates
// 46.5 -> 48 us.)  (Several warps fetching a worker's slots into shared memory for the one that adds: 1 worker 14.9 -> 13.4
// us, 2 to 4 workers no faster, and with 40 KB of it the kernel in front, beside whose CTAs these start, took 4 %
// longer; norms of 25.6 M bf16 coordinates in one segment.)
template <int NORM, int K>
__global__ void __launch_bounds__(512)
norm_finalize_kernel(const double *__restrict__ part, int M, int64_t d, int nseg,
                     const int64_t *__restrict__ seg_off, int64_t ntiles, float *__restrict__ W, uint32_t *__restrict__ status)
{
    grid_dependency_prologue();
    const int j = blockIdx.x;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarps = blockDim.x >> 5;
    int64_t a = seg_off ? __ldg(seg_off + j) : 0;
    int64_t b = seg_off ? __ldg(seg_off + j + 1) : d;
    const bool bad = a < 0 || b > d || a > b || (j == 0 && a != 0) || (j == nseg - 1 && b != d);
    a = min(max(a, (int64_t)0), d);
    b = min(max(b, a), d);

    __shared__ double sh[UQ_MAX_WORKERS];
    const int first = (int)(a / kNormTile), last = a < b ? (int)((b - 1) / kNormTile) : first - 1;
    for (int m = warp; m < M; m += nwarps) {
        const double *prow = part + (size_t)m * (size_t)(ntiles + nseg) + j;
        double acc = 0.0;
        for (int t = first + lane; t <= last; t += 32 * K) {
            double v[K];
#pragma unroll
            for (int k = 0; k < K; ++k) v[k] = t + k * 32 <= last ? __ldcg(prow + t + k * 32) : 0.0;      // 0 is neutral for both norms
#pragma unroll
            for (int k = 0; k < K; ++k) acc = combine<NORM>(acc, v[k]);
        }
        __syncwarp();
        const double r = warp_reduce<NORM>(acc);
        if (lane == 0) sh[m] = r;
    }
    __syncthreads();
    if (warp == 0) {
        // fmax drops NaN, so look for it explicitly
        bool nan = false;
        double top = 0.0;
        for (int m = lane; m < M; m += 32) {
            nan |= sh[m] != sh[m];
            top = fmax(top, sh[m]);
        }
        nan = __any_sync(0xFFFFFFFFu, nan);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) top = fmax(top, __shfl_xor_sync(0xFFFFFFFFu, top, o));
        if (lane == 0) {
            float w;
            if (NORM == UQ_NORM_L2) w = nan ? __uint_as_float(0x7FC00000u) : __double2float_rn(sqrt(top));
            else w = __uint_as_float((uint32_t)top);
            W[j] = w;
            uint32_t flags = 0;
            if ((__float_as_uint(w) & 0x7F800000u) == 0x7F800000u) flags |= UQ_STATUS_NONFINITE;
            if (bad) flags |= UQ_STATUS_BAD_SEGMENTS;
            if (flags && status) atomicOr(status, flags);
        }
    }
}

template <int DT, int NORM>
static cudaError_t launch(const uq_layout &L, const void *g, float *W, uint32_t *status, double *part,
                          int64_t ntiles, cudaStream_t st)
{
    if (L.d > 0 && L.nseg > 1 && ntiles * L.M <= kStagedTiles) {
        const dim3 grid((unsigned)ntiles, (unsigned)L.M);
        if (ntiles * L.M <= kDealtTiles)
            launch_k(norm_staged_kernel<DT, NORM, 2>, grid, kThreads * 2, st, g, L.d, L.worker_stride, L.nseg, L.seg_off, ntiles, part);
        else
            launch_k(norm_staged_kernel<DT, NORM, 1>, grid, kThreads, st, g, L.d, L.worker_stride, L.nseg, L.seg_off, ntiles, part);
    } else if (L.d > 0) {
        if (ntiles > 0x7FFFFFFFLL) return cudaErrorInvalidConfiguration;
        // binary32 takes several rows per CTA where that leaves eight waves and boundaries are rare (the rows of a
        // tile that one crosses are worked through one after the other): 16 rows of 33.6 M coordinates 342 ->
        // 300 us, 2 of 60 M 86 -> 71 us, sustained; with 161 segments in 25.6 M the slow tiles cost what the
        // others gain.  bf16 does not: its conversions to binary64 (8 cycles each per warp and scheduler) bound
        // it either way, and it wants a worker's row streamed front to back (13 M coordinates, 8 workers: 34 us
        // against 42)
        const int groups = (L.M + kNormItems - 1) / kNormItems;
        if (DT == UQ_F32 && L.M > 1 && ntiles * groups >= 148 * 4 * 8 && (int64_t)L.nseg * 64 <= ntiles) {
            const dim3 grid((unsigned)groups * (unsigned)min(ntiles, (int64_t)kSlab), (unsigned)((ntiles + kSlab - 1) / kSlab));
            launch_k(norm_rows_kernel<UQ_F32, NORM>, grid, kThreads, st, g, L.d, L.worker_stride, L.M, L.nseg, L.seg_off, ntiles, part);
        } else {
            // fp32: tile-major order is 5 % faster on the layer-segmented workloads and neutral on the
            // one-segment ones; bf16: it is 20 % slower than worker-major order
            dim3 grid((unsigned)ntiles, (unsigned)L.M);
            if (DT == UQ_F32)
                grid = dim3((unsigned)L.M * (unsigned)min(ntiles, (int64_t)kSlab), (unsigned)((ntiles + kSlab - 1) / kSlab));
            launch_k(norm_partials_kernel<DT, NORM>, grid, kThreads, st, g, L.d, L.worker_stride, L.nseg, L.seg_off, ntiles, part);
        }
    }
    // segments of more than eight loads per lane: 16 workers side by side, and more loads
    if (ntiles / L.nseg >= 256)
        launch_k(norm_finalize_kernel<NORM, 32>, L.nseg, 32 * min(L.M, 16), st, part, L.M, L.d, L.nseg, L.seg_off, ntiles, W, status);
    else
        launch_k(norm_finalize_kernel<NORM, 8>, L.nseg, kThreads, st, part, L.M, L.d, L.nseg, L.seg_off, ntiles, W, status);
    return cudaGetLastError();
}

int64_t norm_tiles(const uq_layout &L) { return (L.d + kNormTile - 1) / kNormTile; }

cudaError_t launch_agree_scale(const uq_layout &L, const void *g, int norm, float *W, uint32_t *status,
                               void *workspace, cudaStream_t st)
{
    const int64_t ntiles = norm_tiles(L);
    double *part = (double *)workspace;
    if (L.dtype == UQ_F32)
        return norm == UQ_NORM_L2 ? launch<UQ_F32, UQ_NORM_L2>(L, g, W, status, part, ntiles, st)
                                  : launch<UQ_F32, UQ_NORM_LINF>(L, g, W, status, part, ntiles, st);
    return norm == UQ_NORM_L2 ? launch<UQ_BF16, UQ_NORM_L2>(L, g, W, status, part, ntiles, st)
                              : launch<UQ_BF16, UQ_NORM_LINF>(L, g, W, status, part, ntiles, st);
}

}  // namespace uq

// ---------------------------------------------------------------------------------------------
// uq_agree_scale_static: the same computation with the scratch held inside the library
// ---------------------------------------------------------------------------------------------
#include <mutex>

namespace uq { int record_cuda_error(cudaError_t e); }

namespace {

// Scratch for the norm partials, part of the library image: every GPU that loads the library
// holds these bytes until the process exits.  In host code this name is only a handle; the
// device address comes from cudaGetSymbolAddress.
static __device__ __align__(256) unsigned char g_static_scratch[UQ_STATIC_SCRATCH_BYTES];

constexpr int kMaxDevices = 64;
std::mutex g_scratch_mutex;
void *g_scratch_addr[kMaxDevices] = {};      // device address of g_static_scratch, per device ordinal

// Device address of the scratch array on the current device, resolved once per device.
cudaError_t static_scratch(void **out)
{
    int dev = -1;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(g_scratch_mutex);
    if (g_scratch_addr[dev] == nullptr) {
        void *addr = nullptr;
        e = cudaGetSymbolAddress(&addr, g_static_scratch);
        if (e != cudaSuccess) return e;
        if (addr == nullptr) return cudaErrorInvalidSymbol;
        g_scratch_addr[dev] = addr;
    }
    *out = g_scratch_addr[dev];
    return cudaSuccess;
}

}  // namespace

extern "C" int uq_agree_scale_static(const uq_layout *layout, const void *g, int norm, float *W,
                                     uint32_t *status, void *stream)
{
    // size first: a layout that cannot fit is refused before CUDA is touched
    const size_t need = uq_workspace_bytes(layout);
    if (need == 0) return UQ_ERR_BAD_ARG;                       // the layout itself is invalid
    if (need > (size_t)UQ_STATIC_SCRATCH_BYTES) return UQ_ERR_WORKSPACE;
    void *scratch = nullptr;
    const cudaError_t e = static_scratch(&scratch);
    if (e != cudaSuccess) return uq::record_cuda_error(e);      // the code is kept for uq_last_cuda_error()
    // the partials are all written before they are read, so nothing in the array needs clearing
    return uq_agree_scale(layout, g, norm, W, status, scratch, (size_t)UQ_STATIC_SCRATCH_BYTES, stream);
}
