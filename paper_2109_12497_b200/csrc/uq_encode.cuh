// Stochastic quantization of every worker's gradient to small signed integers:
// Q_s (Section "QSGDMaxNorm Quantization", Algorithm 1 line "Quantize gradient") and
// Q_{s_} with the shared per-coordinate scale (Section "QSGDMaxNormMultiScale Quantization",
// Algorithm 2 line "Quantize with s*"), optionally with what stands around it in the algorithms
// when all workers are in this buffer: the choice and sharing of the scale indices in front (SEL),
// the integer sum over the workers and the reconstructed average behind (DEC).
//
// One streaming pass.  A thread owns 8 consecutive coordinates (a warp a row of 256 of them) and takes the
// workers' rows G at a time, straight-line; a worker's registers are filled again with the bytes of the
// worker G places on as soon as they are quantized.  What does not depend on the worker is done once: the
// segment lookup, the factors s_k / W of the coordinates, and the first two rounds of the Philox block,
// whose counter differs between workers in one word only; the G workers' blocks advance together, so
// that one fetch of a round key serves all of them.  The levels are added up in packed lanes as they are
// made, and the average leaves with them: the level rows are written (they are what crosses the wire)
// but never read back.  SEL: a first pass over the workers' rows takes the largest magnitude of every
// coordinate, which decides the shared index; the rows of 8 bf16 workers are kept in shared memory for
// the second pass, others come from the caches.  A warp is on its own (no barrier: with one lookup per CTA
// the warps waited for it longer than their own lookups take).
//
// Measured on a B200 (25.6 M binary32 coordinates in 161 layers, 8 workers, int8 levels, 32-bit draws;
// sustained): 235 us for quantization + sum + reconstruction, where two kernels took 210 + 53 us; with
// selection among 4 scales 266 us, where three took 130 + 216 + 53 us.
#pragma once
#include <type_traits>

#include "uq_device.cuh"
#include "uq_select.cuh"
#include "uq_unit.cuh"

namespace uq {

struct EncodeParams {
    SelectView v;             // g, W, seg_off, d, stride, nseg, M, scales (single-scale: every entry is s) and
                              // s_hat = (float) of the smallest scale: the largest level
    void *lev;
    float *out;               // the reconstructed average [d], or NULL
    int32_t *S;               // the integer sums [d], or NULL (needs out)
    uint8_t *idx;             // shared scale indices: read, or (select) written by this launch
    uint32_t *status;
    int32_t select;           // multi-scale: 1 = find the shared indices here instead of reading them
    int32_t idx_bits;         // 1, 2, 4 or 8; 0 for the single-scale quantizer
    int32_t worker0;          // number, in the whole job, of the worker in row 0 (keys the draws)
    uint32_t blk_hi;          // high word of the Philox block numbers the table below was made for
    int32_t split;            // workers per CTA (grid.y = ceil(M / split)); M unless only the levels are wanted
    int64_t coord0;           // index, in the whole gradient, of coordinate 0 (keys the draws)
    PhiloxKey key;            // the ten round keys of the seed; 16-bit draws: the last round's complemented, so that
                              // words 0 and 2 of a block come out complemented
    alignas(16) PhiloxWorkerPart wpart[UQ_MAX_WORKERS];   // per-worker words of the first two Philox rounds (row m)
};

constexpr int kGroup = 8;     // the number of workers that has kernels of its own (all of them straight-line)

// Launch shape per variant.  The kernel's time is its instructions: a warp scheduler issues one per cycle,
// except that a 32 x 32 -> 64 bit multiply (two per Philox round) holds it for about four (measured alone:
// multiply 4.3 cycles, with a logic operation beside it 4.5, with n additions beside it 4.3 + n - 0.4).
// So the shape is the one with the fewest instructions that still hides the loads: four chains of Philox
// rounds advance together, and four CTAs of 64 registers share an SM.  Measured on a B200 (8 workers,
// quantization + sum + reconstruction, sustained): bf16 with 32-bit draws 3 CTAs 188 us, 4 CTAs 197 us
// (26.2 M coordinates); binary32, selecting, 32-bit draws: one worker at a time 266 us, two 273 us (25.6 M).
//
// binary32, 2 and 4 workers: the kernels of 8 with fewer of them, no loop, nothing spilled.  Steps, general kernel / these:
// 4 workers of 25 M coordinates 176 / 173 us, of 25 M in 161 layers with 4 scales 247 / 218, 4-bit levels 171 / 165; 14.7 M with
// two scales and 6-bit levels 156.6 / 141.0; of 40 003, whose last row is no slow one now, 12.5 / 9.6 and with 4 scales 17.6 / 9.8.
// Levels alone, 2 / 4 workers of 25 M: 16-bit draws 48.9 / 46.2, 81.5 / 77.1; 32-bit draws 62.4 / 59.7, 103 / 96; with the index
// given 66.2 / 61.3, 108 / 102; selecting, without the average, 94.8 / 83.3, 149 / 131.  (Of 20 003 and of 1 M: 0.98 to 1.08 times.)
//
// Few workers (1 to 4 of bf16): what does not depend on the worker is then most of a lane's work, so all workers' blocks
// go together straight-line, their rows are staged as the eight's are, and fewer registers let more warps hide the way
// to memory.  25.6 M coordinates, 16-bit draws, general kernel / this / an encoder of two units per lane: levels alone,
// one worker in 161 layers 40.9 / 33.2 / 32.9 us, two workers in one segment 47.9 / 41.5 / 38.2; with selection, two
// workers 88.6 / 66.4 / 67.4.
template <int DT, int RNG, bool SEL, int WK> struct EncodeShape {
    static constexpr bool FEW = DT == UQ_BF16 && WK > 0 && WK < kGroup;
    static constexpr int V = 8 * Elem<DT>::BYTES / 16;                        // 16-byte words per thread and worker
    static constexpr int NB = RNG == 32 ? 2 : 1;                              // Philox blocks per thread and worker
    static constexpr int G = FEW ? (RNG == 16 ? WK : WK % 2 == 0 ? 2 : 1)      // workers whose blocks advance together
                                 : DT == UQ_F32 ? (SEL ? 1 : 2) : RNG == 32 ? 2 : 4;
    static constexpr int CTAS = FEW ? (WK <= 2 ? 5 : 4) : DT == UQ_BF16 && RNG == 32 ? 3 : 4;           // per SM
    static constexpr int TILE = kThreads * 8;
};

// ---------------------------------------------------------------------------------------------
// the packed indices of a unit: coordinates 0..3 in fields of ib bits from bit 0 of kw[0],
// coordinates 4..7 in kw[1] (loaded: bits beyond a word's four fields are anything; stored: they must be 0)
// ---------------------------------------------------------------------------------------------
__device__ __forceinline__ void load_indices(const uint8_t *idx, int64_t i, int ib, uint32_t (&kw)[2])
{
    const uint8_t *p = idx + ((i * ib) >> 3);
    if (ib == 8) {
        const uint2 x = __ldg((const uint2 *)p);
        kw[0] = x.x; kw[1] = x.y;
        return;
    }
    kw[0] = ib == 4 ? __ldg((const uint32_t *)p) : ib == 2 ? __ldg((const uint16_t *)p) : __ldg(p);
    kw[1] = kw[0] >> (4 * ib);
}

__device__ __forceinline__ void store_indices(uint8_t *idx, int64_t i, int ib, const uint32_t (&kw)[2])
{
    uint8_t *p = idx + ((i * ib) >> 3);
    if (ib == 8) { *(uint2 *)p = make_uint2(kw[0], kw[1]); return; }
    const uint32_t x = kw[0] | (kw[1] << (4 * ib));
    if (ib == 4) *(uint32_t *)p = x;
    else if (ib == 2) *(uint16_t *)p = (uint16_t)x;
    else *p = (uint8_t)x;
}

// ---------------------------------------------------------------------------------------------
// slow forms, out of line
// ---------------------------------------------------------------------------------------------

// Everything for the coordinates [r0, min(r0 + 256, d)), looked up coordinate by coordinate, in plain
// arithmetic: the row that d ends in, in the kernels that do not take it as the others, rows whose Philox
// block numbers leave the launch's high word, and rows whose factors are too small or too large for the
// rescaled forms.  Workers m_first .. m_last - 1 (all of them if the sums are wanted).  One warp; a lane
// takes a unit of 8 coordinates.
template <int DT, int FMT, int RNG, bool MULTI>
__device__ __noinline__ void encode_row_slow(const EncodeParams &p, int64_t r0, int m_first, int m_last)
{
    using E = Elem<DT>;
    using LF = LevelFmt<FMT>;
    const int64_t i = r0 + (threadIdx.x & 31) * 8, d = p.v.d;
    if (i >= min(r0 + 256, d)) return;
    int j = find_segment(p.v.seg_off, p.v.nseg, i);
    uint32_t kw[2] = {0u, 0u};
    if (MULTI) {
        if (p.select) {
            uint32_t amag[8];
            unit_max_magnitude<DT>(p.v, i, true, amag);
            const uint64_t packed = select_general(p.v, i, amag, p.idx_bits, j);
            kw[0] = (uint32_t)packed & (uint32_t)((1ull << (4 * p.idx_bits)) - 1ull);
            kw[1] = (uint32_t)(packed >> (4 * p.idx_bits));
            store_indices(p.idx, i, p.idx_bits, kw);
        } else {
            load_indices(p.idx, i, p.idx_bits, kw);
        }
    }
    float inv[8], c[8];
    bool overflow = false;
#pragma unroll
    for (int e = 0; e < 8; ++e) {
        inv[e] = c[e] = 0.0f;
        if (i + e < d) {
            j = advance_segment(p.v.seg_off, p.v.nseg, j, i + e);
            const float W = __ldg(p.v.W + j);
            const uint32_t k = MULTI ? (kw[e >> 2] >> ((e & 3) * p.idx_bits)) & ((1u << p.idx_bits) - 1u) & (UQ_MAX_SCALES - 1) : 0u;
            inv[e] = inv_scale(p.v.scales.s[k], W);
            c[e] = decode_factor(W, p.v.scales.s[k], p.v.M);
            overflow |= not_finite(inv[e]);
        }
    }
    if (overflow && p.status) atomicOr(p.status, (uint32_t)UQ_STATUS_SCALE_OVERFLOW);
    const uint64_t blk = RNG == 32 ? (uint64_t)((p.coord0 + i) >> 2) : (uint64_t)((p.coord0 + i) >> 3);
    int S[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    constexpr int G = 4, H = 8 / E::G;                              // workers whose loads are in flight together
    for (int m0 = m_first; m0 < m_last; m0 += G) {
        uint4 q[G][H];
#pragma unroll
        for (int g = 0; g < G; ++g) {
            const int m = min(m0 + g, m_last - 1);
#pragma unroll
            for (int h = 0; h < H; ++h)
                q[g][h] = ld_stream((const char *)p.v.g + ((size_t)m * (size_t)p.v.stride + i + h * E::G) * E::BYTES);
        }
#pragma unroll
        for (int g = 0; g < G; ++g) {
            const int m = m0 + g;
            if (m >= m_last) break;
            float v[8];
#pragma unroll
            for (int h = 0; h < H; ++h) E::unpack(q[g][h], *(float(*)[E::G])(v + h * E::G));
            uint32_t neg_lo, neg_hi, lo, hi;
            unit_signs<DT>(q[g], neg_lo, neg_hi);       // the sign of a padding coordinate is harmless: its level is 0
#pragma unroll
            for (int e = 0; e < 8; ++e)
                if (i + e >= d) v[e] = 0.0f;
            UnitWords<RNG> words = unit_words<RNG>(p.key, (uint32_t)blk, (uint32_t)(blk >> 32), (uint32_t)(m + p.worker0));
            if (RNG == 16) { words.r[0].x = ~words.r[0].x; words.r[0].z = ~words.r[0].z; }
            quantize_unit_bytes<RNG>(v, inv, p.v.s_hat, neg_lo, neg_hi, words, lo, hi);
            char *lrow = (char *)p.lev + (size_t)m * LF::row_bytes(p.v.stride);
            store_unit<FMT>(lo, hi, lrow + LF::off(i), lrow + LF::off2(i, p.v.stride));
#pragma unroll
            for (int e = 0; e < 8; ++e) S[e] += (int)(int8_t)((e < 4 ? lo : hi) >> (8 * (e & 3)));
        }
    }
    if (p.out == nullptr) return;
    for (int e = 0; e < 8 && i + e < d; ++e) {
        p.out[i + e] = __fmul_rn((float)S[e], c[e]);
        if (p.S != nullptr) p.S[i + e] = S[e];
    }
}

// The scales of the four coordinates at i (the first or the second half of a lane's unit) in a row that segment
// boundaries cross.  j: the segment that the row starts in.  The whole warp: lane l holds where segment j + l ends and its
// scale, and a coordinate's segment is the number of ends at or before it.  (Before, every lane walked along the table for
// every coordinate, loads behind each other, and the row that d ends in took the slow form above.  Steps of 8 binary32
// workers in 161 layers, before / with both changed: 100 003 coordinates 22.9 / 21.2 us, 16 384 coordinates with 6-bit
// levels 28.2 / 25.4; of 4 workers of 14.7 M with two scales, where it is the boundaries alone, 157.2 / 155.4.)
// The counts share a word: with a register each, the kernels of 1 and 2 bf16 workers spilled (2 workers of 45.9 M in 161 layers
// 134.4 us walking, 137.4 with a register each, 136.1 like this; of 64 M with two scales 265.8 / 264.3 / 262.9).
__device__ __forceinline__ float4 mixed_row_scales(const SelectView &v, int64_t i, int j)
{
    const int lane = threadIdx.x & 31, c = (int)(i & 255), at = min(j + lane, v.nseg - 1);
    // boundaries inside the row (a sorted table's are the first lanes), counted from the row's beginning
    const int rel = at == v.nseg - 1 ? 512 : (int)min(__ldg(v.seg_off + at + 1) - (i - c), (int64_t)512);
    const float W = __ldg(v.W + at);
    const int n = __popc(__ballot_sync(0xFFFFFFFFu, rel < 256));
    if (n < 32) {
        uint32_t k = 0;                                          // four counts of at most 31, a byte each
        for (int b = 0; b < n; ++b) {
            const int e = max(__shfl_sync(0xFFFFFFFFu, rel, b) - c, 0);
            k += e < 4 ? 0x01010101u << (8 * e) : 0u;
        }
        return make_float4(__shfl_sync(0xFFFFFFFFu, W, k & 31), __shfl_sync(0xFFFFFFFFu, W, k >> 8 & 31), __shfl_sync(0xFFFFFFFFu, W, k >> 16 & 31),
                           __shfl_sync(0xFFFFFFFFu, W, k >> 24));
    }
    // 32 and more: from where i is, along the table.  Steps of 2 to 8 workers of 1 000 to 3 000 coordinates in up to 161
    // layers, walking all the way from where the row starts / like this: 44 to 70 us / 38 to 59.
    float f[4];
    j = find_segment(v.seg_off, v.nseg, i);
#pragma unroll
    for (int x = 0; x < 4; ++x) {
        j = advance_segment(v.seg_off, v.nseg, j, i + x);
        f[x] = __ldg(v.W + j);
    }
    __syncwarp();
    return make_float4(f[0], f[1], f[2], f[3]);
}

// The factors of these coordinates: s_k / W for the quantization (dec = false) or W / (s_k * M) for the reconstruction.
// LANES: the scales come from the lanes; else every lane walks along the table, which leaves more registers to the caller.
template <bool LANES>
static __device__ __noinline__ float4 mixed_row_factors(const EncodeParams &p, int64_t i, int j, uint32_t kw, bool dec)
{
    const uint32_t mask = p.idx_bits == 0 ? 0u : ((1u << p.idx_bits) - 1u) & (UQ_MAX_SCALES - 1);
    const float4 w = LANES ? mixed_row_scales(p.v, i, j) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    float W[4] = {w.x, w.y, w.z, w.w};
    bool overflow = false;
    float f[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        if (!LANES) {
            j = advance_segment(p.v.seg_off, p.v.nseg, j, i + e);
            W[e] = __ldg(p.v.W + j);
        }
        const int32_t s = p.v.scales.s[(kw >> (e * p.idx_bits)) & mask];
        f[e] = dec ? decode_factor(W[e], s, p.v.M) : inv_scale(s, W[e]);
        overflow |= !dec && (!LANES || i + e < p.v.d) && not_finite(f[e]);     // (a walked row is a whole one)
    }
    if (overflow && p.status) atomicOr(p.status, (uint32_t)UQ_STATUS_SCALE_OVERFLOW);
    return make_float4(f[0], f[1], f[2], f[3]);
}

// The shared indices of these coordinates, from the largest magnitudes over the workers: the largest index that passes,
// by bisection (see uq_select.cuh: those that pass are the first ones).
static __device__ __noinline__ uint32_t mixed_row_select(const EncodeParams &p, int64_t i, int j, uint32_t a0, uint32_t a1, uint32_t a2,
                                                         uint32_t a3)
{
    const float4 w = mixed_row_scales(p.v, i, j);
    const float W[4] = {w.x, w.y, w.z, w.w};
    const uint32_t amag[4] = {a0, a1, a2, a3};
    uint32_t packed = 0;
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const float a = __uint_as_float(amag[e]);
        int k = 0;
        for (int step = UQ_MAX_SCALES / 2; step >= 1; step >>= 1)
            if (k + step < p.v.scales.N && __fmul_rn(a, inv_scale(p.v.scales.s[k + step], W[e])) <= p.v.s_hat) k += step;
        packed |= (uint32_t)k << (e * p.idx_bits);
    }
    return packed;
}

// What is left to do in the unit that d ends in, after the straight-line path: level 0 (and index 0, where this launch has
// found the indices) for the coordinates d and up, whatever the padding held.
template <int FMT> static __device__ __noinline__ void clear_padding(const EncodeParams &p, int64_t i)
{
    using LF = LevelFmt<FMT>;
    const int live = (int)(p.v.d - i), M = p.v.M;
    const size_t lrow = LF::row_bytes(p.v.stride);
    char *row = (char *)p.lev;
    for (int m = 0; m < M; ++m, row += lrow) {
        char *a = row + LF::off(i);
        if (FMT == UQ_FMT_I8) {
            for (int e = live; e < 8; ++e) a[e] = 0;
        } else if (FMT == UQ_FMT_I2X4) {
            *(uint16_t *)a &= (uint16_t)((1u << (2 * live)) - 1u);
        } else {
            *(uint32_t *)a &= (1u << (4 * live)) - 1u;
            if (FMT == UQ_FMT_I6P) *(uint16_t *)(row + LF::off2(i, p.v.stride)) &= (uint16_t)((1u << (2 * live)) - 1u);
        }
    }
    if (p.select) {
        const int ib = p.idx_bits;
        uint8_t *k = p.idx + ((i * ib) >> 3);
        if (ib == 8) for (int e = live; e < 8; ++e) k[e] = 0;
        else for (int b = 0; b < ib; ++b) k[b] &= (uint8_t)((1u << min(max(live * ib - b * 8, 0), 8)) - 1u);
    }
}

// ---------------------------------------------------------------------------------------------
// the straight-line path
// ---------------------------------------------------------------------------------------------

// The order in which a unit's levels sit in the bytes of its two level words: byte `b` of word `w` is
// coordinate coord(w, b).  Natural order, except for binary32 gradients and 4-bit levels, where the even
// coordinates in one word and the odd ones in the other let the nibbles merge with one shift.
template <int DT, int FMT> struct LevelOrder {
    static constexpr bool EO = DT == UQ_F32 && FMT == UQ_FMT_I4X2;
    static __host__ __device__ constexpr int coord(int w, int b) { return EO ? 2 * b + w : 4 * w + b; }
};

// Constants of the fast level arithmetic.
struct LevelConstants {
    float c0;                 // 16-bit draws: 1 - cap / 256
    uint32_t k_pos, k_neg;    // 16-bit draws: bias of the level bytes, and 128 + it, in every byte
    float cap23;              // 32-bit draws: cap * 2^23
};

// One worker's unit (q) turned into signed level bytes: w[k] holds four levels (see LevelOrder).
// 16-bit draws: the random words come complemented; with h' = 2^16 - 1 - h the carry out of
// rint(p * 2^16) + h' is the rounding decision, and one dp2a picks the half word and adds it.
// 32-bit draws: half an instruction per coordinate less with the products taken in pairs (8 workers, 25.6 M
// coordinates, binary32: 238 -> 230.6 us; 13.1 M bf16: 97.2 -> 95.1 us).
template <int DT, int FMT, int RNG>
__device__ __forceinline__ void quantize_fast(const uint4 *q, const float (&inv)[8], const LevelConstants &lc, const uint4 *r,
                                              uint32_t (&w)[2])
{
    using E = Elem<DT>;
    using O = LevelOrder<DT, FMT>;
    float v[8], x[8];
#pragma unroll
    for (int h = 0; h < 8 / E::G; ++h) E::unpack(q[h], *(float(*)[E::G])(v + h * E::G));
    if (RNG == 32) {
#pragma unroll
        for (int e = 0; e < 8; e += 2) mul_pair(v[e], v[e + 1], inv[e], inv[e + 1], x[e], x[e + 1]);
    }
    uint32_t z[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) {
        if (RNG == 16) {
            const uint4 b = r[0];
            const uint32_t word = (e >> 1) == 0 ? b.x : (e >> 1) == 1 ? b.y : (e >> 1) == 2 ? b.z : b.w;
            z[e] = __dp2a_lo(word, (e & 1) ? 0x100u : 0x1u, __float_as_uint(add_sat(mul_sat(fabsf(v[e]), inv[e]), lc.c0)));
        } else {
            const uint4 b = r[e >> 2];
            const uint32_t word = (e & 3) == 0 ? b.x : (e & 3) == 1 ? b.y : (e & 3) == 2 ? b.z : b.w;
            z[e] = level_draw23_fixed(x[e], lc.cap23, word);
        }
    }
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const int a = O::coord(k, 0), b = O::coord(k, 1), c = O::coord(k, 2), d = O::coord(k, 3);
        uint32_t neg;
        if (DT == UQ_F32) neg = sign_bytes_f32(v[a], v[b], v[c], v[d]);
        else neg = k == 0 ? sign_bytes_bf16(q[0].x, q[0].y) : sign_bytes_bf16(q[0].z, q[0].w);
        if (RNG == 16) {
            // byte B = L + bias (bias = 128 - cap): L = B - bias, and 128 - L = (128 + bias) - B, neither of
            // which borrows from the next byte; flipping its top bit makes the latter -L
            const uint32_t B = gather_bytes<2>(z[a], z[b], z[c], z[d]);
            const uint32_t plus = B - lc.k_pos, minus = lc.k_neg - B;
            w[k] = ((plus & ~neg) | (minus & neg)) ^ (neg & 0x80808080u);
        } else {
            w[k] = negated_bytes_to_signed(gather_bytes<kLevelByte23Fixed>(z[a], z[b], z[c], z[d]), neg);
        }
    }
}

// SEL without staging: a row's first read asks the caches to keep the line for the second one, which lets it
// go (binary32, 8 workers, 4 scales, 25.6 M coordinates: 285 us with the hints on L1 and L2, 290 us without,
// as a burst; 295 and 320 us sustained).
__device__ __forceinline__ uint64_t policy_keep()
{
    uint64_t p;
    asm("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(p));
    return p;
}
__device__ __forceinline__ uint64_t policy_drop()
{
    uint64_t p;
    asm("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
    return p;
}
__device__ __forceinline__ uint4 ld_keep(const void *p, uint64_t policy)
{
    uint4 v;
    asm volatile("ld.global.nc.L1::evict_last.L2::cache_hint.v4.u32 {%0,%1,%2,%3}, [%4], %5;"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p), "l"(policy));
    return v;
}
__device__ __forceinline__ uint4 ld_drop(const void *p, uint64_t policy)
{
    uint4 v;
    asm volatile("ld.global.nc.L1::no_allocate.L2::cache_hint.v4.u32 {%0,%1,%2,%3}, [%4], %5;"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p), "l"(policy));
    return v;
}

__device__ __forceinline__ uint4 ld_shared16(uint32_t a)
{
    uint4 v;
    asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a) : "memory");
    return v;
}

// WK: 8, with bf16 also 1 to 4, with binary32 2 and 4 = exactly that many workers (known at compile time), 0 = any number.
template <int DT, int FMT, int RNG, bool MULTI, bool SEL, bool DEC, int WK>
__global__ void __launch_bounds__(kThreads, (EncodeShape<DT, RNG, SEL, WK>::CTAS))
encode_kernel(const __grid_constant__ EncodeParams p)
{
    grid_dependency_prologue();
    using E = Elem<DT>;
    using S = EncodeShape<DT, RNG, SEL, WK>;
    using LF = LevelFmt<FMT>;
    using O = LevelOrder<DT, FMT>;
    constexpr int V = S::V, NB = S::NB, G = S::G, BSH = RNG == 32 ? 2 : 3;
    constexpr bool STAGED = SEL && DT == UQ_BF16 && WK > 0;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, M = WK ? WK : p.v.M, ib = p.idx_bits;
    const int64_t d = p.v.d;
    // CTAs walk the tiles back to front: the kernel before this one in a step (the norms) ends on the
    // high tiles, so part of what is read first is still in L2
    const int64_t t0 = (int64_t)(gridDim.x - 1 - blockIdx.x) * S::TILE;
    // my warp's row and my coordinates.  In the row that d ends in, the lanes beyond d do what the last one before it does,
    // down to the bytes that they store: such a row runs as the others do.  Only in a step of binary32 gradients whose number
    // of workers is known: with a loop around the workers the kernels have no register left for it (16 workers of 67 M
    // coordinates 1.2 % slower), and 8 bf16 workers of 335 M coordinates or levels alone lose 0.7 % by it.
    constexpr bool RAGGED = DT == UQ_F32 && DEC && WK > 0;
    // Where the callee's registers cost the rows without boundaries more than the lanes give the others, rows with
    // boundaries walk.  From the lanes / walking, us: levels alone, 16 workers of 5 715 coordinates 10.3 / 10.0; a step of 32
    // workers of 131 355 25.8 / 25.3, of 3 workers of 2 465 in 161 layers 47.3 / 46.3; levels alone inside a training step, 8
    // workers of 1.1 M 28.5 / 27.8.  With selection the lanes win: 12 workers of 172 032 in 161 layers 28.5 / 29.8.
    constexpr bool LANES = DT == UQ_BF16 || SEL || RAGGED;
    const int64_t r0 = t0 + warp * 256, i = RAGGED ? min(r0 + lane * 8, (d - 1) & ~(int64_t)7) : r0 + lane * 8;
    const uint64_t blk0 = (uint64_t)(p.coord0 + r0) >> BSH;
    if (r0 >= d) return;
    bool slow = (!RAGGED && r0 + 256 > d) || (uint32_t)(blk0 >> 32) != p.blk_hi || (uint32_t)blk0 > 0xFFFFFFFFu - (256u >> BSH);
    const size_t grow = (size_t)p.v.stride * E::BYTES, lrow = LF::row_bytes(p.v.stride);
    // my workers: all of them, or (only the levels wanted) one of grid.y groups
    constexpr bool SPLIT = !WK && !SEL && !DEC;
    const int m_first = SPLIT ? blockIdx.y * p.split : 0, m_last = SPLIT ? min(m_first + p.split, M) : M;
    const char *gp = (const char *)p.v.g + (size_t)i * E::BYTES + (SPLIT ? m_first * grow : 0);
    extern __shared__ uint4 stage[];                             // STAGED: [worker][thread]
    const uint32_t sp = (uint32_t)__cvta_generic_to_shared(stage) + threadIdx.x * 16;
    uint64_t policy = 0;
    uint4 q[G][V];
    uint32_t kw[2] = {0u, 0u};
    auto load = [&](int m, uint4 (&x)[V]) {                      // worker m's bytes (called for m = 0, 1, 2, ...)
        if (STAGED) {
            x[0] = ld_shared16(sp + m * (kThreads * 16));
            return;
        }
#pragma unroll
        for (int h = 0; h < V; ++h) x[h] = SEL ? ld_drop(gp + h * 16, policy) : ld_stream(gp + h * 16);
        gp += grow;
    };
    if (!slow) {
        // the first rows and the shared indices are on their way during the set-up below
        if (STAGED) {
            // every thread copies what it reads back itself
            const char *gs = gp;
#pragma unroll
            for (int m = 0; m < WK; ++m, gs += grow) copy_async16(sp + m * (kThreads * 16), gs);
        } else if (!SEL) {
#pragma unroll
            for (int c = 0; c < G; ++c)
                if (WK || m_first + c < m_last) load(c, q[c]);
            if (MULTI) load_indices(p.idx, i, ib, kw);
        }
    }
    const int j = warp_find_segment(p.v.seg_off, p.v.nseg, r0);
    const bool mixed = segment_end(p.v.seg_off, p.v.nseg, j, d) < (RAGGED ? min(r0 + 256, d) : r0 + 256);          // a boundary inside my row
    const int kmask = !MULTI ? 0 : ib < 4 ? (1 << ib) - 1 : UQ_MAX_SCALES - 1;      // lane L holds scale L & kmask
    const float W = __ldg(p.v.W + j);
    float inv_lane = inv_scale(p.v.scales.s[lane & kmask], W);
    if (!mixed && !slow) {
        if (lane < p.v.scales.N && not_finite(inv_lane) && p.status) atomicOr(p.status, (uint32_t)UQ_STATUS_SCALE_OVERFLOW);
        // a W so large (16-bit draws) or so small (32-bit) that the rescaled factors of the fast forms would leave
        // the normal range: the plain arithmetic
        const float edge = MULTI ? __shfl_sync(0xFFFFFFFFu, inv_lane, RNG == 16 ? 0 : p.v.scales.N - 1) : inv_lane;
        slow = RNG == 16 ? !sat_form_exact(edge) : !fixed_form_exact(edge);
    }
    float inv[8];
    if (SEL && !slow) {
        // Scale selection and sharing (Algorithm 2 lines "Compute coordinate scales" and "Scale sharing"): the
        // largest magnitude over the workers decides the shared index (see uq_select.cuh), found by bisection
        // over the pass thresholds that lanes 0 .. N-1 hold.
        const int top = p.v.scales.N > 1 ? 1 << (31 - __clz(p.v.scales.N - 1)) : 0;   // first step of the bisection
        const int32_t thr = lane < p.v.scales.N ? pass_threshold(inv_lane, p.v.s_hat) : -1;
        const int32_t thr_top = __shfl_sync(0xFFFFFFFFu, thr, top);
        if (STAGED) copy_async_wait();
        else policy = policy_keep();
        uint32_t amag[8];
        const char *gs = gp;
        if (DT == UQ_F32) {
            float a[8] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
            auto four = [&](int left) {                               // four workers' loads in flight
                uint4 x[4][V];
#pragma unroll
                for (int k = 0; k < 4; ++k) {
#pragma unroll
                    for (int h = 0; h < V; ++h) x[k][h] = (WK ? k < WK : k < left) ? ld_keep(gs + h * 16, policy) : make_uint4(0u, 0u, 0u, 0u);
                    gs += grow;
                }
#pragma unroll
                for (int k = 0; k < 4; ++k)
#pragma unroll
                    for (int h = 0; h < V; ++h) {
                        a[4 * h + 0] = fmaxf(a[4 * h + 0], fabsf(__uint_as_float(x[k][h].x)));
                        a[4 * h + 1] = fmaxf(a[4 * h + 1], fabsf(__uint_as_float(x[k][h].y)));
                        a[4 * h + 2] = fmaxf(a[4 * h + 2], fabsf(__uint_as_float(x[k][h].z)));
                        a[4 * h + 3] = fmaxf(a[4 * h + 3], fabsf(__uint_as_float(x[k][h].w)));
                    }
            };
            if (WK == kGroup) { four(4); four(4); }
            else if (WK) four(WK);
            else {
#pragma unroll 1
                for (int m = 0; m < M; m += 4) four(M - m);
            }
#pragma unroll
            for (int e = 0; e < 8; ++e) amag[e] = __float_as_uint(a[e]);
        } else {
            // bf16 halves read as signed 16-bit integers order the positive values, as unsigned ones the
            // negative values above all others: max |x| = max(smax & 0x7FFF, umax & 0x7FFF)
            uint32_t smax[4] = {0u, 0u, 0u, 0u}, umax[4] = {0u, 0u, 0u, 0u};
            auto eight = [&](int left) {                              // eight workers' loads in flight
                uint4 x[8];
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    x[k] = STAGED && k < WK ? ld_shared16(sp + k * (kThreads * 16)) : !STAGED && k < left ? ld_keep(gs, policy) : make_uint4(0u, 0u, 0u, 0u);
                    gs += grow;
                }
#pragma unroll
                for (int k = 0; k < 8; k += 2) {
                    smax[0] = __vimax3_s16x2(smax[0], x[k].x, x[k + 1].x); umax[0] = __vimax3_u16x2(umax[0], x[k].x, x[k + 1].x);
                    smax[1] = __vimax3_s16x2(smax[1], x[k].y, x[k + 1].y); umax[1] = __vimax3_u16x2(umax[1], x[k].y, x[k + 1].y);
                    smax[2] = __vimax3_s16x2(smax[2], x[k].z, x[k + 1].z); umax[2] = __vimax3_u16x2(umax[2], x[k].z, x[k + 1].z);
                    smax[3] = __vimax3_s16x2(smax[3], x[k].w, x[k + 1].w); umax[3] = __vimax3_u16x2(umax[3], x[k].w, x[k + 1].w);
                }
            };
            if (WK) eight(8);
            else {
#pragma unroll 1
                for (int m = 0; m < M; m += 8) eight(M - m);
            }
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const uint32_t am = __vmaxu2(smax[c] & 0x7FFF7FFFu, umax[c] & 0x7FFF7FFFu);
                amag[2 * c] = am << 16; amag[2 * c + 1] = am & 0xFFFF0000u;
            }
        }
        if (!mixed) {
            int k[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) k[e] = (top != 0 && (int32_t)amag[e] <= thr_top) ? top : 0;
#pragma unroll 1
            for (int step = top >> 1; step >= 1; step >>= 1) {
#pragma unroll
                for (int e = 0; e < 8; ++e)
                    if ((int32_t)amag[e] <= __shfl_sync(0xFFFFFFFFu, thr, k[e] + step)) k[e] += step;
            }
            const float f = __fmul_rn(inv_lane, RNG == 16 ? 0.00390625f : 8388608.0f);
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                kw[e >> 2] |= (uint32_t)k[e] << ((e & 3) * ib);
                inv[e] = __shfl_sync(0xFFFFFFFFu, f, k[e]);
            }
        } else {
            kw[0] = mixed_row_select(p, i, j, amag[0], amag[1], amag[2], amag[3]);
            kw[1] = mixed_row_select(p, i + 4, j, amag[4], amag[5], amag[6], amag[7]);
            __syncwarp();
        }
        store_indices(p.idx, i, ib, kw);
        if (!STAGED) policy = policy_drop();
#pragma unroll
        for (int c = 0; c < G; ++c)
            if (WK || c < M) load(c, q[c]);
    }

    // the factors of my coordinates.  The shuffle reads its source lane modulo 32 and the table repeats every
    // 2^ib lanes: the index needs no mask
    if (!mixed && SEL && !slow) {
        // known from the selection
    } else if (!mixed) {
        inv_lane = __fmul_rn(inv_lane, RNG == 16 ? 0.00390625f : 8388608.0f);
#pragma unroll
        for (int e = 0; e < 8; ++e)
            inv[e] = MULTI ? __shfl_sync(0xFFFFFFFFu, inv_lane, (int)(kw[e >> 2] >> ((e & 3) * ib))) : inv_lane;
    } else if (!slow) {
        bool inexact = false;
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const float4 f = mixed_row_factors<LANES>(p, i + 4 * k, j, kw[k], false);
            const float g[4] = {f.x, f.y, f.z, f.w};
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                inexact |= RNG == 16 ? !sat_form_exact(g[e]) : !fixed_form_exact(g[e]);
                inv[4 * k + e] = __fmul_rn(g[e], RNG == 16 ? 0.00390625f : 8388608.0f);
            }
        }
        slow = __any_sync(0xFFFFFFFFu, inexact);
    }
    if (slow) {
        if (STAGED) copy_async_wait();                           // copies may be on their way: W came after them
        encode_row_slow<DT, FMT, RNG, MULTI>(p, r0, m_first, m_last);
        return;
    }
    LevelConstants lc;
    lc.c0 = __fsub_rn(1.0f, __fmul_rn(p.v.s_hat, 0.00390625f));
    lc.k_pos = (128u - (uint32_t)p.v.s_hat) * 0x01010101u;
    lc.k_neg = (256u - (uint32_t)p.v.s_hat) * 0x01010101u;
    lc.cap23 = __fmul_rn(p.v.s_hat, 8388608.0f);
    PhiloxBlockPart blk[NB];
#pragma unroll
    for (int b = 0; b < NB; ++b)
        blk[b] = philox_block_part(p.key, RAGGED ? (uint32_t)((uint64_t)(p.coord0 + i) >> BSH) + (uint32_t)b
                                                 : (uint32_t)blk0 + (uint32_t)(lane * NB + b));

    // The workers, straight-line.  The sums of two levels share a word: dp2a adds byte 0 and 2^14 times byte 1
    // (64 workers * 127 < 2^13, so the fields come apart again).
    int sum[2][2] = {{0, 0}, {0, 0}};
    char *lp = (char *)p.lev + LF::off(i) + (SPLIT ? m_first * lrow : 0), *lp2 = lp + (LF::off2(i, p.v.stride) - LF::off(i));
    // workers m0 .. m0 + GG - 1; ahead: the worker GG places on, if there is one, is fetched into the registers that become free
    auto group = [&](auto gg_tag, int m0, auto ahead) {
        constexpr int GG = decltype(gg_tag)::value;
        uint4 r[GG][NB];
        philox_join<GG, NB>(p.key, blk, p.wpart + m0, r);
#pragma unroll
        for (int c = 0; c < GG; ++c) {
            if (RNG == 16) { r[c][0].y = ~r[c][0].y; r[c][0].w = ~r[c][0].w; }
            uint32_t w[2];
            quantize_fast<DT, FMT, RNG>(q[c], inv, lc, r[c], w);
            if (ahead(m0 + c + GG)) load(m0 + c + GG, q[c]);
            if (O::EO) store_unit_even_odd(w[0], w[1], lp);
            else store_unit<FMT>(w[0], w[1], lp, lp2);
            lp += lrow;
            if (FMT == UQ_FMT_I6P) lp2 += lrow;
            if (DEC) {
#pragma unroll
                for (int k = 0; k < 2; ++k) {
                    sum[k][0] = __dp2a_lo(0x40000001, (int)w[k], sum[k][0]);
                    sum[k][1] = __dp2a_hi(0x40000001, (int)w[k], sum[k][1]);
                }
            }
        }
    };
    if (WK) {
#pragma unroll
        for (int m = 0; m < WK; m += G) group(std::integral_constant<int, G>(), m, [](int m) { return m < WK; });
    } else {
        // Eight workers whose levels alone are wanted go straight-line; else whole groups, and the rest by twos and
        // one, so that a worker that is not there costs no draws.  (With groups of four chains for whoever is there: one
        // bf16 worker of 25.6 M coordinates, levels alone, 16-bit draws 53 us, 34 like this; five of them 1.2 times as long.
        // With a loop around the eight: 16 binary32 workers 3 % longer.)
        int m = m_first;
        if (SPLIT && m_last - m_first == kGroup) {
#pragma unroll
            for (int k = 0; k < kGroup; k += G) group(std::integral_constant<int, G>(), m_first + k, [&](int x) { return x < m_first + kGroup; });
            return;
        }
#pragma unroll 1
        for (; m + G <= m_last; m += G) group(std::integral_constant<int, G>(), m, [&](int m) { return m < m_last; });
        const auto never = [](int) { return false; };
        if (G > 2 && ((m_last - m) & 2)) {
            group(std::integral_constant<int, (G > 2 ? 2 : 1)>(), m, never);
            m += 2;
#pragma unroll
            for (int h = 0; h < V; ++h) q[0][h] = q[G > 2 ? 2 : 0][h];
        }
        if (G > 1 && m < m_last) group(std::integral_constant<int, 1>(), m, never);
    }
    if (DEC) {
        // Algorithm 1 / 2, lines "AllReduce gradients" and "Reconstruct gradient": the sum of a coordinate times
        // the factor of its scale (the same operations as the aggregation kernel's)
        float c[8];
        if (!mixed) {
            const float c_lane = decode_factor(W, p.v.scales.s[lane & kmask], M);
#pragma unroll
            for (int e = 0; e < 8; ++e)
                c[e] = MULTI ? __shfl_sync(0xFFFFFFFFu, c_lane, (int)(kw[e >> 2] >> ((e & 3) * ib))) : c_lane;
        } else {
            const float4 a = mixed_row_factors<LANES>(p, i, j, kw[0], true), b = mixed_row_factors<LANES>(p, i + 4, j, kw[1], true);
            c[0] = a.x; c[1] = a.y; c[2] = a.z; c[3] = a.w; c[4] = b.x; c[5] = b.y; c[6] = b.z; c[7] = b.w;
        }
        uint32_t s[8], r[8];
#pragma unroll
        for (int k = 0; k < 2; ++k)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int hi = (sum[k][h] + 0x2000) >> 14;
                s[O::coord(k, 2 * h + 1)] = (uint32_t)hi;
                s[O::coord(k, 2 * h)] = (uint32_t)(sum[k][h] - (hi << 14));
            }
#pragma unroll
        for (int e = 0; e < 8; ++e) r[e] = __float_as_uint(__fmul_rn((float)(int)s[e], c[e]));
        if (RAGGED) __syncwarp();                                 // what the lanes of the last unit store comes before its correction
        if (RAGGED && i + 8 > p.v.d) {                           // d ends in my unit: the first of its lanes does the rest
            if (((int)i & 255) >> 3 != (threadIdx.x & 31)) return;
            __shared__ uint32_t part[16];
#pragma unroll
            for (int e = 0; e < 8; ++e) { part[e] = r[e]; part[8 + e] = s[e]; }
            for (int e = 0; i + e < p.v.d; ++e) {
                p.out[i + e] = __uint_as_float(part[e]);
                if (p.S != nullptr) p.S[i + e] = (int32_t)part[8 + e];
            }
            clear_padding<FMT>(p, i);
            return;
        }
        st_stream256(p.out + i, r);
        if (p.S != nullptr) st_stream256(p.S + i, s);
    }
}

template <int DT, int FMT, int RNG, bool MULTI, bool SEL, bool DEC, int WK>
static cudaError_t launch(EncodeParams p, cudaStream_t st)
{
    using S = EncodeShape<DT, RNG, SEL, WK>;
    const int64_t blocks = (p.v.d + S::TILE - 1) / S::TILE;
    if (blocks == 0) return cudaSuccess;
    if (blocks > 0x7FFFFFFFLL) return cudaErrorInvalidConfiguration;
    constexpr int BSH = RNG == 32 ? 2 : 3;
    p.blk_hi = (uint32_t)((uint64_t)(p.coord0 >> BSH) >> 32);
    if (RNG == 16) { p.key.k[18] = ~p.key.k[18]; p.key.k[19] = ~p.key.k[19]; }
    for (int m = 0; m < p.v.M; ++m) p.wpart[m] = philox_worker_part(p.key, p.blk_hi, (uint32_t)(p.worker0 + m));
    // bf16, selecting: the workers' rows of the tile, where their number is known
    const size_t smem = SEL && DT == UQ_BF16 && WK > 0 ? (size_t)WK * S::TILE * Elem<DT>::BYTES : 0;
    // only the levels wanted: groups of 8 workers are independent, which gives small gradients of many workers
    // as many warps as they have groups
    p.split = !WK && !SEL && !DEC ? kGroup : p.v.M;
    const dim3 grid((unsigned)blocks, (unsigned)((p.v.M + p.split - 1) / p.split));
    launch_k_smem(encode_kernel<DT, FMT, RNG, MULTI, SEL, DEC, WK>, grid, kThreads, smem, st, p);
    return cudaGetLastError();
}

// All wire formats and modes of one element type and draw width (one translation unit each, so that
// the variants build in parallel).
template <int DT, int FMT, int RNG, int WK> static cudaError_t dispatch_mode(const EncodeParams &p, cudaStream_t st)
{
    const bool dec = p.out != nullptr;
    if (p.idx_bits == 0)
        return dec ? launch<DT, FMT, RNG, false, false, true, WK>(p, st) : launch<DT, FMT, RNG, false, false, false, WK>(p, st);
    if (p.select)
        return dec ? launch<DT, FMT, RNG, true, true, true, WK>(p, st) : launch<DT, FMT, RNG, true, true, false, WK>(p, st);
    return dec ? launch<DT, FMT, RNG, true, false, true, WK>(p, st) : launch<DT, FMT, RNG, true, false, false, WK>(p, st);
}

template <int DT, int FMT, int RNG> static cudaError_t dispatch_workers(const EncodeParams &p, cudaStream_t st)
{
    if constexpr (DT == UQ_BF16) {
        if (p.v.M == 1) return dispatch_mode<DT, FMT, RNG, 1>(p, st);
        if (p.v.M == 2) return dispatch_mode<DT, FMT, RNG, 2>(p, st);
        if (p.v.M == 3) return dispatch_mode<DT, FMT, RNG, 3>(p, st);
        if (p.v.M == 4) return dispatch_mode<DT, FMT, RNG, 4>(p, st);
    } else {
        // 2 workers, one scale, 32-bit draws, with the average: the general kernel is behind up to some 12 M coordinates (the
        // row that d ends in) and ahead beyond.  Steps, general / own, us, int8 levels: 4 M 20.9 / 20.8, 8.4 M 36.9 / 37.5,
        // 16 M 68.8 / 70.8, 60 M 241 / 249; 6-bit levels: 8.4 M 38.5 / 37.3, 16 M 70.4 / 71.2, 60 M 250.4 / 252.4.
        const bool general = RNG == 32 && p.idx_bits == 0 && p.out != nullptr && p.v.d > 12000000;
        if (p.v.M == 2 && !general) return dispatch_mode<DT, FMT, RNG, 2>(p, st);
        if (p.v.M == 4) return dispatch_mode<DT, FMT, RNG, 4>(p, st);
    }
    return p.v.M == kGroup ? dispatch_mode<DT, FMT, RNG, kGroup>(p, st) : dispatch_mode<DT, FMT, RNG, 0>(p, st);
}

template <int DT, int RNG> static cudaError_t dispatch_fmt(const EncodeParams &p, int fmt, cudaStream_t st)
{
    if (fmt == UQ_FMT_I8) return dispatch_workers<DT, UQ_FMT_I8, RNG>(p, st);
    if (fmt == UQ_FMT_I4X2) return dispatch_workers<DT, UQ_FMT_I4X2, RNG>(p, st);
    if (fmt == UQ_FMT_I2X4) return dispatch_workers<DT, UQ_FMT_I2X4, RNG>(p, st);
    return dispatch_workers<DT, UQ_FMT_I6P, RNG>(p, st);
}

cudaError_t launch_encode_f32_r16(const EncodeParams &p, int fmt, cudaStream_t st);
cudaError_t launch_encode_f32_r32(const EncodeParams &p, int fmt, cudaStream_t st);
cudaError_t launch_encode_bf16_r16(const EncodeParams &p, int fmt, cudaStream_t st);
cudaError_t launch_encode_bf16_r32(const EncodeParams &p, int fmt, cudaStream_t st);

}  // namespace uq
