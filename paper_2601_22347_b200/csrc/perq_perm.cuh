// Permuted rows, Hadamard blocks of 16 .. 128, MXFP4 or INT4 per 128, many rows: eight token rows at a time.
//
// The kernels that take a permuted row by itself gather it with one 2-byte load per element: 32 random banks, 3.5 wavefronts
// a load, 112 per 1024 elements of the 194 that a segment costs in all, and a hundred instructions.  Here the eight rows of
// a set are first interleaved in shared memory, a channel's eight values in 16 adjacent bytes.  ldmatrix takes a row address
// from every lane, so that one instruction then gathers 32 channels of eight rows; its transposed form hands a lane pairs of
// adjacent positions of one row, which is the operand of mma.sync as it stands.  1024 elements: 32 wavefronts to interleave, about
// 41 (eight random bank groups, 2.6 to a phase) and four instructions to gather, nothing to write back.
//
// A unit is 128 positions of the eight rows.  As in perq_fast.cuh a quad of lanes holds 128 adjacent outputs, a lane four of each of
// the eight chunks of 16, only that the eight quads have the same positions of different rows.  So all that a range or an MX group
// needs is in its quad: the inputs too (the operand's registers), from which exact sums are formed for all eight rows at once.
//
// A CTA per SM, 16 warps.  A set: the rows come in TMA boxes of eight rows by 512 channels (128-byte swizzle), a stage of the ring to a
// warp, which interleaves a box and loads the next one into its place; a barrier; units of 128 positions in turn; a barrier.
//
// What bounds it: 325 (MXFP4, b = 32) to 617 (per 128, b = 128) instructions and 100 wavefronts a segment of 1024 at 31 to 45 % of the issue slots, and
// the time in which rows are interleaved, 64 wavefronts for 512 channels each way, by warps that then wait for each other (barriers are its
// largest stall).  8192 x 9728, permuted, MXFP4, b = 32: 82 us (row kernel 176), INT4 per 128, b = 128: 106 (282).
//
// Exactness rules as in perq_fast.cuh, whose arithmetic this is: one tensor-core step for a chunk of 16, then fp32 stages over the C
// chunks of a block.  What they lose, in 2^-24 of the block's largest output M: a step loses 7.5 T + 2 P (perq_tile.cuh; measured here
// too: mma.sync gives the bits of that model), T the chunk's largest input, P its output.  Over the chunks both sum to sqrt(C) M
// at most (Cauchy; Parseval: M is at least the 2-norm of the inputs, and of the chunks' outputs that meet in one).  The stages round to
// nearest: sqrt(C/2) + sqrt(C/4) + .. + 1.  In all 9.5, 14.4, 21.4 and 31.3 for b = 16, 32, 64, 128 (perm_err; the worst rows found lose 17).
// The model of perq_fast.cuh is 16, 20, 24 and 28, of which MXFP4 takes twice.
#pragma once
#include <cuda.h>

#include "perq_tile.cuh"

namespace perq {

constexpr int PERM_WARPS = 16;
constexpr int PERM_THREADS = PERM_WARPS * 32;
constexpr int PERM_ROWS = 8;                  // token rows of a set
constexpr int PERM_BOX = 512;                 // channels of a TMA box
constexpr uint32_t PERM_STAGE = PERM_ROWS * PERM_BOX * 2;
constexpr int PERM_MAX_STAGES = 12;

struct PermParams {
    const int32_t *perm;
    uint8_t *out_codes;
    void *out_scales;
    uint32_t T, sets;
    int d, units;            // units of 128 positions in a row
    int boxes;               // per set
    int parts;               // CTAs to a set of the last round
    int stages;
    uint32_t off_ring, off_tab, off_bars;
    double sqrt_b, inv_7_sqrt_b;
};

// Interleaved rows first (16 bytes a channel), then the ring, the permutation, barriers.  The permutation's channels lie in the
// order in which a lane needs them: unit, lane, four of 16 bits (positions lane, lane + 32, ...).
struct PermLayout {
    uint32_t ring, tab, bars, total;
    int stages;
    __host__ __device__ PermLayout(int d, int boxes, uint32_t limit)
    {
        ring = (uint32_t)d * 16u;
        const uint32_t rest = (uint32_t)d * 2u + PERM_MAX_STAGES * 8u + 1024u;
        stages = limit > ring + rest ? (int)((limit - ring - rest) / PERM_STAGE) : 0;
        stages = stages > PERM_MAX_STAGES ? PERM_MAX_STAGES : stages;
        stages = stages > 2 * boxes ? 2 * boxes : stages;
        tab = ring + (uint32_t)stages * PERM_STAGE;
        bars = tab + (uint32_t)d * 2u;
        total = bars + PERM_MAX_STAGES * 8u + 1024u;
    }
};

__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap *map, int x, int y, int z, uint32_t bar)
{
    asm volatile("cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
                 ::"r"(dst), "l"(map), "r"(x), "r"(y), "r"(z), "r"(bar) : "memory");
}
__device__ __forceinline__ void tma_prefetch_3d(const CUtensorMap *map, int x, int y, int z)
{
    asm volatile("cp.async.bulk.prefetch.tensor.3d.L2.global.tile [%0, {%1, %2, %3}];" ::"l"(map), "r"(x), "r"(y), "r"(z) : "memory");
}
__device__ __forceinline__ void ldmatrix_x4_trans(uint32_t (&r)[4], uint32_t addr)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void stmatrix_x4(uint32_t addr, const uint32_t (&r)[4])
{
    asm volatile("stmatrix.sync.aligned.m8n8.x4.shared.b16 [%0], {%1,%2,%3,%4};" ::"r"(addr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]) : "memory");
}

// Place of a unit's position in the table: the lane that gathers it (eight lanes for eight positions; the first halves of two chunks come
// before the second ones, the order of the operand's registers), and which of its four.
__device__ __forceinline__ int perm_entry(int k) { return ((k & 7) | (k & 16) >> 1 | (k & 8) << 1) * 4 + (k >> 5); }
// The operand of a unit: x[4 t + r] holds of chunk 2 t + r % 2 of row lane / 4 the positions 2 q, 2 q + 1 (r < 2) or eight further on.
// rows: the interleaved rows, at: the lane's four channels.
__device__ __forceinline__ void perm_gather(uint32_t rows, uint2 at, uint32_t (&x)[16])
{
    const uint32_t c[4] = {at.x & 0xffffu, at.x >> 16, at.y & 0xffffu, at.y >> 16};
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        uint32_t r[4];
        ldmatrix_x4_trans(r, rows + c[j] * 16u);
        x[4 * j] = r[0]; x[4 * j + 1] = r[1]; x[4 * j + 2] = r[2]; x[4 * j + 3] = r[3];
    }
}
// Error bound of an fp32 output, relative to the largest of its block.
__host__ __device__ constexpr float perm_err(int log2b, bool ranges) { return (ranges && log2b == 7 ? 32.0f : 4.0f * log2b) * 0x1p-24f; }
// Rounding window of E2M1 codes in scaled units: ref the largest magnitude of the element's block, m the multiplier.  Twice the model's error
// in blocks of 64 and 128.  Blocks up to 32: once, and the scaled values are below 8: one window for all groups.
template <int LOG2B>
__device__ __forceinline__ float perm_window(float err, float ref, float m) { return LOG2B <= 5 ? 8.01f * err + 2.0e-6f : 2.0f * err * ref * m + 2.0e-6f; }
// Columns of H_16 for a lane's four adjacent outputs: column n of contraction m is output 4 (n / 2) + n % 2 + 2 m.
__device__ __forceinline__ void perm_operand(uint32_t (&hb)[2][2], int lane)
{
    const int g = lane >> 2, q = lane & 3;
#pragma unroll
    for (int m = 0; m < 2; ++m) {
        const int col = 4 * (g >> 1) + (g & 1) + 2 * m;
        hb[m][0] = hadamard_bf16(2 * q, col) | (hadamard_bf16(2 * q + 1, col) << 16);
        hb[m][1] = hadamard_bf16(2 * q + 8, col) | (hadamard_bf16(2 * q + 9, col) << 16);
    }
}
// v[c][h]: outputs 16 c + 4 q + 2 h and one more of the quad's row, unnormalised.
template <int LOG2B>
__device__ __forceinline__ void perm_rotate(const uint32_t (&x)[16], const uint32_t (&hb)[2][2], f32x2 (&v)[8][2])
{
#pragma unroll
    for (int t = 0; t < 4; ++t) {
        const uint32_t a[4] = {x[4 * t], x[4 * t + 1], x[4 * t + 2], x[4 * t + 3]};       // chunk 2 t in the first eight rows
        float c0[4], c1[4];
        mma_bf16(c0, a, hb[0][0], hb[0][1]);
        mma_bf16(c1, a, hb[1][0], hb[1][1]);
        v[2 * t][0] = pack2(c0[0], c0[1]);
        v[2 * t][1] = pack2(c1[0], c1[1]);
        v[2 * t + 1][0] = pack2(c0[2], c0[3]);
        v[2 * t + 1][1] = pack2(c1[2], c1[3]);
    }
#pragma unroll
    for (int t = 0; t < LOG2B - 4; ++t) {
#pragma unroll
        for (int c = 0; c < 8; ++c) {
            if ((c & (1 << t)) == 0) {
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const f32x2 a = v[c][h], b = v[c | (1 << t)][h];
                    v[c][h] = add2(a, b);
                    v[c | (1 << t)][h] = sub2(a, b);
                }
            }
        }
    }
}
__device__ __forceinline__ float perm_max4(const f32x2 (&w)[2]) { return fmaxf(max3abs(fabsf(w[0].x), w[0].y, w[1].x), fabsf(w[1].y)); }
__device__ __forceinline__ float perm_quad_max(float a)
{
    a = fmaxf(a, __shfl_xor_sync(0xffffffffu, a, 1));
    return fmaxf(a, __shfl_xor_sync(0xffffffffu, a, 2));
}

// Selections by the lane's place in its quad as byte permutations (a register each, where predicates would be formed again and again).
struct PermSelect {
    uint32_t keep2, give2, keep1, give1;      // by bit 1 and bit 0 of lane % 4: the first or the second word, and the other one
    __device__ __forceinline__ explicit PermSelect(int q)
    {
        keep2 = (q & 2) ? 0x7654u : 0x3210u;
        keep1 = (q & 1) ? 0x7654u : 0x3210u;
        // (volatile: as for the thread's number)
        asm volatile("xor.b32 %0, %1, 0x4444;" : "=r"(give2) : "r"(keep2));
        asm volatile("xor.b32 %0, %1, 0x4444;" : "=r"(give1) : "r"(keep1));
        asm volatile("mov.b32 %0, %0;" : "+r"(keep2));
        asm volatile("mov.b32 %0, %0;" : "+r"(keep1));
    }
    __device__ __forceinline__ float pick(uint32_t sel, float a, float b) const { return __uint_as_float(__byte_perm(__float_as_uint(a), __float_as_uint(b), sel)); }
};
// As quad_codes, from words of two slots.
__device__ __forceinline__ uint4 perm_quad_words(const uint32_t (&w)[4], const PermSelect &S)
{
    // kept and received: of the lane's own half of the words, then of its own word
    const uint32_t k0 = __byte_perm(w[0], w[2], S.keep2), k1 = __byte_perm(w[1], w[3], S.keep2);
    const uint32_t r0 = __shfl_xor_sync(0xffffffffu, __byte_perm(w[0], w[2], S.give2), 2), r1 = __shfl_xor_sync(0xffffffffu, __byte_perm(w[1], w[3], S.give2), 2);
    // (lower lanes first: what was kept by lanes 0 and 1, received by 2 and 3)
    const uint32_t l0 = __byte_perm(k0, r0, S.keep2), h0 = __byte_perm(k0, r0, S.give2), l1 = __byte_perm(k1, r1, S.keep2), h1 = __byte_perm(k1, r1, S.give2);
    const uint32_t kl = __byte_perm(l0, l1, S.keep1), kh = __byte_perm(h0, h1, S.keep1);
    const uint32_t rl = __shfl_xor_sync(0xffffffffu, __byte_perm(l0, l1, S.give1), 1), rh = __shfl_xor_sync(0xffffffffu, __byte_perm(h0, h1, S.give1), 1);
    const uint32_t t0 = __byte_perm(kl, rl, S.keep1), t1 = __byte_perm(kl, rl, S.give1), t2 = __byte_perm(kh, rh, S.keep1), t3 = __byte_perm(kh, rh, S.give1);
    return make_uint4(__byte_perm(t0, t1, 0x5410), __byte_perm(t2, t3, 0x5410), __byte_perm(t0, t1, 0x7632), __byte_perm(t2, t3, 0x7632));
}

// -------------------------------------------------------------------------------------------- exact values
//
// Every quad for its own row, from the operand's registers; all lanes of the warp call.  The functions that are not inlined gather
// and rotate again: had they taken the registers, these would stay alive through every unit.

// Sums for the four outputs of slot (chunk c, lane qs) of the quad's row: p and m are the sums of the outputs without and with bit 0
// over the inputs without (even lanes) or with (odd lanes) bit 1.
template <int LOG2B>
__device__ __forceinline__ void perm_slot(const uint32_t (&x)[16], int c, int qs, int q, double &p, double &m)
{
    constexpr int CB = LOG2B - 4, CH = 1 << CB;
    uint32_t y[2 * CH];                                       // the block's registers: chunk k, half h in y[2 k + h]
#pragma unroll
    for (int k = 0; k < CH; ++k) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            uint32_t w = x[4 * (k >> 1) + (k & 1) + 2 * h];
#pragma unroll
            for (int j = 1; j < 8 / CH; ++j) w = (c >> CB) == j ? x[4 * ((CH * j + k) >> 1) + ((CH * j + k) & 1) + 2 * h] : w;
            y[2 * k + h] = w;
        }
    }
    const uint32_t walsh = ((c & 1) ? 0xAAu : 0u) ^ ((c & 2) ? 0xCCu : 0u) ^ ((c & 4) ? 0xF0u : 0u);      // bit k: parity of c & k
    double S[2][2] = {{0.0, 0.0}, {0.0, 0.0}};               // by half of the chunk and parity of the position
#pragma unroll
    for (int k = 0; k < CH; ++k) {
        const double f = __hiloint2double((int)((walsh << (31 - k)) & 0x80000000u) | 0x77f00000, 0);             // +-2^896
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            S[h][0] = fma(bf16_raw_f64(y[2 * k + h] << 16), f, S[h][0]);
            S[h][1] = fma(bf16_raw_f64(y[2 * k + h]), f, S[h][1]);
        }
    }
    const double s3 = (qs & 2) ? -1.0 : 1.0, s2 = ((qs & 1) && (q & 2)) ? -1.0 : 1.0;        // position bits 3 and 2
    double a = s2 * fma(s3, S[1][0], S[0][0]), b = s2 * fma(s3, S[1][1], S[0][1]);
    a += __shfl_xor_sync(0xffffffffu, a, 2);
    b += __shfl_xor_sync(0xffffffffu, b, 2);
    p = a + b;
    m = a - b;
}
// Their largest magnitude, or output j (the same in all lanes of the quad).
__device__ __forceinline__ double perm_slot_max(double p, double m)
{
    const double P = __shfl_xor_sync(0xffffffffu, p, 1), M = __shfl_xor_sync(0xffffffffu, m, 1);
    return fmax(fabs(p) + fabs(P), fabs(m) + fabs(M));
}
__device__ __forceinline__ double perm_slot_output(double p, double m, int j, int q)
{
    const double P = __shfl_xor_sync(0xffffffffu, p, 1), M = __shfl_xor_sync(0xffffffffu, m, 1);
    const double own = (j & 1) ? m : p, other = (j & 1) ? M : P;
    const double lower = (q & 1) ? other : own, upper = (q & 1) ? own : other;
    return ((j & 2) ? lower - upper : lower + upper) + 0.0;   // (+0 for a sum of zeros of either sign)
}

// Whether the fp32 outputs of the quad's row are exact in this unit (see RowSpan).
__device__ __forceinline__ bool perm_row_exact(const uint32_t (&x)[16])
{
    RowSpan s = {0.0f, 1 << 20};
#pragma unroll
    for (int j = 0; j < 32; ++j) {
        const uint32_t a = (x[j >> 1] >> (16 * (j & 1))) & 0x7fffu;
        s.sum += __uint_as_float(a << 16);
        if (a != 0u) s.low = min(s.low, a < 0x80u ? __ffs(a) : (int)(a >> 7) + __ffs((a & 0x7fu) | 0x80u) - 1);
    }
#pragma unroll
    for (int o = 1; o <= 2; o <<= 1) {
        s.sum += __shfl_xor_sync(0xffffffffu, s.sum, o);
        s.low = min(s.low, __shfl_xor_sync(0xffffffffu, s.low, o));
    }
    return row_span_exact(s);
}

// Wanted elements or slots of the lanes, one of every quad at a time.
struct PermQueue {
    uint32_t want;
    int lane, src;
    // false: nothing is left in the warp.  bit: the quad's (-1: none), of lane src.
    __device__ __forceinline__ bool next(int &bit)
    {
        const unsigned b = __ballot_sync(0xffffffffu, want != 0u);
        if (b == 0u) return false;
        const unsigned mine = (b >> (lane & 28)) & 0xFu;
        src = (lane & 28) | (mine ? __ffs(mine) - 1 : 0);
        bit = __ffs(__shfl_sync(0xffffffffu, want, src)) - 1;
        if (lane == src) want &= want - 1u;
        return true;
    }
};

// Per range: the exact maximum of the quad's row where several slots reach the threshold.
template <int LOG2B>
__device__ __noinline__ double perm_many_max(uint32_t rows, const uint2 *at, uint32_t slots, float a32, int lane)
{
    uint32_t x[16];
    perm_gather(rows, *at, x);
    double best = 0.0;
    if (__any_sync(0xffffffffu, __popc(slots) > 2)) {         // flat rows, small integers
        if (perm_row_exact(x)) { best = (double)a32; slots = 0u; }
    }
    PermQueue queue = {slots, lane, 0};
    int s;
#pragma unroll 1
    while (queue.next(s)) {
        double p, m;
        perm_slot<LOG2B>(x, max(s, 0), queue.src & 3, lane & 3, p, m);
        const double t = perm_slot_max(p, m);
        if (s >= 0) best = fmax(best, t);
    }
    return best;
}

// MX: the exact maximum of group lane % 4 of the quad's row, for every lane with `near`, from the elements that reach a - tol.
template <int LOG2B>
__device__ __noinline__ double perm_group_max(uint32_t rows, const uint2 *at, bool near, float a, float tol, int lane)
{
    const int q = lane & 3;
    uint32_t x[16], hb[2][2];
    f32x2 v[8][2];
    perm_gather(rows, *at, x);
    perm_operand(hb, lane);
    perm_rotate<LOG2B>(x, hb, v);
    double best = 0.0;
    if (__popc(__ballot_sync(0xffffffffu, near)) > 4) {
        if (perm_row_exact(x) && near) { best = (double)a; near = false; }
    }
    __syncwarp();
#pragma unroll 1
    for (int g = 0; g < 4; ++g) {
        const unsigned todo = __ballot_sync(0xffffffffu, near && q == g);
        if (todo == 0u) continue;
        const float t = __shfl_sync(0xffffffffu, a - tol, (lane & 28) | g);
        uint32_t want = 0u;
#pragma unroll
        for (int e = 0; e < 32; ++e) {
            const float f = (e & 1) ? v[e >> 2][(e >> 1) & 1].y : v[e >> 2][(e >> 1) & 1].x;
            if ((e >> 3) == g && fabsf(f) >= t) want |= 1u << e;
        }
        if (((todo >> (lane & 28)) & 0xFu) == 0u) want = 0u;
        PermQueue queue = {want, lane, 0};
        double top = 0.0;
        int e;
#pragma unroll 1
        while (queue.next(e)) {
            double p, m;
            perm_slot<LOG2B>(x, max(e, 0) >> 2, queue.src & 3, q, p, m);
            const double u = perm_slot_output(p, m, max(e, 0) & 3, q);
            if (e >= 0) top = fmax(top, fabs(u));
        }
        if (near && q == g) best = top;
    }
    return best;
}

// Codes of a unit with doubtful elements: codes as they are (nibble e % 8 of word e / 8 for element e = 4 slot + output), with those
// settled.  Per 128: a the exact maximum, inv 7 / a, tau the rounding window.  MX: ex the exponents of the row's four groups.
template <int LOG2B, int MODE>
__device__ __noinline__ uint4 perm_mend(uint32_t rows, const uint2 *at, uint4 codes, double sqrt_b, double a, float inv, float tau, uint32_t ex, int lane)
{
    constexpr float err = perm_err(LOG2B, false);
    const int q = lane & 3;
    uint32_t x[16], hb[2][2];
    f32x2 v[8][2];
    perm_gather(rows, *at, x);
    perm_operand(hb, lane);
    perm_rotate<LOG2B>(x, hb, v);
    uint32_t cw[4] = {codes.x, codes.y, codes.z, codes.w}, flags = 0u;
    if (MODE == ROW_GROUP) {
        const float lim = 0.5f - tau;
        const f32x2 m2 = pack2(inv, inv), mg = pack2(12584968.0f, 12584968.0f);
#pragma unroll
        for (int e = 0; e < 16; ++e) {
            const f32x2 f = v[e >> 1][e & 1], d = fma2(f, m2, sub2(mg, fma2(f, m2, mg)));
            flags |= (fabsf(d.x) > lim ? 1u : 0u) << (2 * e) | (fabsf(d.y) > lim ? 2u : 0u) << (2 * e);
        }
    } else {
        // the multipliers as they were; windows that are not smaller (from the largest magnitude of group and block)
        constexpr int CH = LOG2B <= 5 ? 2 : 1 << (LOG2B - 4);
        float ref[8 / CH];
#pragma unroll
        for (int b = 0; b < 8 / CH; ++b) {
            float r = 0.0f;
#pragma unroll
            for (int k = 0; k < CH; ++k) r = fmaxf(r, perm_max4(v[b * CH + k]));
            ref[b] = perm_quad_max(r);
        }
#pragma unroll
        for (int s = 0; s < 8; ++s) {
            const uint32_t Eb = (ex >> (8 * (s >> 1))) & 0xffu;
            const float m = __uint_as_float((uint32_t)min(max(254 - (int)Eb - LOG2B / 2, 1), 254) << 23) * ((LOG2B & 1) ? 0.70710678118654752f : 1.0f);
            // (a byte of 0 may stand for a group of zeros)
            const float r = ref[s / CH], t = r > 0.0f ? (Eb == 0u ? 3.0e38f : perm_window<LOG2B>(err, r, m) * 1.0001f) : 0.0f;
            const f32x2 m2 = pack2(m, m), tp = pack2(t, t), tm = pack2(0.0f - t, 0.0f - t);
            const f32x2 u0 = fma2(v[s][0], m2, tp), u1 = fma2(v[s][1], m2, tp), d0 = fma2(v[s][0], m2, tm), d1 = fma2(v[s][1], m2, tm);
            const uint32_t h = cvt_e2m1x4_pair(u0.x, u0.y, u1.x, u1.y, d0.x, d0.y, d1.x, d1.y), n = (h ^ (h >> 16)) & 0xffffu;
#pragma unroll
            for (int j = 0; j < 4; ++j) flags |= ((n >> (4 * j)) & 0xFu) ? 1u << (4 * s + j) : 0u;
        }
    }
    auto put = [&](int e, double u) {
        const uint32_t code = MODE == ROW_GROUP ? (a > 0.0 ? row_int4_code<false>(u, a, 0.0f, sqrt_b) : 0u)
                                                : row_exact_code<ROW_MX>(u, sqrt_b, 0.0, 0.0, (int)((ex >> (8 * (e >> 3))) & 0xffu) - 127);
        const uint32_t sh = 4u * (uint32_t)(e & 7);
#pragma unroll
        for (int w = 0; w < 4; ++w)
            if ((e >> 3) == w) cw[w] = (cw[w] & ~(0xFu << sh)) | (code << sh);
    };
    if (__reduce_add_sync(0xffffffffu, (uint32_t)__popc(flags)) > 16u) {
        uint32_t own = perm_row_exact(x) ? flags : 0u;
        flags &= ~own;
        if (MODE == ROW_MX) {                                 // zeros beside others, flagged for their sign: all at once (2048 x 9728, b = 128, equal values: 342 -> 113 us)
            uint32_t zero = 0u;
#pragma unroll
            for (int j = 0; j < 32; ++j) zero |= (((j & 1) ? v[j >> 2][(j >> 1) & 1].y : v[j >> 2][(j >> 1) & 1].x) == 0.0f) ? 1u << j : 0u;
            zero &= own;
            own &= ~zero;
#pragma unroll
            for (int w = 0; w < 4; ++w) {
                uint32_t m = (zero >> (8 * w)) & 0xffu;       // a bit to a nibble
                m = (m | m << 12) & 0x000f000fu;
                m = (m | m << 6) & 0x03030303u;
                m = (m | m << 3) & 0x11111111u;
                cw[w] &= ~(m * 15u);
            }
        }
#pragma unroll 1
        while (own) {
            const int e = __ffs(own) - 1;
            own &= own - 1u;
            float f = 0.0f;
#pragma unroll
            for (int j = 0; j < 32; ++j) f = e == j ? ((j & 1) ? v[j >> 2][(j >> 1) & 1].y : v[j >> 2][(j >> 1) & 1].x) : f;
            put(e, (double)f + 0.0);                          // (+0 for a zero, as the sums give)
        }
    }
    __syncwarp();
    PermQueue queue = {flags, lane, 0};
    int e;
#pragma unroll 1
    while (queue.next(e)) {
        double p, m;
        perm_slot<LOG2B>(x, max(e, 0) >> 2, queue.src & 3, q, p, m);
        const double u = perm_slot_output(p, m, max(e, 0) & 3, q);
        if (e >= 0 && lane == queue.src) put(e, u);
        __syncwarp();
    }
    return make_uint4(cw[0], cw[1], cw[2], cw[3]);
}

// -------------------------------------------------------------------------------------------- the kernel

template <int LOG2B, int MODE>
__global__ void __launch_bounds__(PERM_THREADS, 1) perq_perm_kernel(const __grid_constant__ CUtensorMap map, const __grid_constant__ PermParams p)
{
    static_assert(MODE == ROW_MX || MODE == ROW_GROUP, "ranges inside a unit");
    constexpr int CB = LOG2B - 4;
    constexpr float err = perm_err(LOG2B, MODE == ROW_GROUP);
    extern __shared__ __align__(128) unsigned char psmem_raw[];
    unsigned char *smem = psmem_raw + ((1024u - (smem_u32(psmem_raw) & 1023u)) & 1023u);
    const uint32_t base = smem_u32(smem), ring = base + p.off_ring, full = base + p.off_bars;
    uint16_t *tab = reinterpret_cast<uint16_t *>(smem + p.off_tab);
    const uint2 *tab2 = reinterpret_cast<const uint2 *>(tab);
    int tid;
    asm volatile("mov.u32 %0, %%tid.x;" : "=r"(tid));         // (volatile: kept in a register, where the compiler would read it again for every unit)
    const int lane = tid & 31, warp = tid >> 5;
    const int g = lane >> 2, q = lane & 3;

    if (tid < p.stages) {
        mbar_init(full + tid * 8, 1);
        mbar_init_fence();
    }
    __syncthreads();
    griddep_wait();             // nothing above reads or writes global memory
    griddep_launch();
    // whole rounds of a set to a CTA; the sets of the last round are split among the CTAs, each with a part of the units
    const uint32_t rounds = p.sets / gridDim.x, tail = p.sets - rounds * gridDim.x;
    const bool last = blockIdx.x < tail * (uint32_t)p.parts;
    const uint32_t mine = rounds + (last ? 1u : 0u);
    auto set_of = [&](uint32_t it) { return it < rounds ? blockIdx.x + it * gridDim.x : rounds * gridDim.x + blockIdx.x / (uint32_t)p.parts; };
    auto prefetch = [&](uint32_t it, uint32_t box) { tma_prefetch_3d(&map, 0, (int)(set_of(it) * PERM_ROWS), (int)box * (PERM_BOX / 64)); };
    auto load = [&](uint32_t s, uint32_t it, uint32_t box) {  // one thread: a box of the CTA's set it into stage s
        mbar_expect_tx(full + s * 8, PERM_STAGE);             // (positions past the row or the last row are filled with zeros, and count)
        tma_load_3d(ring + s * PERM_STAGE, &map, 0, (int)(set_of(it) * PERM_ROWS), (int)box * (PERM_BOX / 64), full + s * 8);
    };
    // warp w reads the boxes w, w + stages, ... of the CTA's sets, all from stage w (so that no one waits for a phase before the one
    // that is due).  The next one to read, and the next one to load:
    uint32_t read_box = (uint32_t)warp, read_it = 0u, load_box = read_box, load_it = 0u, parity = 0u;
    auto step = [&](uint32_t &box, uint32_t &it) {
        box += (uint32_t)p.stages;
        while (box >= (uint32_t)p.boxes) { box -= (uint32_t)p.boxes; ++it; }
    };
    const bool reader = warp < p.stages;
    if (read_box >= (uint32_t)p.boxes) { read_box -= (uint32_t)p.boxes; read_it = 1u; load_box = read_box; load_it = 1u; }      // (at most two sets' boxes fit)
    if (reader && load_it < mine) {
        if (lane == 0) load((uint32_t)warp, load_it, load_box);
        step(load_box, load_it);
        if (lane == 0 && load_it < mine) prefetch(load_it, load_box);
    }
    for (int k = tid; k < p.d; k += PERM_THREADS)             // (out-of-range entries are clamped)
        tab[(k & ~127) + perm_entry(k & 127)] = (uint16_t)min(max(__ldg(p.perm + k), 0), p.d - 1);
    uint32_t hb[2][2];
    perm_operand(hb, lane);
    const PermSelect select(q);
    // what the lane reads of a box: row lane % 8, 16-byte piece lane / 8 (and 4 further on) of 64 channels
    const uint32_t read_at = (uint32_t)((lane & 7) * 128 + (((lane >> 3) ^ (lane & 7)) << 4));
    bool dead = false;                                        // a load never came: go on to the barriers without waiting again

    auto interleave = [&](uint32_t it) {
#pragma unroll 1
        while (reader && read_it == it) {
            if (!dead && !__all_sync(0xffffffffu, mbar_wait_fast(full + warp * 8, parity))) {
                if (lane == 0) atomicOr(&g_perq_device_error, 1u);
                dead = true;
            }
            const int box = (int)read_box;
            if (!dead) parity ^= 1u;
            step(read_box, read_it);
            const uint32_t from = ring + (uint32_t)warp * PERM_STAGE + read_at, to = base + (uint32_t)(box * PERM_BOX + lane) * 16u;
            const int tasks = min(PERM_BOX, p.d - box * PERM_BOX) / 32;       // (a multiple of 4)
#pragma unroll 1
            for (int t = 0; t < tasks; t += 4) {
                uint32_t r[4][4];
#pragma unroll
                for (int e = 0; e < 4; ++e) ldmatrix_x4_trans(r[e], (from ^ ((e & 1) << 6)) + (uint32_t)(t + e) / 2 * 1024u);
#pragma unroll
                for (int e = 0; e < 4; ++e) stmatrix_x4(to + (uint32_t)(t + e) * 512u, r[e]);
            }
            __syncwarp();
            if (load_it < mine && !dead) {                    // the next box into this one's place, and the one after it into L2
                if (lane == 0) load((uint32_t)warp, load_it, load_box);
                step(load_box, load_it);
                if (lane == 0 && load_it < mine) prefetch(load_it, load_box);
            }
        }
    };
    if (mine > 0) interleave(0);
    __syncthreads();

    for (uint32_t it = 0; it < mine; ++it) {
        const uint32_t row = set_of(it) * PERM_ROWS + (uint32_t)g;
        const bool live = row < p.T;
        int u = warp, u_end = p.units;
        if (it == rounds) {
            const int part = (int)(blockIdx.x % (uint32_t)p.parts);
            u = warp + p.units * part / p.parts;
            u_end = p.units * (part + 1) / p.parts;
        }
        const uint2 *at = tab2 + u * 32 + lane;
        const size_t unit = (size_t)row * p.units + u;
        uint8_t *codes = p.out_codes + unit * 64 + 16 * q;
        uint32_t *scales = reinterpret_cast<uint32_t *>(p.out_scales) + unit;
#pragma unroll 1
        for (; u < u_end; u += PERM_WARPS, at += PERM_WARPS * 32, codes += PERM_WARPS * 64, scales += PERM_WARPS) {
            f32x2 v[8][2];
            uint32_t cw[4];                                   // codes, two slots to a word
            if (MODE == ROW_GROUP) {
                uint32_t x[16];
                perm_gather(base, *at, x);
                perm_rotate<LOG2B>(x, hb, v);
                // (after a call: values that live across one are spilled in every unit)
                auto again = [&]() { perm_gather(base, *at, x); perm_rotate<LOG2B>(x, hb, v); };
                // ---- exact maximum of the range
                float ms[8];
#pragma unroll
                for (int s = 0; s < 8; ++s) ms[s] = perm_max4(v[s]);
                const float a32 = perm_quad_max(fmaxf(fmaxf(fmaxf(ms[0], ms[1]), fmaxf(ms[2], ms[3])), fmaxf(fmaxf(ms[4], ms[5]), fmaxf(ms[6], ms[7]))));
                const float thr = a32 * (1.0f - 2.0f * err - 2.4e-7f);
                uint32_t slots = 0u;
#pragma unroll
                for (int s = 0; s < 8; ++s) slots |= ms[s] >= thr ? 1u << s : 0u;
                if (!(a32 > 0.0f)) slots = 0u;
                // nearly always one slot reaches the threshold: the quad sums its four outputs
                const unsigned cand = (__ballot_sync(0xffffffffu, slots != 0u) >> (lane & 28)) & 0xFu;
                const int src = (lane & 28) | (cand ? __ffs(cand) - 1 : 0);
                const uint32_t m = __shfl_sync(0xffffffffu, slots, src);
                double a;
                if (!__any_sync(0xffffffffu, (cand & (cand - 1u)) != 0u || (m & (m - 1u)) != 0u)) {
                    double sp, sm;
                    perm_slot<LOG2B>(x, m ? __ffs(m) - 1 : 0, src & 3, q, sp, sm);
                    a = perm_slot_max(sp, sm);
                    if (!m) a = 0.0;
                } else {
                    a = perm_many_max<LOG2B>(base, at, slots, a32, lane);
                    again();
                }
                if (q == 0 && live) *scales = __float_as_uint(row_scale(a, p.inv_7_sqrt_b, p.sqrt_b, 7.0));
                // ---- quantise: distance to the rounded value
                const float inv = row_inverse((float)a);
                const float tau = (err + 5.0e-7f) * (inv * a32) + 2.0e-7f;       // the element's error and the multiplier's (three roundings); the distance's own
                const f32x2 m2 = pack2(inv, inv), mg = pack2(12584968.0f, 12584968.0f), up = pack2(-256.0f, -256.0f);     // 1.5 * 2^23 + 8 * 257
                float far0 = 0.0f, far1 = 0.0f;
#pragma unroll
                for (int w = 0; w < 4; ++w) {
                    uint32_t h[2];
#pragma unroll
                    for (int j = 0; j < 2; ++j) {
                        const f32x2 r0 = fma2(v[2 * w + j][0], m2, mg), r1 = fma2(v[2 * w + j][1], m2, mg);
                        const f32x2 n0 = sub2(mg, r0), n1 = sub2(mg, r1);            // minus the rounded values
                        const f32x2 e0 = fma2(v[2 * w + j][0], m2, n0), e1 = fma2(v[2 * w + j][1], m2, n1);
                        far0 = max3abs(far0, e0.x, e0.y);
                        far1 = max3abs(far1, e1.x, e1.y);
                        const f32x2 t = fma2(n1, up, r0);
                        h[j] = __float_as_uint(t.y) * 16u + __float_as_uint(t.x);
                    }
                    cw[w] = __byte_perm(h[0], h[1], 0x5410) ^ 0x88888888u;
                }
                if (__any_sync(0xffffffffu, fmaxf(far0, far1) > 0.5f - tau)) {
                    const uint4 r = perm_mend<LOG2B, MODE>(base, at, make_uint4(cw[0], cw[1], cw[2], cw[3]), p.sqrt_b, a, inv, tau, 0u, lane);
                    cw[0] = r.x; cw[1] = r.y; cw[2] = r.z; cw[3] = r.w;
                }
            } else {
                {
                    uint32_t x[16];
                    perm_gather(base, *at, x);
                    perm_rotate<LOG2B>(x, hb, v);
                }
                // ---- maxima of the groups: lane q gets group q (slots 2 q and 2 q + 1 of the four lanes)
                float a32;
                {
                    float k[4];
#pragma unroll
                    for (int m = 0; m < 4; ++m) k[m] = fmaxf(perm_max4(v[2 * m]), perm_max4(v[2 * m + 1]));
                    const float l0 = fmaxf(select.pick(select.keep2, k[0], k[2]), __shfl_xor_sync(0xffffffffu, select.pick(select.give2, k[0], k[2]), 2));
                    const float l1 = fmaxf(select.pick(select.keep2, k[1], k[3]), __shfl_xor_sync(0xffffffffu, select.pick(select.give2, k[1], k[3]), 2));
                    a32 = fmaxf(select.pick(select.keep1, l0, l1), __shfl_xor_sync(0xffffffffu, select.pick(select.give1, l0, l1), 1));
                }
                float bref = a32;                             // the largest magnitude of the Hadamard block
                if (CB >= 2) bref = fmaxf(bref, __shfl_xor_sync(0xffffffffu, bref, 1));
                if (CB >= 3) bref = fmaxf(bref, __shfl_xor_sync(0xffffffffu, bref, 2));
                // ---- E + 127 with E = floor(log2(a / sqrt(b))) - 2, from the bits of a32; near a boundary the exact maximum
                const uint32_t bits = __float_as_uint(a32);
                const int e8 = (int)(bits >> 23);
                int Eb;
                float dist;
                if ((LOG2B & 1) == 0) {
                    Eb = e8 - LOG2B / 2 - 2;
                    const float lower = __uint_as_float(bits & 0x7f800000u);
                    dist = fminf(a32 - lower, 2.0f * lower - a32);
                } else {
                    Eb = e8 - (LOG2B - 1) / 2 - 3 + ((bits & 0x7fffffu) >= 0x3504f4u ? 1 : 0);
                    dist = fabsf(a32 - __uint_as_float((bits & 0x7f800000u) | 0x3504f3u));
                }
                const float tol = 2.0f * err * bref + a32 * 2.4e-7f;
                // (a group inside a longer block can be zero in fp32 and not in truth)
                const bool near = (LOG2B <= 5 ? a32 : bref) > 0.0f && (dist <= tol || e8 == 0);
                bool zero = !(a32 > 0.0f);
                if (__any_sync(0xffffffffu, near)) {          // rare
                    const double best = perm_group_max<LOG2B>(base, at, near, a32, tol, lane);
                    uint32_t x[16];                           // (again: values that live across a call are spilled in every unit)
                    perm_gather(base, *at, x);
                    perm_rotate<LOG2B>(x, hb, v);
                    if (near) {
                        int ex;
                        (void)frexp(best / p.sqrt_b, &ex);
                        Eb = ex - 3 + 127;
                        zero = best == 0.0;                   // (the fp32 values of a group that cancels exactly are rounding noise)
                    }
                }
                Eb = min(max(Eb, 0), 254);
                float c1 = __uint_as_float((uint32_t)min(max(254 - Eb - LOG2B / 2, 1), 254) << 23) * ((LOG2B & 1) ? 0.70710678118654752f : 1.0f);     // 2^-E / sqrt(b)
                if (zero) { Eb = 0; c1 = 0.0f; }
                // (a block of zeros is exact: no window, so that its zeros are not flagged for their sign)
                const bool exact = !(bref > 0.0f) || (near && zero);
                const float tau = exact ? 0.0f : perm_window<LOG2B>(err, bref, c1);
                uint32_t word = (uint32_t)Eb << (8 * q);
                word |= __shfl_xor_sync(0xffffffffu, word, 1);
                word |= __shfl_xor_sync(0xffffffffu, word, 2);
                if (q == 0 && live) *scales = word;
                // ---- quantise: both codes of the value plus and minus the window
                uint32_t diff[4];
#pragma unroll
                for (int m = 0; m < 4; ++m) {
                    const float c_m = __shfl_sync(0xffffffffu, c1, (lane & 28) | m);
                    const float t_m = LOG2B <= 5 ? perm_window<LOG2B>(err, 0.0f, 0.0f) : __shfl_sync(0xffffffffu, tau, (lane & 28) | m);
                    const f32x2 mc = pack2(c_m, c_m), tp = pack2(t_m, t_m), tm = pack2(0.0f - t_m, 0.0f - t_m);      // (+0 for no window)
                    uint32_t h[2];
#pragma unroll
                    for (int j = 0; j < 2; ++j) {
                        const f32x2 u0 = fma2(v[2 * m + j][0], mc, tp), u1 = fma2(v[2 * m + j][1], mc, tp);
                        const f32x2 d0 = fma2(v[2 * m + j][0], mc, tm), d1 = fma2(v[2 * m + j][1], mc, tm);
                        h[j] = cvt_e2m1x4_pair(u0.x, u0.y, u1.x, u1.y, d0.x, d0.y, d1.x, d1.y);
                    }
                    cw[m] = __byte_perm(h[0], h[1], 0x5410);
                    diff[m] = cw[m] ^ __byte_perm(h[0], h[1], 0x7632);
                }
                bool doubt = (diff[0] | diff[1] | diff[2] | diff[3]) != 0u;
                if (LOG2B <= 5 && __any_sync(0xffffffffu, doubt)) {      // (without the groups of zeros)
                    const unsigned e4 = __ballot_sync(0xffffffffu, exact) >> (lane & 28);
                    doubt = ((e4 & 1u ? 0u : diff[0]) | (e4 & 2u ? 0u : diff[1]) | (e4 & 4u ? 0u : diff[2]) | (e4 & 8u ? 0u : diff[3])) != 0u;
                }
                if (__any_sync(0xffffffffu, doubt)) {
                    const uint4 r = perm_mend<LOG2B, MODE>(base, at, make_uint4(cw[0], cw[1], cw[2], cw[3]), p.sqrt_b, 0.0, 0.0f, 0.0f, word, lane);
                    cw[0] = r.x; cw[1] = r.y; cw[2] = r.z; cw[3] = r.w;
                }
            }
            // ---- the quad's 64 bytes: lane q stores slots 2 q and 2 q + 1
            const uint4 out = perm_quad_words(cw, select);
            if (live) *reinterpret_cast<uint4 *>(codes) = out;
        }
        __syncthreads();
        if (it + 1 < mine) {
            interleave(it + 1);
            __syncthreads();
        }
    }
    // (nothing is in flight when the CTA ends, also after a load that did not come in time)
    if (dead && warp < p.stages) (void)mbar_wait_fast(full + warp * 8, parity);
}

}  // namespace perq
