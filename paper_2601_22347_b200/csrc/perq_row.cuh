// Row rotate+quantize kernel: one CTA per token row, the rotated row in an fp32 tile of shared memory.
//
//   b a power of two (16 <= b <= d)     rows of d % 128 == 0 channels, d <= 16384
//   b == d = 2^k * 4t (no power of two) 6 <= k <= 10 (base matrices of order 12, 28, 36, 60, 76)
// with or without a permutation, every quantised format (INT4 per token or per 32 .. 1024, MXFP4, FP4,
// asymmetric INT4).  It takes what the segment kernels (perq_fast, perq_tok, perq_mx, perq_full) do not: ragged
// widths, blocks longer than 128 with a permutation or another scale mode, rotations of order 2^k * 4t.
//
// One 1024-element segment per warp, 32 outputs per lane, and every value makes one or two round trips through
// the tile:
//   stage    bf16 row by bulk copy into a ring of two rows; permuted rows are gathered into a second bf16 row
//   pass 1   on the tensor cores from the bf16 row (products exact, fp32 accumulators), the first butterfly
//            stages on the accumulators in registers, result into the tile.  Power of two: H_16 and up to three
//            stages, a chunk of 128 per quad, as in the segment kernels.  2^k * 4t: the base matrix on the 4t
//            adjacent inputs of a group, then the k - 5 stages over the group bits that a lane's rows of the 16-group tiles hold
//   pass 2   the remaining stages: a lane reads 32 values (up to 5 index bits), packed add/sub, and writes them
//            back; consecutive lanes are consecutive columns
//   quantise a lane reads 32 CONSECUTIVE outputs (16-byte pieces in an order rotated by the lane, so that eight
//            lanes meet eight bank quads), which makes maxima, packing and the 16-byte code store lane-local
//
// What bounds it: shared-memory passes (4 bytes per element and trip) and, for per-token scales of whole-row
// blocks, the exact row maximum, a d-term fp64 sum that all warps of the row share.  The general kernel, which
// these shapes ran on, made a trip per three stages with eight warps per row and left each exact sum to one warp:
// 1024 x 14336 with b = d took 928 us there and takes 57 here, 1531 x 9728 with b = 128 asymmetric 94 and 32,
// 16384 x 4096 with b = d (group kernel) 228 and 114.
//
// Exactness rules as in perq_generic.cuh: |u32 - u| <= err_rel * (largest |u32| of the block); every value that
// decides an output bit and lies within that bound of a boundary is re-derived in fp64 from the bf16 row.
// Blocks up to 1024 are summed by one warp (per-range scales: by a quad), longer ones by the whole CTA.
#pragma once
#include "perq_full.cuh"

namespace perq {

// Where the Hadamard block lies: inside a segment; over warps (columns of pass 2 kept in registers for 2048 and
// 4096 per token); 2^k * 4t.
enum RowRot { ROT_LOCAL = 0, ROT_WIDE = 1, ROT_COL1 = 2, ROT_COL2 = 3, ROT_NP2 = 4 };
enum RowMode { ROW_TOKEN = 0, ROW_GROUP = 1, ROW_MX = 2, ROW_FP4 = 3, ROW_ASYM = 4 };
constexpr int ROW_MAX_WARPS = 16;
constexpr int ROW_MAX_D = 16384;
constexpr int ROW_REGS = 96;
constexpr int ROW_SM_WARPS = 20;              // as many as the registers allow
constexpr int ROW_CTA_WARPS = 5;              // short rows share a CTA up to this many warps
constexpr int ROW_NSTAGE = 2;
constexpr int ROW_CAP = 16;                   // entries per list and round of the CTA-wide exact sums
constexpr int ROW_WARP_LOG2B = 10;            // blocks up to here are summed by one warp
constexpr int ROW_MANY = 8;                   // of a lane's 32 outputs: from here on exactness is asked (see RowSpan)

struct RowParams {
    const uint16_t *x;
    const int32_t *perm;
    uint8_t *out_codes;
    void *out_scales;
    uint32_t T;
    int d;
    int log2b;               // power of two: log2 of the block; 2^k * 4t: k
    int n0;                  // 4t, or 0
    int log2g;               // ROW_GROUP: log2 of the scale range
    int pad;                 // 2^k * 4t: extra words of the tile per eight groups
    float err_rel;
    double sqrt_b, inv_7_sqrt_b, inv_15_sqrt_b;
    int row_warps;           // warps per row
    // shared memory, from a 1024-byte aligned base: tables of the CTA, then `group_bytes` for every row in flight
    uint32_t off_perm, off_quad, off_bmat, off_hrow, off_group, group_bytes;
    uint32_t off_xs, off_tile, off_misc;                        // from the row's part (its stages come first)
    uint32_t hrow[GEN_MAX_BASE][3];
};

// Reduction space and lists of one row.
struct RowMisc {
    unsigned long long full[ROW_NSTAGE];
    unsigned long long amax;                  // exact largest magnitude (bits) of rows whose candidates are summed by warps
    unsigned long long ahi, alo;              // the same for signed extremes (order keys)
    float wmax[ROW_MAX_WARPS], wmin[ROW_MAX_WARPS];
    uint32_t cnt[2];                          // list lengths: candidates, ties
    uint32_t list[2 * ROW_CAP];               // row positions
    double part[2 * ROW_CAP][ROW_MAX_WARPS];
    float span_sum[ROW_MAX_WARPS];            // see RowSpan
    int span_low[ROW_MAX_WARPS];
};

// 2^k * 4t: the tile holds the groups of n0 values in order, with `pad` extra words after every eight groups:
// 14 n0 + 2 pad = 0 (mod 32), which makes pad an odd multiple of 4.  The lanes of pass 2, which walk a pair of
// groups and go on 16 groups later, then stay on consecutive banks, and so do the stores of pass 1 (even groups
// 0 .. 14, four adjacent words each).
__host__ __device__ constexpr int row_pad(int n0) { return (32 - (14 * n0) % 32) % 32 / 2; }

// Output columns of the base matrix, padded to pairs of tiles.
__host__ __device__ constexpr int row_base_np(int n0) { return (n0 + 15) / 16 * 16; }

// -------------------------------------------------------------------------------------------- exact sums

// Exact unnormalised output at row position pos of a power-of-two block of up to 1024, by one warp.
__device__ __noinline__ double row_exact_warp(const uint16_t *xs, uint32_t pos, int log2b, int lane)
{
    const uint32_t b = 1u << log2b, blk = (pos >> log2b) << log2b, i = pos - blk;
    const uint32_t *src = reinterpret_cast<const uint32_t *>(xs + blk);
    double e = 0.0, o = 0.0;                 // even and odd inputs (times 2^-896, see bf16_bits_to_f64)
#pragma unroll 2
    for (uint32_t w = lane; w < b / 2; w += 32) {
        const uint32_t v = src[w] ^ ((__popc(i & (2 * w)) & 1) ? 0x80008000u : 0u);
        e += bf16_raw_f64(v << 16);
        o += bf16_raw_f64(v);
    }
    double acc = (i & 1u) ? e - o : e + o;
#pragma unroll
    for (int s = 16; s > 0; s >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, s);
    return __shfl_sync(0xffffffffu, acc, 0) * 0x1p896;
}

// The same by the four lanes of a quad, every quad with a position of its own (all 32 lanes call; quads
// without one pass any valid position).
__device__ __forceinline__ double row_exact_quad(const uint16_t *xs, uint32_t pos, int log2b, int lane)
{
    const uint32_t per = 1u << (log2b - 2), blk = (pos >> log2b) << log2b, i = pos - blk, k0 = (lane & 3) * per;
    const uint32_t *src = reinterpret_cast<const uint32_t *>(xs + blk + k0);
    double e = 0.0, o = 0.0;
#pragma unroll 4
    for (uint32_t w = 0; w < per / 2; ++w) {
        const uint32_t v = src[w] ^ ((__popc(i & (k0 + 2 * w)) & 1) ? 0x80008000u : 0u);
        e += bf16_raw_f64(v << 16);
        o += bf16_raw_f64(v);
    }
    double acc = (i & 1u) ? e - o : e + o;
    acc += __shfl_xor_sync(0xffffffffu, acc, 1);
    acc += __shfl_xor_sync(0xffffffffu, acc, 2);
    return __shfl_sync(0xffffffffu, acc, lane & 28) * 0x1p896;
}

// Signs of eight adjacent inputs (bit j set: input k + j is subtracted) of the output at position i, in blocks of a
// power of two: parity of i & (k + j), k a multiple of 8.
__device__ __forceinline__ uint32_t row_sign_pattern(uint32_t i)
{
    return ((i & 1u) ? 0xAAu : 0u) ^ ((i & 2u) ? 0xCCu : 0u) ^ ((i & 4u) ? 0xF0u : 0u);
}
// The same for 2^k * 4t: four inputs lie inside a group of n0; base matrix row at hr, group i2, two table entries qi.
__device__ __forceinline__ uint32_t row_base_signs(const uint32_t *hr, uint32_t i2, uint32_t qi)
{
    uint32_t s = 0u;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const uint32_t ent = (qi >> (16 * h)) & 0xffffu, k2 = ent >> 5, c = (ent & 31u) * 4u;
        uint32_t nib = (hr[c >> 5] >> (c & 31u)) & 0xFu;
        nib ^= ((uint32_t)__popc(i2 & k2) & 1u) ? 0xFu : 0u;
        s |= nib << (4 * h);
    }
    return s;
}

// This warp's part of the exact sum of one listed position: its 1024 inputs, eight adjacent ones per lane and step.
// An input enters as its bf16 fields placed in a double, times 2^896 in the multiply-add (see bf16_bits_to_f64);
// signs: a word per place in the eight (power of two: the same for all steps, the step's own parity in the sign of
// the factor).  (Adding neighbours in fp32 first and converting the sums was slower: the conversion instruction.)
template <bool NP2>
__device__ __forceinline__ double row_partial(const RowParams &p, const uint16_t *xs, const unsigned char *tabs, uint32_t pos, int warp, int lane)
{
    double acc[4] = {0.0, 0.0, 0.0, 0.0};
    uint32_t i = pos, sgn[8];
    const uint32_t *hr = nullptr;
    if (NP2) {
        i = pos / (uint32_t)p.n0;
        hr = reinterpret_cast<const uint32_t *>(tabs + p.off_hrow) + (pos - i * (uint32_t)p.n0) * 3u;
    } else {
        const uint32_t pat = row_sign_pattern(i);
#pragma unroll
        for (int j = 0; j < 8; ++j) sgn[j] = (pat << (31 - j)) & 0x80000000u;
    }
    const uint32_t in_block = NP2 ? 0u : i & ((1u << p.log2b) - 1u);
    // (not unrolled: these kernels are short of instruction cache)
#pragma unroll 1
    for (int r = 0; r < 4; ++r) {
        const uint32_t k = (uint32_t)(warp * SEG_ELEMS + r * 256 + lane * 8);
        if (k >= (uint32_t)p.d || (!NP2 && ((i ^ k) >> p.log2b) != 0u)) continue;       // beyond the row, or another block
        const uint4 w4 = *reinterpret_cast<const uint4 *>(xs + k);
        const uint32_t w[4] = {w4.x, w4.y, w4.z, w4.w};
        double c = 0x1p896;
        if (NP2) {
            const uint32_t s = row_base_signs(hr, i, *reinterpret_cast<const uint32_t *>(tabs + p.off_quad + k / 2));
#pragma unroll
            for (int j = 0; j < 8; ++j) sgn[j] = (s << (31 - j)) & 0x80000000u;
        } else if (__popc(in_block & k) & 1) {
            c = -0x1p896;
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const uint32_t lo = ((uint32_t)((int)(w[j] << 16) >> 3) & 0x8fffe000u) ^ sgn[2 * j];
            const uint32_t hi = ((uint32_t)((int)w[j] >> 3) & 0x8fffe000u) ^ sgn[2 * j + 1];
            acc[(2 * j) & 3] = fma(__hiloint2double((int)lo, 0), c, acc[(2 * j) & 3]);
            acc[(2 * j + 1) & 3] = fma(__hiloint2double((int)hi, 0), c, acc[(2 * j + 1) & 3]);
        }
    }
    return (acc[0] + acc[1]) + (acc[2] + acc[3]);
}

// This warp's parts of the first n0 slots of list 0 and the first n1 of list 1.
template <bool NP2>
__device__ __forceinline__ void row_all_partials(const RowParams &p, const uint16_t *xs, const unsigned char *tabs, unsigned char *smem, int n0, int n1,
                                              int warp, int lane)
{
    RowMisc *ms = reinterpret_cast<RowMisc *>(smem + p.off_misc);
#pragma unroll 1
    for (int e = 0; e < n0 + n1; ++e) {
        const int slot = e < n0 ? e : ROW_CAP + e - n0;
        double v = row_partial<NP2>(p, xs, tabs, ms->list[slot], warp, lane);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == 0) ms->part[slot][warp] = v;
    }
}

__device__ __forceinline__ double row_sum_parts(const RowMisc *ms, int slot)
{
    // (parts of warps that do not exist are zero)
    double v[ROW_MAX_WARPS];
#pragma unroll
    for (int w = 0; w < ROW_MAX_WARPS; ++w) v[w] = ms->part[slot][w];
#pragma unroll
    for (int h = ROW_MAX_WARPS / 2; h > 0; h >>= 1) {
#pragma unroll
        for (int w = 0; w < h; ++w) v[w] += v[w + h];
    }
    return v[0];
}

// Position in the row of element e of a lane: 32 consecutive outputs from i0, in 16-byte pieces rotated by rot
// (cols 0), or one / two adjacent columns of a block's chunks, i0 in the first chunk (cols 1, 2).
__device__ __forceinline__ uint32_t row_position(uint32_t i0, int rot, int cols, int e)
{
    if (cols == 1) return i0 + 128u * (uint32_t)e;
    if (cols == 2) return i0 + 128u * (uint32_t)(e >> 1) + (e & 1u);
    return i0 + 4u * (((uint32_t)(e >> 2) + rot) & 7u) + (e & 3u);
}

// One round of a CTA-wide list: the lane appends the positions of its set bits (as many as fit), in bit order.
// Returns how many it placed; the first one's slot is *slot.
__device__ __forceinline__ int row_append(RowMisc *ms, int which, uint32_t bits, uint32_t i0, int rot, int cols, int &slot)
{
    if (bits == 0u) return 0;
    const int n = __popc(bits);
    const int base = (int)atomicAdd(&ms->cnt[which], (uint32_t)n);
    const int take = min(n, max(0, ROW_CAP - base));
    slot = which * ROW_CAP + base;
#pragma unroll 1
    for (int t = 0; t < take; ++t) {
        const int e = __ffs(bits) - 1;
        bits &= bits - 1;
        ms->list[which * ROW_CAP + base + t] = row_position(i0, rot, cols, e);
    }
    return take;
}

// -------------------------------------------------------------------------------------------- rotation passes

// The permutation as byte offsets into a staged row; out-of-range entries are clamped.
__device__ __forceinline__ void row_load_perm(const RowParams &p, unsigned char *smem, int tid, int nthr)
{
    uint16_t *pt = reinterpret_cast<uint16_t *>(smem + p.off_perm);
    const int4 *p4 = reinterpret_cast<const int4 *>(p.perm);
    const int last = p.d - 1;
#pragma unroll 4
    for (int i = tid; i < p.d / 4; i += nthr) {
        const int4 e = __ldg(p4 + i);
        const uint32_t o0 = (uint32_t)(2 * min(max(e.x, 0), last)), o1 = (uint32_t)(2 * min(max(e.y, 0), last));
        const uint32_t o2 = (uint32_t)(2 * min(max(e.z, 0), last)), o3 = (uint32_t)(2 * min(max(e.w, 0), last));
        reinterpret_cast<uint2 *>(pt)[i] = make_uint2(o0 | (o1 << 16), o2 | (o3 << 16));
    }
}

// This warp's segment of the permuted row (raw: the staged row): lane l takes positions r*256 + 8l .. +7.
__device__ __forceinline__ void row_gather(const RowParams &p, const unsigned char *tabs, unsigned char *smem, uint32_t raw, int warp, int lane)
{
    const uint32_t dst = smem_u32(smem) + p.off_xs + (uint32_t)warp * SEG_BYTES + (uint32_t)lane * 16u;
    const uint4 *offs = reinterpret_cast<const uint4 *>(tabs + p.off_perm) + warp * 128 + lane;
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        if (warp * SEG_ELEMS + r * 256 + lane * 8 < p.d) {
            const uint4 o = offs[r * 32];
            const uint32_t ow[4] = {o.x, o.y, o.z, o.w};
            uint32_t wv[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) wv[e] = lds_u16(raw + (ow[e] & 0xffffu)) | (lds_u16(raw + (ow[e] >> 16)) << 16);
            sts_v4(dst + r * 512, wv[0], wv[1], wv[2], wv[3]);
        }
    }
}

// Stages over C chunk-index bits from bit s on (power-of-two blocks): a lane takes two adjacent columns
// (C <= 4) of 2^C chunk rows at a time, 32 values in all.  LOCAL: inside the warp's segment.
template <int C, bool LOCAL>
__device__ __forceinline__ void row_stages(uint32_t tile, int d, int s, int tid, int nthr)
{
    constexpr int R = 1 << C, NI = 16 >> C;
    const int lane = tid & 31, warp = tid >> 5;
#pragma unroll
    for (int k = 0; k < NI; ++k) {
        int chunk, col;
        if (LOCAL) {
            const int t = lane + 32 * k;
            chunk = warp * 8 + ((t >> 6) << C);
            col = 2 * (t & 63);
            if (chunk * 128 >= d) continue;
        } else {
            const int t = tid + nthr * k;
            if (t >= d / (2 * R)) continue;
            const int rest = t >> 6;
            col = 2 * (t & 63);
            chunk = ((rest >> s) << (s + C)) | (rest & ((1 << s) - 1));
        }
        // (bit 7 of a position flips bit 4 of its tile word: see pass 1)
        const uint32_t a0 = tile + (uint32_t)(chunk * 128 + col) * 4u;
        f32x2 u[R];
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const uint32_t par = (uint32_t)((chunk + (r << s)) & 1) * 64u;
            lds_v2f((a0 + (uint32_t)(r << s) * 512u) ^ par, u[r].x, u[r].y);
        }
#pragma unroll
        for (int t = 0; t < C; ++t) {
#pragma unroll
            for (int r = 0; r < R; ++r) {
                if ((r & (1 << t)) == 0) {
                    const f32x2 x = u[r], y = u[r | (1 << t)];
                    u[r] = add2(x, y);
                    u[r | (1 << t)] = sub2(x, y);
                }
            }
        }
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const uint32_t par = (uint32_t)((chunk + (r << s)) & 1) * 64u;
            sts_v2f((a0 + (uint32_t)(r << s) * 512u) ^ par, u[r].x, u[r].y);
        }
    }
}

// The whole of pass 2 in registers for blocks of 2048 and 4096 (16 or 32 chunks): a lane takes two adjacent columns
// or one, and keeps its 32 outputs.
__device__ __forceinline__ void row_columns(uint32_t tile, int cols, uint32_t i0, f32x2 (&u)[16])
{
    const uint32_t a0 = tile + i0 * 4u;
    if (cols == 2) {
#pragma unroll
        for (int k = 0; k < 16; ++k) lds_v2f((a0 + k * 512u) ^ ((k & 1) * 64u), u[k].x, u[k].y);
    } else {
#pragma unroll
        for (int m = 0; m < 16; ++m) {
            const float a = lds_f(a0 + m * 1024u), b = lds_f((a0 + m * 1024u + 512u) ^ 64u);
            u[m] = pack2(a + b, a - b);
        }
    }
#pragma unroll
    for (int t = 0; t < 4; ++t) {
#pragma unroll
        for (int m = 0; m < 16; ++m) {
            if ((m & (1 << t)) == 0) {
                const f32x2 x = u[m], y = u[m | (1 << t)];
                u[m] = add2(x, y);
                u[m | (1 << t)] = sub2(x, y);
            }
        }
    }
}

// 32 x 32 codes of a warp, a column (or two) per lane -> a run of 32 adjacent positions per lane: bit s of the
// nibble index changes places with bit s - (cols - 1) of the lane.  Ten shuffles of packed codes in place of a
// second trip of the fp32 values through shared memory.
__device__ __forceinline__ void row_transpose_codes(uint32_t (&w)[4], int cols, int lane)
{
    const int c = cols - 1;
#pragma unroll
    for (int s = 0; s < 3; ++s) {
        if (s < c) continue;
        const int bit = 1 << (s - c), sh = 4 << s;
        const uint32_t M = s == 0 ? 0x0f0f0f0fu : s == 1 ? 0x00ff00ffu : 0x0000ffffu;
        const bool up = (lane & bit) != 0;
        const int a = up ? 0 : sh, b = sh - a;
        const uint32_t keep = up ? ~M : M;
#pragma unroll
        for (int h = 0; h < 4; h += 2) {
            const uint32_t out = ((w[h] >> a) & M) | ((w[h + 1] << b) & ~M);
            const uint32_t in = __shfl_xor_sync(0xffffffffu, out, bit);
            w[h] = (w[h] & keep) | ((in << a) & ~keep);
            w[h + 1] = (w[h + 1] & keep) | ((in >> b) & ~keep);
        }
    }
#pragma unroll
    for (int s = 3; s < 5; ++s) {
        const int bit = 1 << (s - c), dist = s - 2;
        const bool up = (lane & bit) != 0;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int lo = s == 3 ? 2 * h : h, hi = lo + dist;
            const uint32_t in = __shfl_xor_sync(0xffffffffu, up ? w[lo] : w[hi], bit);
            if (up) w[lo] = in; else w[hi] = in;
        }
    }
}

// Pass 1 of a 2^k * 4t rotation: task = NTT output tiles (8 columns each) of the base matrix and MT tiles of 16
// groups.  Row g of a tile is group 2 g and row g + 8 group 2 g + 1, so that the eight groups of a fragment load lie
// on different banks (n0 is an odd multiple of 4: the words of even groups start at different multiples of 4).
// Columns 2 q, 2 q + 1 of a tile are outputs q and q + 4: two stores of four adjacent words per group.  Stages over
// group bit 0 (the two rows of a lane) and the tile bits, then into the fp32 tile.
template <int MT, int NTT>
__device__ __forceinline__ void row_base_pass(const RowParams &p, const uint16_t *xs, const unsigned char *tabs, uint32_t tile, int warp,
                                              int warps, int lane)
{
    const int n0 = p.n0, KT = (n0 + 15) >> 4, NG = ((n0 + 7) / 8 + NTT - 1) / NTT, LDK = gen_base_ldk(n0);
    const int g = lane >> 2, q = lane & 3;
    const uint16_t *bm = reinterpret_cast<const uint16_t *>(tabs + p.off_bmat);
    for (int task = warp; task < 4 * NG; task += warps) {
        const int nt0 = (task >> 2) * NTT, mg = task & 3;
        float c[NTT][MT][4];
#pragma unroll
        for (int n = 0; n < NTT; ++n) {
#pragma unroll
            for (int m = 0; m < MT; ++m) c[n][m][0] = c[n][m][1] = c[n][m][2] = c[n][m][3] = 0.0f;
        }
        const uint16_t *arow = xs + (size_t)(mg * MT * 16 + 2 * g) * n0 + 2 * q;
        const uint16_t *brow = bm + (nt0 * 8 + g) * LDK + 2 * q;
        for (int kt = 0; kt < KT; ++kt) {
            uint32_t b[NTT][2];
#pragma unroll
            for (int n = 0; n < NTT; ++n) {
                b[n][0] = *(const uint32_t *)(brow + n * 8 * LDK + kt * 16);
                b[n][1] = *(const uint32_t *)(brow + n * 8 * LDK + kt * 16 + 8);
            }
            const bool in0 = kt * 16 + 2 * q < n0, in1 = kt * 16 + 8 + 2 * q < n0;      // (n0 is even)
#pragma unroll
            for (int m = 0; m < MT; ++m) {
                const uint16_t *ar = arow + m * 16 * n0 + kt * 16;
                uint32_t a[4];
                a[0] = in0 ? *(const uint32_t *)ar : 0u;
                a[1] = in0 ? *(const uint32_t *)(ar + n0) : 0u;
                a[2] = in1 ? *(const uint32_t *)(ar + 8) : 0u;
                a[3] = in1 ? *(const uint32_t *)(ar + n0 + 8) : 0u;
#pragma unroll
                for (int n = 0; n < NTT; ++n) gen_mma_bf16(c[n][m], a, b[n][0], b[n][1]);
            }
        }
#pragma unroll
        for (int n = 0; n < NTT; ++n) {
            f32x2 v[2 * MT];                   // index bit 0: group bit 0, the others: tile bits
#pragma unroll
            for (int m = 0; m < MT; ++m) { v[2 * m] = pack2(c[n][m][0], c[n][m][1]); v[2 * m + 1] = pack2(c[n][m][2], c[n][m][3]); }
#pragma unroll
            for (int t = 1; t < 2 * MT; t <<= 1) {
#pragma unroll
                for (int r = 0; r < 2 * MT; ++r) {
                    if ((r & t) == 0) {
                        const f32x2 x = v[r], y = v[r | t];
                        v[r] = add2(x, y);
                        v[r | t] = sub2(x, y);
                    }
                }
            }
            const int col = (nt0 + n) * 8 + q;             // outputs col and col + 4
            const uint32_t step = (uint32_t)(16 * n0 + 2 * p.pad) * 4u, next = (uint32_t)n0 * 4u;
            uint32_t a = tile + (uint32_t)(mg * MT) * step + (uint32_t)(2 * g * n0 + (g >> 2) * p.pad + col) * 4u;
#pragma unroll
            for (int m = 0; m < MT; ++m) {
                if (col < n0) { sts_f(a, v[2 * m].x); sts_f(a + next, v[2 * m + 1].x); }
                if (col + 4 < n0) { sts_f(a + 16, v[2 * m].y); sts_f(a + next + 16, v[2 * m + 1].y); }
                a += step;
            }
        }
    }
}

// Pass 2 of a 2^k * 4t rotation: group bits 1..3 and the two highest, a lane one column of a group parity.
__device__ __forceinline__ void row_base_stages(const RowParams &p, uint32_t tile, int tid)
{
    if (tid >= p.d / 32) return;
    const uint32_t mid = (uint32_t)tid / (uint32_t)(2 * p.n0), r = (uint32_t)tid - mid * (uint32_t)(2 * p.n0);
    const uint32_t step = (uint32_t)(16 * p.n0 + 2 * p.pad) * 4u;
    const uint32_t quarter = step << (p.log2b - 6);            // 2^(k - 2) groups
    const uint32_t a0 = tile + mid * step + r * 4u, pair = (uint32_t)(2 * p.n0) * 4u, half = (uint32_t)p.pad * 4u;
    auto addr = [&](int m) { return a0 + (uint32_t)(m & 7) * pair + ((m & 4) ? half : 0u) + (uint32_t)(m >> 3) * quarter; };
    f32x2 u[16];                                               // .x / .y: the highest group bit; index bit 3: the one below
#pragma unroll
    for (int m = 0; m < 16; ++m) {
        u[m].x = lds_f(addr(m));
        u[m].y = lds_f(addr(m) + 2 * quarter);
    }
#pragma unroll
    for (int t = 0; t < 4; ++t) {
#pragma unroll
        for (int m = 0; m < 16; ++m) {
            if ((m & (1 << t)) == 0) {
                const f32x2 x = u[m], y = u[m | (1 << t)];
                u[m] = add2(x, y);
                u[m | (1 << t)] = sub2(x, y);
            }
        }
    }
#pragma unroll
    for (int m = 0; m < 16; ++m) {
        sts_f(addr(m), u[m].x + u[m].y);
        sts_f(addr(m) + 2 * quarter, u[m].x - u[m].y);
    }
}

// -------------------------------------------------------------------------------------------- codes

// Exact code of an element from its exact unnormalised value u, in the operation order of the definition.
template <int MODE>
__device__ __noinline__ uint32_t row_exact_code(double u, double sqrt_b, double s64, double z64, int E)
{
    const double y = u / sqrt_b;
    if (MODE == ROW_MX) return e2m1_code_exact(scalbn(y, -E), signbit(y));
    if (MODE == ROW_FP4) return e2m1_code_exact((s64 == 0.0) ? 0.0 : y / s64, signbit(y));
    if (s64 == 0.0) return 0u;
    if (MODE == ROW_ASYM) return (uint32_t)((int)fmin(fmax(rint(y / s64) - z64, 0.0), 15.0));
    return (uint32_t)((int)fmin(fmax(rint(y / s64), -8.0), 7.0)) & 0xFu;
}

// Symmetric INT4: exact code of a doubtful element, u its exact value, a the exact maximum of its range.  The tie
// is between |y / s| = n and n + 1, y / s = 7 u / a: the sign of 14 |u| - (2 n + 1) a decides (two products whose
// rounding errors are far below the margin), the definition's divisions only an all but exact tie.
// n from the fp32 multiplier where that is 7 / a to a few ulp (scales of whole rows, or from exact values).  In a range
// that is small beside its block (PINNED false) the fp32 maximum is partly rounding noise: its multiplier can be off by
// any factor and every element of the range comes here, so n is formed from the exact values.
template <bool PINNED>
__device__ __forceinline__ uint32_t row_int4_code(double u, double a, float mul, double sqrt_b)
{
    const int n = PINNED ? (int)(fabsf((float)u) * mul) : (int)(7.0 * fabs(u) / a);
    const double diff = 14.0 * fabs(u) - (double)(2 * n + 1) * a;
    if (!(fabs(diff) > a * 1.0e-12)) return row_exact_code<ROW_TOKEN>(u, sqrt_b, a / sqrt_b / 7.0, 0.0, 0);
    const int k = n + (diff > 0.0 ? 1 : 0);
    return (uint32_t)(u < 0.0 ? -k : k) & 0xFu;
}

// 7 / a, capped.  The approximate division gives 0 for divisors above 2^126, which unnormalised maxima of finite rows do
// reach: a quarter of one does not.  (A true division: 32.3 against 32.1 us for 4096 x 2048, b = d, per 128.)
__device__ __forceinline__ float row_inverse(float a) { return (a > 0.0f) ? fminf(__fdividef(1.75f, 0.25f * a), 3.0e38f) : 0.0f; }

// (float)(a / sqrt(b) / k), inv = 1 / (k sqrt(b)): one product unless the result is all but on a rounding boundary.
__device__ __forceinline__ float row_scale(double a, double inv, double sqrt_b, double k)
{
    const double s = a * inv;
    const float f = (float)(s * (1.0 - 0x1p-50));
    return f == (float)(s * (1.0 + 0x1p-50)) ? f : (float)(a / sqrt_b / k);
}

// Replace the code of bit e in the lane's (logically ordered) code words.
__device__ __forceinline__ void row_patch(uint32_t (&cw)[4], int e, int rot, uint32_t code)
{
    const uint32_t le = 4u * (((uint32_t)(e >> 2) + rot) & 7u) + (e & 3u), sh = 4u * (le & 7u);
#pragma unroll
    for (int w = 0; w < 4; ++w)
        if ((le >> 3) == (uint32_t)w) cw[w] = (cw[w] & ~(0xFu << sh)) | (code << sh);
}

// Rows in which many outputs tie for the maximum or sit on rounding ties (one nonzero, +-constant, few small integers)
// would pay a sum for each.  Their fp32 rotation is exact: where all inputs are multiples of 2^l and their magnitudes
// add up to no more than 2^(l + 22), so is every partial sum, and all of them are floats (on the tensor cores too: 23
// bits below the largest product).  Then the fp32 outputs stand for the sums.  1024 rows of 4096 with one nonzero each,
// b = d, INT4: 7642 us with a sum for every output, four outputs to a sum (the group kernel before) 2040, 43 now; one
// nonzero per block of 128, 512 rows of 1152: 312 and 7.
struct RowSpan {
    float sum;               // of the magnitudes
    int low;                 // exponent of the lowest set bit, plus 134
};
__device__ __forceinline__ bool row_span_exact(RowSpan s) { return s.sum <= __uint_as_float((uint32_t)min(s.low + 15, 254) << 23); }

// One warp's 1024 inputs (n of them valid).
__device__ __noinline__ RowSpan row_segment_span(const uint16_t *seg, int n, int lane)
{
    RowSpan s = {0.0f, 1 << 20};
#pragma unroll 1
    for (int k = lane * 8; k < min(n, SEG_ELEMS); k += 256) {
        const uint4 w4 = *reinterpret_cast<const uint4 *>(seg + k);
        const uint32_t w[4] = {w4.x, w4.y, w4.z, w4.w};
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const uint32_t a = (w[e >> 1] >> (16 * (e & 1))) & 0x7fffu;
            s.sum += __uint_as_float(a << 16);
            // (the mantissa with its leading one; subnormals have the exponent of the smallest normal)
            if (a != 0u) s.low = min(s.low, a < 0x80u ? __ffs(a) : (int)(a >> 7) + __ffs((a & 0x7fu) | 0x80u) - 1);
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s.sum += __shfl_xor_sync(0xffffffffu, s.sum, o);
    s.low = __reduce_min_sync(0xffffffffu, s.low);
    return s;
}

// The whole row: every warp its segment, a barrier of the row, then the verdict.
__device__ __forceinline__ void row_put_span(RowMisc *ms, const uint16_t *xs, int d, int segs, int warp, int lane)
{
    if (warp >= segs) return;
    const RowSpan s = row_segment_span(xs + warp * SEG_ELEMS, d - warp * SEG_ELEMS, lane);
    if (lane == 0) { ms->span_sum[warp] = s.sum; ms->span_low[warp] = s.low; }
}
__device__ __forceinline__ bool row_all_exact(const RowMisc *ms, int segs, int lane)
{
    RowSpan s = {0.0f, 1 << 20};
    if (lane < segs) { s.sum = ms->span_sum[lane & 15]; s.low = ms->span_low[lane & 15]; }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s.sum += __shfl_xor_sync(0xffffffffu, s.sum, o);
    s.low = __reduce_min_sync(0xffffffffu, s.low);
    return row_span_exact(s);
}

// What the quantiser of a lane's 32 values needs: multiplier, rounding window, zero point.
struct RowQuant {
    float mul, tau, magic;
};

// Codes of the lane's values (pieces as read), and whether any of them is within the window of a tie.
// Integers: r = round(v * mul) + magic in one packed fma, distance to the rounded value in two more.
// E2M1: two conversions, of the scaled value plus and minus the window.
template <int MODE>
__device__ __forceinline__ bool row_quantise(const f32x2 (&u)[16], const RowQuant &Q, uint32_t (&cw)[4])
{
    const f32x2 m2 = pack2(Q.mul, Q.mul);
    uint32_t h[8], diff = 0u;
    if (MODE == ROW_MX || MODE == ROW_FP4) {
        const f32x2 tp = pack2(Q.tau, Q.tau), tm = pack2(0.0f - Q.tau, 0.0f - Q.tau);
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const f32x2 up0 = fma2(u[2 * j], m2, tp), up1 = fma2(u[2 * j + 1], m2, tp);
            const f32x2 dn0 = fma2(u[2 * j], m2, tm), dn1 = fma2(u[2 * j + 1], m2, tm);
            h[j] = cvt_e2m1x4_pair(up0.x, up0.y, up1.x, up1.y, dn0.x, dn0.y, dn1.x, dn1.y);
            diff |= h[j] ^ (h[j] >> 16);
        }
        diff &= 0xffffu;
    } else {
        const f32x2 mg = pack2(Q.magic, Q.magic);
        float far = 0.0f;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            f32x2 r0 = fma2(u[2 * j], m2, mg), r1 = fma2(u[2 * j + 1], m2, mg);
            const f32x2 e0 = fma2(u[2 * j], m2, sub2(mg, r0)), e1 = fma2(u[2 * j + 1], m2, sub2(mg, r1));
            far = max3abs(far, e0.x, e0.y);
            far = max3abs(far, e1.x, e1.y);
            if (MODE == ROW_ASYM) {            // codes 0 .. 15
                const float lo = 12582912.0f, hi = 12582927.0f;
                r0 = pack2(fminf(fmaxf(r0.x, lo), hi), fminf(fmaxf(r0.y, lo), hi));
                r1 = pack2(fminf(fmaxf(r1.x, lo), hi), fminf(fmaxf(r1.y, lo), hi));
            }
            h[j] = ((__float_as_uint(r1.y) * 16u + __float_as_uint(r1.x)) * 16u + __float_as_uint(r0.y)) * 16u + __float_as_uint(r0.x);
        }
        diff = (far > 0.5f - Q.tau) ? 1u : 0u;
    }
#pragma unroll
    for (int w = 0; w < 4; ++w) {
        cw[w] = __byte_perm(h[2 * w], h[2 * w + 1], 0x5410);
        if (MODE == ROW_TOKEN || MODE == ROW_GROUP) cw[w] ^= 0x88888888u;
    }
    return diff != 0u;
}

// The flagged elements of a lane (bits in the order of its pieces); recomputed only where row_quantise said so.
template <int MODE>
__device__ __forceinline__ uint32_t row_tie_bits(const f32x2 (&u)[16], const RowQuant &Q)
{
    uint32_t bits = 0u;
#pragma unroll
    for (int m = 0; m < 16; ++m) {
        const float t[2] = {u[m].x, u[m].y};
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            bool f;
            if (MODE == ROW_MX || MODE == ROW_FP4) {
                f = cvt_e2m1x2(fmaf(t[k], Q.mul, Q.tau), 0.0f) != cvt_e2m1x2(fmaf(t[k], Q.mul, 0.0f - Q.tau), 0.0f);
            } else {
                const float r = fmaf(t[k], Q.mul, Q.magic);
                f = fabsf(fmaf(t[k], Q.mul, Q.magic - r)) > 0.5f - Q.tau;
            }
            bits |= (f ? 1u : 0u) << (2 * m + k);
        }
    }
    return bits;
}

// Code words from the order in which the pieces were read to their order in the row: 16-bit piece j -> (j + rot) mod 8.
__device__ __forceinline__ void row_unrotate(uint32_t (&cw)[4], int rot)
{
    if (rot & 4) {
        uint32_t t = cw[0]; cw[0] = cw[2]; cw[2] = t;
        t = cw[1]; cw[1] = cw[3]; cw[3] = t;
    }
    if (rot & 2) { const uint32_t t = cw[3]; cw[3] = cw[2]; cw[2] = cw[1]; cw[1] = cw[0]; cw[0] = t; }
    if (rot & 1) {
        const uint32_t a = __funnelshift_l(cw[3], cw[0], 16), b = __funnelshift_l(cw[0], cw[1], 16);
        const uint32_t c = __funnelshift_l(cw[1], cw[2], 16), d = __funnelshift_l(cw[2], cw[3], 16);
        cw[0] = a; cw[1] = b; cw[2] = c; cw[3] = d;
    }
}

// Bits of the lane's values for which |v| >= thr.
__device__ __forceinline__ uint32_t row_reach(const f32x2 (&u)[16], float thr)
{
    uint32_t bits = 0u;
#pragma unroll
    for (int m = 0; m < 16; ++m) bits |= (fabsf(u[m].x) >= thr ? 1u : 0u) << (2 * m) | (fabsf(u[m].y) >= thr ? 2u : 0u) << (2 * m);
    return bits;
}

// A lane's place in the row, for the functions below.
struct RowLane {
    uint32_t tile, i0, t_read;
    int rot, warp, tid;
};

// Codes of a lane's doubtful elements where the fp32 outputs are exact: read again from the tile (columns: formed again).
template <int MODE, int COLS>
__device__ __forceinline__ void row_settle(uint32_t (&cw)[4], uint32_t tie, const RowLane &L, double a, float mul, double sqrt_b, double s64, double z64,
                                           int E)
{
    f32x2 u[16];
    if (COLS) row_columns(L.tile, COLS, L.i0, u);
#pragma unroll 1
    while (tie) {
        const int e = __ffs(tie) - 1;
        tie &= tie - 1;
        float v = 0.0f;
        if (COLS) {
#pragma unroll
            for (int m = 0; m < 16; ++m) v = (e >> 1) == m ? ((e & 1) ? u[m].y : u[m].x) : v;
        } else {
            v = lds_f(L.t_read + 16u * (uint32_t)(((e >> 2) + L.tid) & 7) + 4u * (uint32_t)(e & 3));
        }
        const double x = (double)v + 0.0;                     // (+0 for a zero, as the sum gives)
        row_patch(cw, e, L.rot, MODE == ROW_TOKEN || MODE == ROW_GROUP ? row_int4_code<MODE == ROW_TOKEN>(x, a, mul, sqrt_b)
                                                                     : row_exact_code<MODE>(x, sqrt_b, s64, z64, E));
    }
}
template <int MODE>
__device__ __noinline__ uint4 row_settle_warp(uint4 words, uint32_t tie, RowLane L, double a, float mul, double sqrt_b, double s64, double z64, int E)
{
    uint32_t cw[4] = {words.x, words.y, words.z, words.w};
    row_settle<MODE, 0>(cw, tie, L, a, mul, sqrt_b, s64, z64, E);
    return make_uint4(cw[0], cw[1], cw[2], cw[3]);
}

// Blocks over several warps: what follows a first round of the lists that did not hold all (all threads of the CTA
// call).  Not inlined: inside the row's loop these paths cost 7 % of the time of 8192 channels, b = d, INT4.
// Per token: candidates and doubtful elements.  Leaves the row's exact extremes in amax, or ahi and alo.
template <int MODE, bool NP2, int COLS>
__device__ __noinline__ uint4 row_many_token(const RowParams &p, const uint16_t *xs, const unsigned char *tabs, unsigned char *smem, RowLane L,
                                             uint32_t want, uint32_t tie, uint4 words, float mul, double a_ex, double hi_ex, double lo_ex)
{
    RowMisc *ms = reinterpret_cast<RowMisc *>(smem + p.off_misc);
    uint32_t cw[4] = {words.x, words.y, words.z, words.w};
    const int lane = L.tid & 31, segs = (p.d + SEG_ELEMS - 1) / SEG_ELEMS;
    double s64 = 0.0;
    bool more = true;
    for (bool first = true; more; first = false) {
        int slot = 0, tslot = 0;
        const int took = row_append(ms, 0, want, L.i0, L.rot, COLS, slot);
        for (int t = 0; t < took; ++t) want &= want - 1;
        const int ttook = row_append(ms, 1, tie, L.i0, L.rot, COLS, tslot);
        if (first) row_put_span(ms, xs, p.d, segs, L.warp, lane);
        __syncthreads();
        const bool exact = first && row_all_exact(ms, segs, lane);
        const int total = exact ? 0 : (int)ms->cnt[0], n = min(total, ROW_CAP);
        const int ttotal = exact ? 0 : (int)ms->cnt[1], tn = min(ttotal, ROW_CAP);
        const bool last = total <= ROW_CAP;
        if (exact) {
            if (MODE == ROW_ASYM) {
                hi_ex = (double)warp_max_f32(lane < segs ? ms->wmax[lane & 15] : -3.0e38f) + 0.0;
                lo_ex = (double)warp_min_f32(lane < segs ? ms->wmin[lane & 15] : 3.0e38f) + 0.0;
            } else {
                a_ex = (double)warp_max_f32(lane < segs ? ms->wmax[lane & 15] : 0.0f);
            }
            if (MODE == ROW_FP4) s64 = a_ex / p.sqrt_b / 7.0;
            if (MODE != ROW_ASYM && tie) row_settle<MODE, COLS>(cw, tie, L, a_ex, mul, p.sqrt_b, s64, 0.0, 0);
            want = tie = 0u;
        }
        row_all_partials<NP2>(p, xs, tabs, smem, n, tn, L.warp, lane);
        more = __syncthreads_or(!last || ttotal > ROW_CAP);          // (of any row of the CTA)
        if (L.tid == 0) ms->cnt[0] = ms->cnt[1] = 0u;
        for (int e = 0; e < n; ++e) {
            const double v = row_sum_parts(ms, e);
            a_ex = fmax(a_ex, fabs(v));
            hi_ex = fmax(hi_ex, v);
            lo_ex = fmin(lo_ex, v);
        }
        if (last && ttook > 0 && !exact) {
            if (MODE == ROW_FP4) s64 = a_ex / p.sqrt_b / 7.0;
            for (int t = 0; t < ttook; ++t) {
                const int e = __ffs(tie) - 1;
                tie &= tie - 1;
                const double v = row_sum_parts(ms, tslot + t);
                row_patch(cw, e, L.rot, MODE == ROW_TOKEN ? row_int4_code<true>(v, a_ex, mul, p.sqrt_b)
                                                          : row_exact_code<MODE>(v, p.sqrt_b, s64, 0.0, 0));
            }
        }
        if (more) __syncthreads();
    }
    // (per token symmetric: only the row's first thread reads it)
    if (L.tid == 0) {
        if (MODE == ROW_ASYM) { ms->ahi = order_key(hi_ex); ms->alo = order_key(lo_ex); }
        else ms->amax = (unsigned long long)__double_as_longlong(a_ex);
    }
    if (MODE == ROW_ASYM) __syncthreads();
    return make_uint4(cw[0], cw[1], cw[2], cw[3]);
}

// Per range: the exact maximum of the lane's candidates; lm is the largest magnitude of its fp32 outputs.  worth: more
// candidates than a few for every range.
template <bool NP2>
__device__ __noinline__ double row_many_max(const RowParams &p, const uint16_t *xs, const unsigned char *tabs, unsigned char *smem, RowLane L,
                                            uint32_t want, bool any, float lm, double a_ex, bool worth)
{
    RowMisc *ms = reinterpret_cast<RowMisc *>(smem + p.off_misc);
    const int lane = L.tid & 31;
    const int segs = (p.d + SEG_ELEMS - 1) / SEG_ELEMS;
    bool more = true;
    for (bool first = worth; more; first = false) {
        int slot = 0;
        int took = row_append(ms, 0, want, L.i0, L.rot, 0, slot);
        for (int t = 0; t < took; ++t) want &= want - 1;
        if (first) row_put_span(ms, xs, p.d, segs, L.warp, lane);
        __syncthreads();
        const bool exact = first && row_all_exact(ms, segs, lane);
        const int total = exact ? 0 : (int)ms->cnt[0], n = min(total, ROW_CAP);
        if (exact) {
            if (any) a_ex = (double)lm;
            want = 0u;
            took = 0;
        }
        row_all_partials<NP2>(p, xs, tabs, smem, n, 0, L.warp, lane);
        more = __syncthreads_or(total > ROW_CAP);
        if (L.tid == 0) ms->cnt[0] = 0u;
        for (int t = 0; t < took; ++t) a_ex = fmax(a_ex, fabs(row_sum_parts(ms, slot + t)));
        if (more) __syncthreads();
    }
    return a_ex;
}

// Doubtful elements of formats that quantise after the exact scale.
template <int MODE, bool NP2, int COLS>
__device__ __noinline__ uint4 row_many_ties(const RowParams &p, const uint16_t *xs, const unsigned char *tabs, unsigned char *smem, RowLane L,
                                            uint32_t tie, uint4 words, float mul, double a, double s64, double z64, int E)
{
    RowMisc *ms = reinterpret_cast<RowMisc *>(smem + p.off_misc);
    uint32_t cw[4] = {words.x, words.y, words.z, words.w};
    const int lane = L.tid & 31;
    const int segs = (p.d + SEG_ELEMS - 1) / SEG_ELEMS;
    bool more = true;
    for (bool first = true; more; first = false) {
        int slot = 0;
        int took = row_append(ms, 1, tie, L.i0, L.rot, COLS, slot);
        if (first) row_put_span(ms, xs, p.d, segs, L.warp, lane);
        __syncthreads();
        const bool exact = first && row_all_exact(ms, segs, lane);
        const int total = exact ? 0 : (int)ms->cnt[1], n = min(total, ROW_CAP);
        if (exact) {
            if (tie) row_settle<MODE, COLS>(cw, tie, L, a, mul, p.sqrt_b, s64, z64, E);
            tie = 0u;
            took = 0;
        }
        row_all_partials<NP2>(p, xs, tabs, smem, 0, n, L.warp, lane);
        more = __syncthreads_or(total > ROW_CAP);
        if (L.tid == 0) ms->cnt[1] = 0u;
        for (int t = 0; t < took; ++t) {
            const int e = __ffs(tie) - 1;
            tie &= tie - 1;
            const double v = row_sum_parts(ms, slot + t);
            row_patch(cw, e, L.rot, MODE == ROW_GROUP ? row_int4_code<false>(v, a, mul, p.sqrt_b) : row_exact_code<MODE>(v, p.sqrt_b, s64, z64, E));
        }
        if (more) __syncthreads();
    }
    return make_uint4(cw[0], cw[1], cw[2], cw[3]);
}

// -------------------------------------------------------------------------------------------- the kernel

template <int ROT, int MODE>
__global__ void __maxnreg__(ROW_REGS) perq_row_kernel(const __grid_constant__ RowParams p)
{
    constexpr bool TOK = MODE == ROW_TOKEN || MODE == ROW_FP4 || MODE == ROW_ASYM;
    constexpr bool NP2 = ROT == ROT_NP2;
    constexpr bool wide = ROT != ROT_LOCAL;                    // a block spans warps
    constexpr bool row_max = TOK || wide;                      // the row maximum is exchanged
    constexpr int cols = ROT == ROT_COL1 ? 1 : ROT == ROT_COL2 ? 2 : 0;
    static_assert(TOK || cols == 0, "columns: per-token formats");
    extern __shared__ __align__(128) unsigned char rsmem_raw[];
    unsigned char *tabs = rsmem_raw + ((1024u - (smem_u32(rsmem_raw) & 1023u)) & 1023u);
    // rows in flight: row_warps warps each, in step (every barrier is the CTA's).  Few per CTA: all rows of an SM in
    // one CTA waited for one another at every barrier (147 us for 16384 x 4096 with b = d; a CTA per row: 116 us).
    const int lane = threadIdx.x & 31, group = (int)(threadIdx.x >> 5) / p.row_warps, warps = p.row_warps;
    const int warp = (int)(threadIdx.x >> 5) - group * warps, tid = warp * 32 + lane, nthr = warps * 32;
    const int groups = (int)blockDim.x / nthr;
    unsigned char *smem = tabs + p.off_group + group * p.group_bytes;
    const int d = p.d, g = lane >> 2, q = lane & 3;
    const int segs = (d + SEG_ELEMS - 1) / SEG_ELEMS;          // warps that hold a part of the row
    const bool permuted = p.perm != nullptr;
    RowMisc *ms = reinterpret_cast<RowMisc *>(smem + p.off_misc);
    const uint32_t base = smem_u32(smem), tile = base + p.off_tile;
    const uint32_t stage_bytes = (uint32_t)segs * SEG_BYTES, full = smem_u32(ms->full);
    const uint32_t row_bytes = (uint32_t)d * 2u;

    if (tid < ROW_NSTAGE) {
        mbar_init(full + tid * 8, 1);
        mbar_init_fence();
    }
    for (int e = tid; e < 2 * ROW_CAP * ROW_MAX_WARPS; e += nthr) (&ms->part[0][0])[e] = 0.0;
    if (tid == 0) {
        ms->cnt[0] = ms->cnt[1] = 0u;
        ms->amax = ms->ahi = 0ull;
        ms->alo = ~0ull;
    }
    if (NP2) {
        // base matrix as bf16 +-1 (0 in the padding), [output][input]; its sign rows; (group, column) of every four inputs
        uint16_t *bm = reinterpret_cast<uint16_t *>(tabs + p.off_bmat);
        const int NP = row_base_np(p.n0), LDK = gen_base_ldk(p.n0);
        for (int e = threadIdx.x; e < NP * LDK; e += blockDim.x) {
            const int c = e / LDK, k = e - c * LDK, n = (c & ~7) + ((c >> 1) & 3) + 4 * (c & 1);     // column c of a tile is output n
            uint16_t v = 0;
            if (n < p.n0 && k < p.n0) v = ((p.hrow[n][k >> 5] >> (k & 31)) & 1u) ? 0xBF80 : 0x3F80;
            bm[e] = v;
        }
        uint32_t *hr = reinterpret_cast<uint32_t *>(tabs + p.off_hrow);
        for (int e = threadIdx.x; e < p.n0 * 3; e += blockDim.x) hr[e] = p.hrow[e / 3][e % 3];
        uint16_t *quad = reinterpret_cast<uint16_t *>(tabs + p.off_quad);
        for (int e = threadIdx.x; e < d / 4; e += blockDim.x) {
            const int k2 = (4 * e) / p.n0, c = 4 * e - k2 * p.n0;
            quad[e] = (uint16_t)((k2 << 5) | (c >> 2));
        }
    }
    griddep_wait();             // nothing above reads or writes global memory
    griddep_launch();
    if (permuted) row_load_perm(p, tabs, threadIdx.x, blockDim.x);
    __syncthreads();

    const uint32_t first = blockIdx.x * groups + group, stride = gridDim.x * groups;
    const uint32_t n_rows = first < p.T ? (p.T - first + stride - 1) / stride : 0u;
    const uint32_t n_iter = (p.T - blockIdx.x * groups + stride - 1) / stride;       // group 0 has the most rows
    auto load_row = [&](uint32_t it) {                                     // one thread of the row
        const uint32_t s = it % ROW_NSTAGE;
        mbar_expect_tx(full + s * 8, row_bytes);
        bulk_load(base + s * stage_bytes, p.x + (size_t)(first + it * stride) * d, row_bytes, full + s * 8);
    };
    if (tid == 0) {
        for (uint32_t s = 0; s < ROW_NSTAGE && s < n_rows; ++s) load_row(s);
    }

    // pass 1 constants (power of two): Hadamard operand, ldmatrix offset, relabelling signs, tile address
    const int cb = NP2 ? 0 : ROT != ROT_LOCAL ? 3 : min(p.log2b, 7) - 4, pm = (1 << cb) - 1, f_g = g & 3;
    uint32_t hb[2][2], lm0 = 0u, t_store = 0u;
    f32x2 sg2[4];
    if (!NP2) {
#pragma unroll
        for (int m = 0; m < 2; ++m) {
            const int col = 4 * (g >> 1) + (g & 1) + 2 * m;
            hb[m][0] = hadamard_bf16(2 * q, col) | (hadamard_bf16(2 * q + 1, col) << 16);
            hb[m][1] = hadamard_bf16(2 * q + 8, col) | (hadamard_bf16(2 * q + 9, col) << 16);
        }
        const int r8 = lane & 7, mi = lane >> 3;
        lm0 = (uint32_t)((r8 * 8 + ((mi & 1) ^ (r8 & 3))) * 32 + (((mi >> 1) ^ (r8 >> 2)) * 16));
        const float half_sign = ((g & 4) && q >= 2) ? -1.0f : 1.0f;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const float s = (__popc(k & f_g & pm) & 1) ? -half_sign : half_sign;
            sg2[k] = pack2(s, s);
        }
        // 16-byte pieces of slot s go to chunk s ^ (f & ~PM) of the lane group's 128 words; odd lane groups
        // flip bit 4 of the word (bit 7 of the position): the two of a quarter warp use different banks
        t_store = tile + (uint32_t)(warp * SEG_ELEMS + g * 128 + 4 * q) * 4u + (uint32_t)((f_g & ~pm) ^ (g & 1)) * 64u;
    }
    // quantiser constants: this lane's 32 outputs, their place in the tile, the order it reads them in
    // (blocks of 2048 and 4096 per token: the columns of pass 2, see row_columns)
    const uint32_t i0 = cols == 1 ? (uint32_t)((tid >> 7) * 4096 + (tid & 127))
                                  : cols == 2 ? (uint32_t)((tid >> 6) * 2048 + 2 * (tid & 63)) : (uint32_t)tid * 32u;
    const uint32_t t_read = tile + (NP2 ? i0 + (uint32_t)p.pad * ((uint32_t)tid / (uint32_t)(NP2 ? p.n0 / 4 : 1)) : i0) * 4u;
    const int rot = cols ? 0 : NP2 ? (lane & 7) : ((lane & 7) ^ (((tid >> 2) & 1) << 2));
    const float err = p.err_rel;

    for (uint32_t it = 0; it < n_iter; ++it) {
        const uint32_t stage = it % ROW_NSTAGE;
        const uint32_t row = first + it * stride;
        // everybody is past the previous row: its stage, the lists and the reduction words are free (whole-row blocks
        // per token: so they were at the last barrier of the previous row, and nothing has touched them since)
        if (!(wide && TOK)) __syncthreads();
        // (a row that is missing, or whose load never completed, runs through as zeros and stores nothing)
        bool have = it < n_rows;
        if (have && !mbar_wait_fast(full + stage * 8, (it / ROW_NSTAGE) & 1u)) {
            have = false;
            if (tid == 0) atomicOr(&g_perq_device_error, 1u);
        }
        const bool live = have && tid < d / 32;
        if (tid == 0) {
            if (it > 0 && it + ROW_NSTAGE - 1 < n_rows) load_row(it + ROW_NSTAGE - 1);
            ms->amax = ms->ahi = 0ull;
            ms->alo = ~0ull;
        }
        const uint32_t raw = base + stage * stage_bytes;
        const uint16_t *xs = reinterpret_cast<const uint16_t *>(smem + stage * stage_bytes);
        if (permuted) {
            row_gather(p, tabs, smem, raw, warp, lane);
            xs = reinterpret_cast<const uint16_t *>(smem + p.off_xs);
            if (NP2) __syncthreads(); else __syncwarp();
        }

        // ---- pass 1
        if (NP2) {
            switch (p.log2b) {
            case 6: row_base_pass<1, 2>(p, xs, tabs, tile, warp, warps, lane); break;
            case 7: row_base_pass<2, 2>(p, xs, tabs, tile, warp, warps, lane); break;
            case 8: row_base_pass<4, 2>(p, xs, tabs, tile, warp, warps, lane); break;
            case 9: row_base_pass<8, 1>(p, xs, tabs, tile, warp, warps, lane); break;
            default: row_base_pass<16, 1>(p, xs, tabs, tile, warp, warps, lane); break;
            }
            __syncthreads();
            row_base_stages(p, tile, tid);
            __syncthreads();
        } else {
            if (warp < segs) {
                f32x2 v[8][2];
                const uint32_t a0 = smem_u32(xs) + (uint32_t)warp * SEG_BYTES + lm0;
#pragma unroll
                for (int t = 0; t < 4; ++t) {
                    uint32_t a[4];
                    if (t & 2) ldmatrix_x4_at<128>(a, a0 ^ (uint32_t)((t & 1) << 6));
                    else ldmatrix_x4_at<0>(a, a0 ^ (uint32_t)((t & 1) << 6));
                    float c0[4], c1[4];
                    mma_bf16(c0, a, hb[0][0], hb[0][1]);
                    mma_bf16(c1, a, hb[1][0], hb[1][1]);
                    v[2 * t][0] = pack2(c0[0], c0[1]);
                    v[2 * t][1] = pack2(c1[0], c1[1]);
                    v[2 * t + 1][0] = pack2(c0[2], c0[3]);
                    v[2 * t + 1][1] = pack2(c1[2], c1[3]);
                }
#pragma unroll
                for (int t = 0; t < 3; ++t) {
                    if (t < cb) {
#pragma unroll
                        for (int s = 0; s < 8; ++s) {
                            if ((s & (1 << t)) == 0) {
#pragma unroll
                                for (int h = 0; h < 2; ++h) {
                                    const f32x2 x = v[s][h], y = v[s | (1 << t)][h];
                                    v[s][h] = add2(x, y);
                                    v[s | (1 << t)][h] = sub2(x, y);
                                }
                            }
                        }
                    }
                }
                if ((warp * 8 + g) * 128 < d) {               // (a partial last segment ends at a multiple of 128)
#pragma unroll
                    for (int s = 0; s < 8; ++s) {
                        const f32x2 x = mul2(v[s][0], sg2[s & 3]), y = mul2(v[s][1], sg2[s & 3]);
                        sts_v4f(t_store ^ (uint32_t)(s * 64), x.x, x.y, y.x, y.y);
                    }
                }
            }
            if (wide) __syncthreads(); else __syncwarp();
            // ---- pass 2: chunk-index bits
            if (ROT == ROT_LOCAL) {
                switch (p.log2b) {
                case 8: row_stages<1, true>(tile, d, 0, tid, nthr); break;
                case 9: row_stages<2, true>(tile, d, 0, tid, nthr); break;
                case 10: row_stages<3, true>(tile, d, 0, tid, nthr); break;
                default: break;
                }
            } else if (ROT == ROT_WIDE) {
                switch (p.log2b) {
                case 11: row_stages<4, false>(tile, d, 0, tid, nthr); break;
                case 12: row_stages<2, false>(tile, d, 0, tid, nthr); __syncthreads(); row_stages<3, false>(tile, d, 2, tid, nthr); break;
                case 13: row_stages<3, false>(tile, d, 0, tid, nthr); __syncthreads(); row_stages<3, false>(tile, d, 3, tid, nthr); break;
                default: row_stages<4, false>(tile, d, 0, tid, nthr); __syncthreads(); row_stages<3, false>(tile, d, 4, tid, nthr); break;
                }
            }
            if (!wide) __syncwarp(); else if (!cols) __syncthreads();
        }

        // ---- the lane's 32 outputs, and maxima
        f32x2 u[16];
        auto read_outputs = [&]() {
            if (cols) row_columns(tile, cols, tid < d / 32 ? i0 : 0u, u);
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                if (cols) {
                    if (!live) u[2 * j] = u[2 * j + 1] = pack2(0.0f, 0.0f);
                } else if (live) {
                    lds_v4f(t_read + 16u * (uint32_t)((j + lane) & 7), u[2 * j].x, u[2 * j].y, u[2 * j + 1].x, u[2 * j + 1].y);
                } else {
                    u[2 * j] = u[2 * j + 1] = pack2(0.0f, 0.0f);
                }
            }
        };
        read_outputs();
        float lm = 0.0f, hi = 0.0f, lo = 0.0f;
        if (MODE == ROW_ASYM) {
            hi = live ? u[0].x : -3.0e38f;
            lo = live ? u[0].x : 3.0e38f;
            if (live) {
#pragma unroll
                for (int m = 0; m < 16; ++m) { hi = fmaxf(fmaxf(hi, u[m].x), u[m].y); lo = fminf(fminf(lo, u[m].x), u[m].y); }
            }
            lm = live ? fmaxf(fabsf(hi), fabsf(lo)) : 0.0f;
        } else {
#pragma unroll
            for (int m = 0; m < 16; ++m) lm = max3abs(lm, u[m].x, u[m].y);
        }
        // largest magnitude of the Hadamard block (blocks of 16: of the lane's two), and of the row
        float bm = lm, a_row = 0.0f, hi_row = 0.0f, lo_row = 0.0f;
        if (!wide) {
            for (int o = 1; o < (1 << p.log2b) / 32; o <<= 1) bm = fmaxf(bm, __shfl_xor_sync(0xffffffffu, bm, o));
        }
        if (row_max) {
            if (MODE == ROW_ASYM) {
                const float wh = warp_max_f32(hi), wl = warp_min_f32(lo);
                if (lane == 0) { ms->wmax[warp] = wh; ms->wmin[warp] = wl; }
                __syncthreads();
                hi_row = warp_max_f32(lane < segs ? ms->wmax[lane & 15] : -3.0e38f);
                lo_row = warp_min_f32(lane < segs ? ms->wmin[lane & 15] : 3.0e38f);
                a_row = fmaxf(fabsf(hi_row), fabsf(lo_row));
            } else {
                const float wm = warp_max_f32(lm);
                if (lane == 0) ms->wmax[warp] = wm;
                __syncthreads();
                a_row = warp_max_f32(lane < segs ? ms->wmax[lane & 15] : 0.0f);
            }
            if (wide) bm = a_row;
        }

        // ---- scale of the lane's range in fp32, and the elements whose exact value it needs
        RowQuant Q;
        Q.magic = 12582920.0f;                // 1.5 * 2^23 + 8: low nibble of the sum = code + 8
        uint32_t cand = 0u;
        int Eb = 0;
        float a32 = a_row, thr = 0.0f;
        bool near = false, zero = false;
        float z32 = 0.0f, vmin = 0.0f, inv = 0.0f;
        if (MODE == ROW_GROUP) {
            a32 = lm;
            for (int o = 1; o < (1 << (p.log2g - 5)); o <<= 1) a32 = fmaxf(a32, __shfl_xor_sync(0xffffffffu, a32, o));
            if (wide || p.log2g > p.log2b) bm = fmaxf(bm, a32);
        }
        if (MODE == ROW_TOKEN || MODE == ROW_GROUP || MODE == ROW_FP4) {
            inv = row_inverse(a32);
            Q.mul = inv;
            const float eb = (MODE == ROW_GROUP) ? bm : a32;             // error reference of the range's maximum
            thr = a32 - 2.0f * err * eb - a32 * 2.4e-7f;
            // (a threshold at or below zero, a range within the error of its block: a value that is zero in fp32 can be the largest)
            if (a32 > 0.0f && lm >= thr) cand = row_reach(u, thr);
            // error of an element and of the fp32 maximum, in code units
            Q.tau = err * (bm * inv + eb * inv) + 4.0e-6f;
            if (MODE == ROW_FP4 && !(bm > 0.0f)) Q.tau = 0.0f;            // an all-zero block is exact
            if (MODE == ROW_FP4 && !(a32 > 0.0f)) Q.tau = 0.0f;
        } else if (MODE == ROW_MX) {
            const uint32_t bits = __float_as_uint(lm);
            const int e8 = (int)(bits >> 23);
            // E + 127 with E = floor(log2(a / sqrt(b))) - 2; the distance of a to a value where the floor changes
            float dist;
            a32 = lm;
            if (NP2) {
                const double yd = (double)lm / p.sqrt_b;
                int ex;
                const double mant = frexp(yd, &ex);                       // [0.5, 1)
                Eb = ex - 3 + 127;
                dist = (float)(fmin(mant - 0.5, 1.0 - mant) / mant) * lm;
            } else if ((p.log2b & 1) == 0) {
                const float lower = __uint_as_float(bits & 0x7f800000u);
                dist = fminf(lm - lower, 2.0f * lower - lm);
                Eb = e8 - p.log2b / 2 - 2;
            } else {
                dist = fabsf(lm - __uint_as_float((bits & 0x7f800000u) | 0x3504f3u));
                Eb = e8 - (p.log2b - 1) / 2 - 3 + ((bits & 0x7fffffu) >= 0x3504f4u ? 1 : 0);
            }
            const float tol = 2.0f * err * bm + lm * 4.8e-7f;
            near = lm > 0.0f && (dist <= tol || e8 == 0);
            thr = lm - tol;
            if (near) cand = row_reach(u, thr);
        } else {
            const float e_abs = a_row * (2.0f * err + 2.4e-7f);
            const bool some = a_row > 0.0f;
            // (extremes that are equal in fp32 need not be: then every element is a candidate and in doubt)
            const bool flat = some && !(hi_row > lo_row);
            if (some && live && (hi >= hi_row - e_abs || lo <= lo_row + e_abs)) {
#pragma unroll
                for (int m = 0; m < 16; ++m) {
                    cand |= (u[m].x >= hi_row - e_abs || u[m].x <= lo_row + e_abs ? 1u : 0u) << (2 * m);
                    cand |= (u[m].y >= hi_row - e_abs || u[m].y <= lo_row + e_abs ? 2u : 0u) << (2 * m);
                }
            }
            // 15 / (hi - lo); the range itself may overflow, and see row_inverse
            inv = (some && !flat) ? fminf(__fdividef(1.875f, 0.125f * hi_row - 0.125f * lo_row), 3.0e38f) : 0.0f;
            Q.mul = inv;
            const float ar = flat ? 3.0e38f : fminf(a_row * inv, 3.0e38f);    // |y|max in steps (7.5 or more)
            vmin = lo_row * inv;
            z32 = rintf(vmin);
            // errors of an element (err * |y|max) and of the step (2 err |y|max / range, relative)
            Q.tau = err * ar * (1.0f + ar * (2.0f / 15.0f)) + (ar + 8.0f) * 6.0e-7f;
            near = some && !(fabsf(vmin - z32) <= 0.5f - Q.tau);
        }
        // ---- integers and E2M1 per token do not wait for the exact scale: codes now, doubtful ones listed
        uint32_t cw[4], tie = 0u;
        const bool quantise_first = MODE == ROW_TOKEN || MODE == ROW_FP4 || MODE == ROW_GROUP;
        if (quantise_first) {
            if (row_quantise<MODE>(u, Q, cw)) tie = row_tie_bits<MODE>(u, Q);
        }

        if (quantise_first) {
            if (!live) tie = 0u;
            row_unrotate(cw, rot);
        }
        double s64 = 0.0, z64 = 0.0;
        double a_ex = 0.0, hi_ex = 0.0, lo_ex = 0.0;                      // exact maximum of the lane's range; row extremes
        const RowLane place = {tile, i0, t_read, rot, warp, tid};
        // blocks inside a segment, many candidates or doubtful elements: are the segment's fp32 outputs exact?  (asked once)
        bool asked = false, exact32 = false;
        auto ask = [&](uint32_t bits) {
            if (!asked && __any_sync(0xffffffffu, __popc(bits) > ROW_MANY)) {
                asked = true;
                exact32 = row_span_exact(row_segment_span(xs + warp * SEG_ELEMS, d - warp * SEG_ELEMS, lane));
                if (!quantise_first) read_outputs();
            }
        };
        if (MODE == ROW_TOKEN || MODE == ROW_FP4 || MODE == ROW_ASYM) {
            hi_ex = -1.7976931348623157e308;
            lo_ex = 1.7976931348623157e308;
            uint32_t want = cand;
            if (wide) {
                // candidates and doubtful elements in one round (ties are settled once no candidate is left)
                int slot = 0, tslot = 0;
                const int took = row_append(ms, 0, want, i0, rot, cols, slot);
                const int ttook = row_append(ms, 1, tie, i0, rot, cols, tslot);
                __syncthreads();
                const int total = (int)ms->cnt[0], n = min(total, ROW_CAP);
                const int ttotal = (int)ms->cnt[1], tn = min(ttotal, ROW_CAP);
                const bool last = total <= ROW_CAP;
                row_all_partials<NP2>(p, xs, tabs, smem, n, tn, warp, lane);
                const bool more = __syncthreads_or(!last || ttotal > ROW_CAP);          // (of any row of the CTA)
                if (tid == 0) ms->cnt[0] = ms->cnt[1] = 0u;
                if (more || tid == 0 || ttook > 0 || MODE == ROW_ASYM) {
                    for (int e = 0; e < n; ++e) {
                        const double v = row_sum_parts(ms, e);
                        a_ex = fmax(a_ex, fabs(v));
                        hi_ex = fmax(hi_ex, v);
                        lo_ex = fmin(lo_ex, v);
                    }
                }
                if (last && ttook > 0) {
                    if (MODE == ROW_FP4) s64 = a_ex / p.sqrt_b / 7.0;
                    for (int t = 0; t < ttook; ++t) {
                        const int e = __ffs(tie) - 1;
                        tie &= tie - 1;
                        const double v = row_sum_parts(ms, tslot + t);
                        row_patch(cw, e, rot, MODE == ROW_TOKEN ? row_int4_code<true>(v, a_ex, Q.mul, p.sqrt_b)
                                                                : row_exact_code<MODE>(v, p.sqrt_b, s64, 0.0, 0));
                    }
                }
                if (more) {
                    for (int t = 0; t < took; ++t) want &= want - 1;
                    if (MODE == ROW_ASYM) {
                        (void)row_many_token<MODE, NP2, cols>(p, xs, tabs, smem, place, want, 0u, make_uint4(0u, 0u, 0u, 0u), 0.0f, 0.0, hi_ex, lo_ex);
                        hi_ex = order_value(ms->ahi);
                        lo_ex = order_value(ms->alo);
                        read_outputs();                        // (again, so that the call has nothing to keep)
                    } else {
                        const uint4 w = row_many_token<MODE, NP2, cols>(p, xs, tabs, smem, place, want, tie, make_uint4(cw[0], cw[1], cw[2], cw[3]),
                                                                        Q.mul, a_ex, hi_ex, lo_ex);
                        cw[0] = w.x; cw[1] = w.y; cw[2] = w.z; cw[3] = w.w;
                        tie = 0u;
                        if (tid == 0) a_ex = __longlong_as_double((long long)ms->amax);
                    }
                }
            } else {
                ask(want);
                if (exact32 && want != 0u) {                  // (a lane with a candidate holds its own extremes among them)
                    a_ex = (double)lm;
                    hi_ex = (double)hi + 0.0;
                    lo_ex = (double)lo + 0.0;
                    want = 0u;
                }
                unsigned cl = __ballot_sync(0xffffffffu, want != 0u);
                while (cl) {
                    const int src = __ffs(cl) - 1;
                    cl &= cl - 1;
                    uint32_t ws = __shfl_sync(0xffffffffu, want, src);
                    const uint32_t is = __shfl_sync(0xffffffffu, i0, src);
                    const int rs = __shfl_sync(0xffffffffu, rot, src);
                    while (ws) {
                        const int e = __ffs(ws) - 1;
                        ws &= ws - 1;
                        const double v = row_exact_warp(xs, row_position(is, rs, 0, e), p.log2b, lane);
                        a_ex = fmax(a_ex, fabs(v));
                        hi_ex = fmax(hi_ex, v);
                        lo_ex = fmin(lo_ex, v);
                    }
                }
                if ((lane == 0 || exact32) && hi_ex >= lo_ex) {
                    if (MODE == ROW_ASYM) {
                        atomicMax(&ms->ahi, order_key(hi_ex));
                        atomicMin(&ms->alo, order_key(lo_ex));
                    } else {
                        atomicMax(&ms->amax, (unsigned long long)__double_as_longlong(a_ex));
                    }
                }
                __syncthreads();
                a_ex = __longlong_as_double((long long)ms->amax);
                if (MODE == ROW_ASYM) {
                    hi_ex = order_value(ms->ahi);
                    lo_ex = order_value(ms->alo);
                }
            }
            if (MODE == ROW_ASYM && !(a_row > 0.0f)) hi_ex = lo_ex = 0.0;
        } else if (MODE == ROW_GROUP) {
            // the exact maximum of every range: its candidates, four lanes to a sum (long blocks: CTA-wide)
            uint32_t want = cand;
            if (wide) {
                int slot = 0;
                const int took = row_append(ms, 0, want, i0, rot, cols, slot);
                __syncthreads();
                const int total = (int)ms->cnt[0], n = min(total, ROW_CAP);
                row_all_partials<NP2>(p, xs, tabs, smem, n, 0, warp, lane);
                const bool more = __syncthreads_or(total > ROW_CAP);
                if (tid == 0) ms->cnt[0] = 0u;
                for (int t = 0; t < took; ++t) { want &= want - 1; a_ex = fmax(a_ex, fabs(row_sum_parts(ms, slot + t))); }
                if (more) a_ex = row_many_max<NP2>(p, xs, tabs, smem, place, want, cand != 0u, lm, a_ex, total > 2 * (d >> p.log2g));
            } else {
                ask(want);
                if (exact32 && want != 0u) { a_ex = (double)lm; want = 0u; }
                // (all quads step together; the lanes of a quad take turns)
                while (__any_sync(0xffffffffu, want != 0u)) {
                    const unsigned have = (__ballot_sync(0xffffffffu, want != 0u) >> (lane & 28)) & 0xFu;
                    const int src = have ? __ffs(have) - 1 : 0;
                    uint32_t pos = (uint32_t)warp * SEG_ELEMS;
                    if ((lane & 3) == src && want) pos = row_position(i0, rot, 0, __ffs(want) - 1);
                    pos = __shfl_sync(0xffffffffu, pos, (lane & 28) | src);
                    const double v = row_exact_quad(xs, pos, p.log2b, lane);
                    if ((lane & 3) == src && want) { want &= want - 1; a_ex = fmax(a_ex, fabs(v)); }
                }
            }
            for (int o = 1; o < (1 << (p.log2g - 5)); o <<= 1) a_ex = fmax(a_ex, __shfl_xor_sync(0xffffffffu, a_ex, o));
        } else {
            // MX: exact exponents of the groups near a boundary; a group whose exact values are all zero
            zero = !(lm > 0.0f);
            if (wide ? __syncthreads_or(near) : __any_sync(0xffffffffu, near)) {
                uint32_t want = cand;
                if (wide) {
                    int slot = 0;
                    const int took = row_append(ms, 0, want, i0, rot, cols, slot);
                    __syncthreads();
                    const int total = (int)ms->cnt[0], n = min(total, ROW_CAP);
                    row_all_partials<NP2>(p, xs, tabs, smem, n, 0, warp, lane);
                    const bool more = __syncthreads_or(total > ROW_CAP);
                    if (tid == 0) ms->cnt[0] = 0u;
                    for (int t = 0; t < took; ++t) { want &= want - 1; a_ex = fmax(a_ex, fabs(row_sum_parts(ms, slot + t))); }
                    if (more) {
                        a_ex = row_many_max<NP2>(p, xs, tabs, smem, place, want, cand != 0u, lm, a_ex, true);
                        read_outputs();
                    }
                } else {
                    ask(want);
                    if (exact32 && want != 0u) { a_ex = (double)lm; want = 0u; }
                    while (__any_sync(0xffffffffu, want != 0u)) {
                        const unsigned have = (__ballot_sync(0xffffffffu, want != 0u) >> (lane & 28)) & 0xFu;
                        const int src = have ? __ffs(have) - 1 : 0;
                        uint32_t pos = (uint32_t)warp * SEG_ELEMS;
                        if ((lane & 3) == src && want) pos = row_position(i0, rot, 0, __ffs(want) - 1);
                        pos = __shfl_sync(0xffffffffu, pos, (lane & 28) | src);
                        const double v = row_exact_quad(xs, pos, p.log2b, lane);
                        if ((lane & 3) == src && want) { want &= want - 1; a_ex = fmax(a_ex, fabs(v)); }
                    }
                }
                if (near) {
                    int ex;
                    (void)frexp(a_ex / p.sqrt_b, &ex);
                    Eb = ex - 3 + 127;
                    zero = a_ex == 0.0;       // (the fp32 values of a group that cancels exactly are rounding noise)
                }
            }
        }

        // ---- stored scales; formats that needed the exact ones quantise here
        if (MODE == ROW_TOKEN || MODE == ROW_FP4) {
            if (tid == 0 && have) reinterpret_cast<float *>(p.out_scales)[row] = row_scale(a_ex, p.inv_7_sqrt_b, p.sqrt_b, 7.0);
        } else if (MODE == ROW_GROUP) {
            if (live && (tid & ((1 << (p.log2g - 5)) - 1)) == 0)
                reinterpret_cast<float *>(p.out_scales)[(size_t)row * (d >> p.log2g) + (i0 >> p.log2g)] =
                    row_scale(a_ex, p.inv_7_sqrt_b, p.sqrt_b, 7.0);
        } else if (MODE == ROW_ASYM) {
            // the fp32 zero point stands unless its rounding was in doubt (near: the same in every thread)
            float s32 = 0.0f;
            bool apart = false;
            if (tid == 0) {
                const double s = (hi_ex - lo_ex) * p.inv_15_sqrt_b;
                s32 = (float)(s * (1.0 - 0x1p-48));
                apart = hi_ex < 0.0 || lo_ex > 0.0 || s32 != (float)(s * (1.0 + 0x1p-48));
            }
            if (near || apart) {
                s64 = (hi_ex / p.sqrt_b - lo_ex / p.sqrt_b) / 15.0;
                z64 = (s64 == 0.0) ? 0.0 : rint(lo_ex / p.sqrt_b / s64);
                s32 = (float)s64;
                if (near) z32 = (float)z64;
            }
            if (tid == 0 && have) reinterpret_cast<float2 *>(p.out_scales)[row] = make_float2(s32, z32);
            Q.magic = 12582912.0f - z32;                                  // 1.5 * 2^23 - z
            if (row_quantise<MODE>(u, Q, cw)) tie = row_tie_bits<MODE>(u, Q);
        } else {
            Eb = min(max(Eb, 0), 254);
            uint32_t byte = (uint32_t)Eb;
            if (NP2) Q.mul = (float)(scalbn(1.0, 127 - Eb) / p.sqrt_b);
            else if ((p.log2b & 1) == 0) Q.mul = __uint_as_float((uint32_t)min(max(254 - Eb - p.log2b / 2, 1), 254) << 23);
            else Q.mul = __uint_as_float((uint32_t)min(max(254 - Eb - (p.log2b - 1) / 2, 1), 254) << 23) * 0.70710678118654752f;
            if (zero) { Eb = 0; Q.mul = 0.0f; byte = 0u; }
            // (an all-zero block is exact, and so is a group whose candidates were all zero: no window, codes 0)
            Q.tau = (bm > 0.0f && !(near && zero)) ? 2.0f * err * bm * Q.mul + 2.0e-6f : 0.0f;
            if (live) (reinterpret_cast<uint8_t *>(p.out_scales))[(size_t)row * (d >> 5) + tid] = (uint8_t)byte;
            if (row_quantise<MODE>(u, Q, cw)) tie = row_tie_bits<MODE>(u, Q);
        }
        if (!quantise_first) {
            if (!live) tie = 0u;
            row_unrotate(cw, rot);
        }

        // ---- exact codes of the doubtful elements (whole-row integers and E2M1 per token: done above)
        if (wide ? (MODE != ROW_TOKEN && MODE != ROW_FP4 && __syncthreads_or(tie != 0u)) : __any_sync(0xffffffffu, tie != 0u)) {
            if (MODE == ROW_FP4) s64 = a_ex / p.sqrt_b / 7.0;
            if (MODE == ROW_ASYM) {
                s64 = (hi_ex / p.sqrt_b - lo_ex / p.sqrt_b) / 15.0;
                z64 = (s64 == 0.0) ? 0.0 : rint(lo_ex / p.sqrt_b / s64);
            }
            if (wide) {
                int slot = 0;
                const int took = row_append(ms, 1, tie, i0, rot, cols, slot);
                __syncthreads();
                const int total = (int)ms->cnt[1], n = min(total, ROW_CAP);
                row_all_partials<NP2>(p, xs, tabs, smem, 0, n, warp, lane);
                const bool more = __syncthreads_or(total > ROW_CAP);
                if (tid == 0) ms->cnt[1] = 0u;
                for (int t = 0; t < took; ++t) {
                    const int e = __ffs(tie) - 1;
                    tie &= tie - 1;
                    const double v = row_sum_parts(ms, slot + t);
                    row_patch(cw, e, rot, MODE == ROW_GROUP ? row_int4_code<false>(v, a_ex, Q.mul, p.sqrt_b)
                                                            : row_exact_code<MODE>(v, p.sqrt_b, s64, z64, Eb - 127));
                }
                if (more) {
                    const uint4 w = row_many_ties<MODE, NP2, cols>(p, xs, tabs, smem, place, tie, make_uint4(cw[0], cw[1], cw[2], cw[3]), Q.mul,
                                                                   a_ex, s64, z64, Eb - 127);
                    cw[0] = w.x; cw[1] = w.y; cw[2] = w.z; cw[3] = w.w;
                }
            } else {
                ask(tie);
                if (exact32 && tie) {
                    const uint4 w = row_settle_warp<MODE>(make_uint4(cw[0], cw[1], cw[2], cw[3]), tie, place, a_ex, Q.mul, p.sqrt_b, s64, z64, Eb - 127);
                    cw[0] = w.x; cw[1] = w.y; cw[2] = w.z; cw[3] = w.w;
                    tie = 0u;
                }
                unsigned tl = __ballot_sync(0xffffffffu, tie != 0u);
                while (tl) {
                    const int src = __ffs(tl) - 1;
                    tl &= tl - 1;
                    uint32_t ts = __shfl_sync(0xffffffffu, tie, src);
                    const uint32_t is = __shfl_sync(0xffffffffu, i0, src);
                    const int rs = __shfl_sync(0xffffffffu, rot, src);
                    while (ts) {
                        const int e = __ffs(ts) - 1;
                        ts &= ts - 1;
                        const double v = row_exact_warp(xs, row_position(is, rs, 0, e), p.log2b, lane);
                        if (lane == src)
                            row_patch(cw, e, rot, MODE == ROW_TOKEN || MODE == ROW_GROUP ? row_int4_code<MODE == ROW_TOKEN>(v, a_ex, Q.mul, p.sqrt_b)
                                                                                       : row_exact_code<MODE>(v, p.sqrt_b, s64, z64, Eb - 127));
                    }
                }
            }
        }
        if (wide && MODE == ROW_ASYM) __syncthreads();          // (the tie round may have been the last to use the lists)
        uint32_t at = (uint32_t)tid * 16u;
        if (cols) {
            row_transpose_codes(cw, cols, lane);
            at = cols == 1 ? (uint32_t)((tid >> 7) * 4096 + lane * 128 + (warp & 3) * 32) / 2u
                           : (uint32_t)((tid >> 6) * 2048 + (lane & 15) * 128 + (warp & 1) * 64 + (lane >> 4) * 32) / 2u;
        }
        if (live) *reinterpret_cast<uint4 *>(p.out_codes + (size_t)row * (d / 2) + at) = make_uint4(cw[0], cw[1], cw[2], cw[3]);
    }
}

// -------------------------------------------------------------------------------------------- long blocks, many ranges
//
// INT4 per range of 32 .. 1024 inside Hadamard blocks of 256 .. 16384: every range needs the exact maximum of its
// outputs, each of which is a sum over the whole block.  For b = 2048 and ranges of 128 that is 16 terms per
// element of the row (157 us for 4096 x 2048 in the general kernel, 87 with the sums shared by a CTA, two thirds of it
// these sums); the butterfly itself in fp64 is 11 additions per element and makes EVERY output exact, so this kernel
// rotates in fp64 and rounds its outputs to fp32 for the quantiser (31.5 us).  Maxima come from the fp64 values; the rounding window is the rounding to fp32 alone.
//
// A warp owns 1024 positions.  Lane l starts with the values at 32 m + l, combined over the block's segments while
// they are converted (2^896 completes the conversion, see bf16_bits_to_f64, and carries the sign), rotates index
// bits 5 .. 9 in registers, regroups through the warp's tile (rows of 32 + 2 doubles: conflict-free both ways;
// half a segment at a time, so that the tile takes 4.3 KB) and rotates bits 0 .. 4 of 32 consecutive positions.

constexpr int ROW64_REGS = 128;
constexpr int ROW64_SM_WARPS = 65536 / (ROW64_REGS * 32);
constexpr int ROW64_CTA_WARPS = 2;
constexpr int ROW64_LD = 34;                                   // doubles per tile row
constexpr int ROW64_TILE = 16 * ROW64_LD * 8;                  // bytes per warp

__device__ __forceinline__ void row64_stage(double (&v)[32], int t)
{
#pragma unroll
    for (int m = 0; m < 32; ++m) {
        if ((m & t) == 0) {
            const double a = v[m], c = v[m | t];
            v[m] = a + c;
            v[m | t] = a - c;
        }
    }
}

__global__ void __maxnreg__(ROW64_REGS) perq_row64_kernel(const __grid_constant__ RowParams p)
{
    extern __shared__ __align__(128) unsigned char r64_raw[];
    unsigned char *tabs = r64_raw + ((1024u - (smem_u32(r64_raw) & 1023u)) & 1023u);
    const int lane = threadIdx.x & 31, group = (int)(threadIdx.x >> 5) / p.row_warps;        // (rows in step, as above)
    const int warp = (int)(threadIdx.x >> 5) - group * p.row_warps, tid = warp * 32 + lane, nthr = p.row_warps * 32;
    const int groups = (int)blockDim.x / nthr;
    unsigned char *smem = tabs + p.off_group + group * p.group_bytes;
    const int d = p.d, segs = nthr >> 5, log2r = max(p.log2b - 10, 0);
    const bool permuted = p.perm != nullptr;
    unsigned long long *full_gen = reinterpret_cast<unsigned long long *>(smem + p.off_misc);
    const uint32_t base = smem_u32(smem), full = smem_u32(full_gen);
    const uint32_t stage_bytes = (uint32_t)segs * SEG_BYTES, row_bytes = (uint32_t)d * 2u;
    double *tile = reinterpret_cast<double *>(smem + p.off_tile + warp * ROW64_TILE);

    // (as mbar_init and mbar_init_fence, in one statement and with thread 0's fence a second time: written the plain way the
    // compiler spills 8 bytes more, 33.1 against 32.1 us for 4096 x 2048, b = d, per 128)
    if (tid < ROW_NSTAGE)
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n\tfence.mbarrier_init.release.cluster;" ::"r"(full + tid * 8) : "memory");
    if (tid == 0) mbar_init_fence();
    griddep_wait();             // nothing above reads or writes global memory
    griddep_launch();
    if (permuted) row_load_perm(p, tabs, threadIdx.x, blockDim.x);
    __syncthreads();
    const uint32_t first = blockIdx.x * groups + group, stride = gridDim.x * groups;
    const uint32_t n_rows = first < p.T ? (p.T - first + stride - 1) / stride : 0u;
    const uint32_t n_iter = (p.T - blockIdx.x * groups + stride - 1) / stride;       // group 0 has the most rows
    auto load_row = [&](uint32_t it) {                                     // one thread of the row
        const uint32_t s = it % ROW_NSTAGE;
        mbar_expect_tx(full + s * 8, row_bytes);
        bulk_load(base + s * stage_bytes, p.x + (size_t)(first + it * stride) * d, row_bytes, full + s * 8);
    };
    if (tid == 0) {
        for (uint32_t s = 0; s < ROW_NSTAGE && s < n_rows; ++s) load_row(s);
    }
    const uint32_t i0 = (uint32_t)tid * 32u;
    const int wb = warp & ~((1 << log2r) - 1), wl = warp - wb;            // first segment of the block, place in it

    for (uint32_t it = 0; it < n_iter; ++it) {
        const uint32_t stage = it % ROW_NSTAGE, row = first + it * stride;
        __syncthreads();                       // everybody is past the previous row
        bool have = it < n_rows;
        if (have && !mbar_wait_fast(full + stage * 8, (it / ROW_NSTAGE) & 1u)) {
            have = false;
            if (tid == 0) atomicOr(&g_perq_device_error, 1u);
        }
        const bool live = have && i0 < (uint32_t)d;
        if (tid == 0 && it > 0 && it + ROW_NSTAGE - 1 < n_rows) load_row(it + ROW_NSTAGE - 1);
        const uint16_t *xs = reinterpret_cast<const uint16_t *>(smem + stage * stage_bytes);
        if (permuted) {
            row_gather(p, tabs, smem, base + stage * stage_bytes, warp, lane);
            xs = reinterpret_cast<const uint16_t *>(smem + p.off_xs);
            if (log2r > 0) __syncthreads(); else __syncwarp();
        }
        double v[32];
#pragma unroll
        for (int m = 0; m < 32; ++m) v[m] = 0.0;
        for (int w = 0; w < (1 << log2r); ++w) {
            const double c = (__popc(w & wl) & 1) ? -0x1p896 : 0x1p896;
            const int16_t *src = reinterpret_cast<const int16_t *>(xs) + (wb + w) * SEG_ELEMS + lane;
#pragma unroll
            for (int m = 0; m < 32; ++m) {
                const uint32_t h = (uint32_t)(int)src[32 * m];          // (sign-extended: the shift puts the sign into bit 31)
                v[m] = fma(__hiloint2double((int)((h << 13) & 0x8fffffffu), 0), c, v[m]);
            }
        }
        row64_stage(v, 1);
        row64_stage(v, 2);
        row64_stage(v, 4);
        if (p.log2b > 8) row64_stage(v, 8);
        if (p.log2b > 9) row64_stage(v, 16);
        // regroup: rows m of half a segment, then lanes 16 h .. 16 h + 15 take a row each
        double u64[32];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            __syncwarp();
#pragma unroll
            for (int m = 0; m < 16; ++m) tile[m * ROW64_LD + lane] = v[16 * h + m];
            __syncwarp();
            if ((lane >> 4) == h) {
#pragma unroll
                for (int m = 0; m < 32; m += 2) {
                    const double2 x = *reinterpret_cast<const double2 *>(tile + (lane & 15) * ROW64_LD + m);
                    u64[m] = x.x;
                    u64[m + 1] = x.y;
                }
            }
        }
        row64_stage(u64, 1);
        row64_stage(u64, 2);
        row64_stage(u64, 4);
        row64_stage(u64, 8);
        row64_stage(u64, 16);
        // exact maximum of the lane's range: high words, then low words of those that share the largest
        uint32_t mh = 0u, ml = 0u;
#pragma unroll
        for (int m = 0; m < 32; ++m) mh = max(mh, (uint32_t)__double2hiint(u64[m]) & 0x7fffffffu);
        for (int o = 1; o < (1 << (p.log2g - 5)); o <<= 1) mh = max(mh, __shfl_xor_sync(0xffffffffu, mh, o));
#pragma unroll
        for (int m = 0; m < 32; ++m) {
            if (((uint32_t)__double2hiint(u64[m]) & 0x7fffffffu) == mh) ml = max(ml, (uint32_t)__double2loint(u64[m]));
        }
        for (int o = 1; o < (1 << (p.log2g - 5)); o <<= 1) ml = max(ml, __shfl_xor_sync(0xffffffffu, ml, o));
        const double a_ex = __hiloint2double((int)mh, (int)ml);
        f32x2 u[16];
#pragma unroll
        for (int m = 0; m < 16; ++m) u[m] = pack2((float)u64[2 * m], (float)u64[2 * m + 1]);
        if (live && (tid & ((1 << (p.log2g - 5)) - 1)) == 0)
            reinterpret_cast<float *>(p.out_scales)[(size_t)row * (d >> p.log2g) + (i0 >> p.log2g)] =
                row_scale(a_ex, p.inv_7_sqrt_b, p.sqrt_b, 7.0);
        const float a32 = (float)a_ex;
        RowQuant Q;
        Q.magic = 12582920.0f;
        Q.mul = row_inverse(a32);
        Q.tau = 14.0f * TWO_M24 + 4.0e-6f;
        uint32_t cw[4], tie = 0u;
        if (row_quantise<ROW_GROUP>(u, Q, cw)) tie = row_tie_bits<ROW_GROUP>(u, Q);
        if (!live) tie = 0u;
        unsigned tl = __ballot_sync(0xffffffffu, tie != 0u);
        while (tl) {
            const int src = __ffs(tl) - 1;
            tl &= tl - 1;
            uint32_t ts = __shfl_sync(0xffffffffu, tie, src);
            const uint32_t is = __shfl_sync(0xffffffffu, i0, src);
            while (ts) {
                const int e = __ffs(ts) - 1;
                ts &= ts - 1;
                const double x = row_exact_warp(xs, is + e, p.log2b, lane);
                if (lane == src) row_patch(cw, e, 0, row_int4_code<true>(x, a_ex, Q.mul, p.sqrt_b));
            }
        }
        if (live) *reinterpret_cast<uint4 *>(p.out_codes + (size_t)row * (d / 2) + (size_t)tid * 16) = make_uint4(cw[0], cw[1], cw[2], cw[3]);
    }
}

}  // namespace perq
