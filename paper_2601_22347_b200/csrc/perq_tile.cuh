// Tile kernel: Hadamard blocks of 16 .. 128 on the fifth-generation tensor cores.
//
// A tile is 128 pieces of 128 adjacent channels.  Its rotation is one contraction, D[piece][column] = X H: the tile
// lies in shared memory as the K-major operand with 128-byte swizzle, H_64 beside it as the other operand (its
// leading 16 and 32 rows and columns are H_16 and H_32; H_128 is four H_64, one of them negated), the fp32 result in
// tensor memory.  The operand holds +-1/2, so that everything below is in halves of the unnormalised outputs: the sum of
// some inputs of a block can be 1.75 times its largest output, which may lie just below 2^128.
//
// What follows the rotation has a piece per lane: a warp reads 32 columns of its 32 pieces with one load, so that the
// maxima of MX groups and of ranges of 128, the rounding, the packing of 32 codes and the test for doubtful elements
// are all lane-local, without a shuffle; per-token scales meet once per tile.  The kernels that rotate in registers (a
// lane holds four adjacent outputs of eight chunks) spend 270 to 750 warp instructions on 1024 elements, this one 220 to 390.
// 65536 x 4096, b = 32, MXFP4: 110 us (floor 105; 135 in registers).  What bounds calls of ordinary size is what they pay
// once: 5 to 8 us of set-up, first load, last tile and last batch of records.
//
// Exactness rules as in perq_generic.cuh: |u32 - u| <= err * (largest |u32| of the block); every value that decides an
// output bit and lies within that bound of a boundary is summed again in fp64 from the bf16 inputs.
// err: a step adds 16 products to the accumulator, cuts all terms toward zero at 2^(e-25), e the exponent of the largest, and
// the sum at 2^(e-23) of its own (measured: a model of that gives the same bits on inputs of 4 to 26 binades).  With T the
// largest term and P the sum, a step loses 8 T + 2 P at most, in 2^-24 (the first, of 15 terms, 7.5 T + 2 P).  In units of the
// block's largest output T is at most 1 for an input (Parseval) and P, after m steps, what the Walsh coefficients of the first
// 16 m inputs' indicator add up to: 1, 1, 1.5, 1, 1.5, 1.5, 1.75, 1.  In all 9.5, 19.5, 44.5 and 102 for b = 16, 32, 64, 128
// (tile_err).  Rows that lose 64 of the 102 are among the tests; gaussian and heavy-tailed ones lose 3, with one
// input 1000 times the others 4, 20000 times 12 (4000 pieces each, by the model).
// The warps that quantise only note these places (candidates for a row's maximum, doubtful elements).  One warp turns
// the notes of a tile into records, two others settle records in batches, one per lane, from the inputs in global
// memory: they store the rows' scales and mend codes.  With the sums inside the quantising warps a tile of token rows took
// those 7000 cycles instead of 5000, 3000 of them waiting for one sum after another.  (Ranges of 128 have a maximum per
// lane: those are summed in place.)
#pragma once
#include <cuda.h>

#include "perq_row.cuh"

namespace perq {

constexpr int TILE_PIECES = 128;              // pieces of a tile, one per lane of tensor memory
constexpr int TILE_ROW_CAP = 32;              // token rows per tile
constexpr uint32_t TILE_H_BYTES = 64 * 128;   // H_64 as an operand
__host__ __device__ constexpr float tile_err(int log2b) { return (log2b == 4 ? 16.0f : log2b == 5 ? 20.0f : log2b == 6 ? 45.0f : 103.0f) * 0x1p-24f; }

struct TileParams {
    const uint16_t *x;
    uint8_t *out_codes;
    void *out_scales;
    uint32_t pieces;         // of the call: T * d / 128
    uint32_t tiles;
    int tile_pieces;         // pieces per tile: 128, or whole rows
    int row_pieces;          // d / 128
    int wide_store;          // codes are 32-byte aligned
    float err;
    double sqrt_b, inv_sqrt_b, inv_7_sqrt_b;         // (tile kernel: sqrt(b) / 2, what its halved outputs are divided by)
};

// fp32 maxima (bits) of token rows that lie in several warps; two tiles' worth, used in turn.
struct TileRows {
    uint32_t mx[2][TILE_ROW_CAP];
};

// What is left to settle of a tile: places, and what their codes depend on.
constexpr int TILE_JOBS = 96;
constexpr int TILE_TIES = 4;                  // notes of a lane and 32 columns
// a job: kind (1 bit), row of the tile (5, from bit 20), code as stored (4, from bit 16), column (7), piece (7)
// Pieces with more places than are worth a note each are left to their lanes (tile_put_maximum, tile_requantise).
enum TileFlat : uint32_t { FLAT_ROWS = 1u, FLAT_CODES = 2u };          // maxima that are in `ex` only; codes
enum TileJob : uint32_t { JOB_MAX = 0u << 30, JOB_TIE = 1u << 30 };     // candidates in a quad; an element
struct TileNotes {
    unsigned long long ex[TILE_ROW_CAP];                               // exact maxima of token rows (bits)
    unsigned long long aux[TILE_PIECES];                               // per piece: exact maximum (ranges), exponents (MX)
    uint32_t settled[4];                                               // pieces whose codes are exact already
    uint32_t flat, count;                                              // (more notes than fit: count goes on)
    uint32_t job[TILE_JOBS];
};
// A note and what its code depends on: exponents or the exact maximum (MX, ranges), or the quad that holds the maximum of
// the element's row (piece and column).
struct TileRecord {
    uint32_t job, piece;
    uint32_t aux[2];
};
constexpr int TILE_RECORDS = 64;              // per batch
constexpr uint32_t TILE_LAST = 1u << 30;

// A barrier of `threads` threads at which they agree: whether it is ok for all of them.  (Each warp polls a bounded wait by itself,
// so that one may have run out and another not: none may go on to a barrier that the others do not reach.)
__device__ __forceinline__ bool named_barrier_all(int id, int threads, bool ok)
{
    uint32_t all;
    asm volatile("{ .reg .pred p, q; setp.ne.u32 p, %1, 0; bar.red.and.pred q, %2, %3, p; selp.u32 %0, 1, 0, q; }"
                 : "=r"(all) : "r"((uint32_t)ok), "r"(id), "r"(threads) : "memory");
    return all != 0u;
}

// -------------------------------------------------------------------------------------------- tensor core and TMA

// Operand descriptor, low and high word: K-major, 128-byte swizzle, eight rows of 128 bytes to an atom, 1024 bytes from
// one to the next.
__device__ __forceinline__ uint32_t tile_desc(uint32_t addr) { return ((addr >> 4) & 0x3fffu) | (1u << 16); }
constexpr uint32_t TILE_DESC_HI = 64u | (1u << 14) | (2u << 29);
// bf16 x bf16 -> fp32, both operands K-major, 128 rows, n columns
__host__ __device__ constexpr uint32_t tile_idesc(int n) { return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | (8u << 24); }

__device__ __forceinline__ void tile_mma(uint32_t d, uint32_t a, uint32_t b, uint32_t idesc, bool accumulate)
{
    asm volatile("{ .reg .pred p; .reg .b64 a, b; setp.ne.b32 p, %4, 0; mov.b64 a, {%1, %5}; mov.b64 b, {%2, %5}; "
                 "tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %3, p; }"
                 ::"r"(d), "r"(a), "r"(b), "r"(idesc), "r"((uint32_t)accumulate), "r"(TILE_DESC_HI) : "memory");
}
__device__ __forceinline__ void tile_commit(uint32_t bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void tmem_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tmem_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tmem_alloc_all(uint32_t slot)
{
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(slot), "r"(512u) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_free_all(uint32_t tmem)
{
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u) : "memory");
}
// 32 columns of this warp's 32 lanes: the load is in flight until tmem_wait (of all loads issued so far), which hands the
// values over.
__device__ __forceinline__ void tmem_issue32(uint32_t addr, f32x2 (&u)[16])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
                 "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
                 : "=f"(u[0].x), "=f"(u[0].y), "=f"(u[1].x), "=f"(u[1].y), "=f"(u[2].x), "=f"(u[2].y), "=f"(u[3].x), "=f"(u[3].y),
                   "=f"(u[4].x), "=f"(u[4].y), "=f"(u[5].x), "=f"(u[5].y), "=f"(u[6].x), "=f"(u[6].y), "=f"(u[7].x), "=f"(u[7].y),
                   "=f"(u[8].x), "=f"(u[8].y), "=f"(u[9].x), "=f"(u[9].y), "=f"(u[10].x), "=f"(u[10].y), "=f"(u[11].x), "=f"(u[11].y),
                   "=f"(u[12].x), "=f"(u[12].y), "=f"(u[13].x), "=f"(u[13].y), "=f"(u[14].x), "=f"(u[14].y), "=f"(u[15].x), "=f"(u[15].y)
                 : "r"(addr) : "memory");
}
__device__ __forceinline__ void tmem_wait(f32x2 (&u)[16])
{
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+f"(u[0].x), "+f"(u[0].y), "+f"(u[1].x), "+f"(u[1].y), "+f"(u[2].x), "+f"(u[2].y), "+f"(u[3].x), "+f"(u[3].y),
                   "+f"(u[4].x), "+f"(u[4].y), "+f"(u[5].x), "+f"(u[5].y), "+f"(u[6].x), "+f"(u[6].y), "+f"(u[7].x), "+f"(u[7].y),
                   "+f"(u[8].x), "+f"(u[8].y), "+f"(u[9].x), "+f"(u[9].y), "+f"(u[10].x), "+f"(u[10].y), "+f"(u[11].x), "+f"(u[11].y),
                   "+f"(u[12].x), "+f"(u[12].y), "+f"(u[13].x), "+f"(u[13].y), "+f"(u[14].x), "+f"(u[14].y), "+f"(u[15].x), "+f"(u[15].y)
                 :: "memory");
}
__device__ __forceinline__ void tmem_load32(uint32_t addr, f32x2 (&u)[16])
{
    tmem_issue32(addr, u);
    tmem_wait(u);
}
__device__ __forceinline__ void tmem_store32(uint32_t addr, const f32x2 (&u)[16])
{
    asm volatile("tcgen05.st.sync.aligned.32x32b.x32.b32 [%32], {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
                 "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31};\n\ttcgen05.wait::st.sync.aligned;"
                 :: "f"(u[0].x), "f"(u[0].y), "f"(u[1].x), "f"(u[1].y), "f"(u[2].x), "f"(u[2].y), "f"(u[3].x), "f"(u[3].y),
                    "f"(u[4].x), "f"(u[4].y), "f"(u[5].x), "f"(u[5].y), "f"(u[6].x), "f"(u[6].y), "f"(u[7].x), "f"(u[7].y),
                    "f"(u[8].x), "f"(u[8].y), "f"(u[9].x), "f"(u[9].y), "f"(u[10].x), "f"(u[10].y), "f"(u[11].x), "f"(u[11].y),
                    "f"(u[12].x), "f"(u[12].y), "f"(u[13].x), "f"(u[13].y), "f"(u[14].x), "f"(u[14].y), "f"(u[15].x), "f"(u[15].y), "r"(addr) : "memory");
}
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap *map, int x, int y, uint32_t bar)
{
    asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
                 ::"r"(dst), "l"(map), "r"(x), "r"(y), "r"(bar) : "memory");
}
// Eight words to 32 adjacent bytes, in one store where they are aligned.
__device__ __forceinline__ void tile_store32(uint8_t *dst, const uint32_t (&w)[8], bool aligned)
{
    if (aligned) {
        asm volatile("st.global.v8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};"
                     ::"l"(dst), "r"(w[0]), "r"(w[1]), "r"(w[2]), "r"(w[3]), "r"(w[4]), "r"(w[5]), "r"(w[6]), "r"(w[7]) : "memory");
    } else {
        reinterpret_cast<uint4 *>(dst)[0] = make_uint4(w[0], w[1], w[2], w[3]);
        reinterpret_cast<uint4 *>(dst)[1] = make_uint4(w[4], w[5], w[6], w[7]);
    }
}

// H_64 / 2 (or smaller), and for blocks of 128 its negative, as operands at h and h + TILE_H_BYTES.
template <int LOG2B>
__device__ __forceinline__ void tile_write_hadamard(unsigned char *h, int tid, int nthr)
{
    constexpr int N = LOG2B >= 6 ? 64 : 1 << LOG2B;
    for (int e = tid; e < N * N / 2; e += nthr) {
        const int n = e / (N / 2), k = 2 * (e - n * (N / 2));
        const uint32_t at = (uint32_t)(n * 128 + (((k >> 3) ^ (n & 7)) << 4) + (k & 7) * 2);
        const uint32_t w = (hadamard_bf16(n, k) | (hadamard_bf16(n, k + 1) << 16)) - 0x00800080u;
        *reinterpret_cast<uint32_t *>(h + at) = w;
        if (LOG2B == 7) *reinterpret_cast<uint32_t *>(h + TILE_H_BYTES + at) = w ^ 0x80008000u;
    }
}

// The rotation of one tile (one thread).  half_bytes: of the tile's first 64 channels.
template <int LOG2B>
__device__ __forceinline__ void tile_rotate(uint32_t tmem, uint32_t tile, uint32_t half_bytes, uint32_t h)
{
    constexpr int B = 1 << LOG2B;
    const uint32_t x[2] = {tile_desc(tile), tile_desc(tile + half_bytes)}, hd = tile_desc(h);      // (16 channels: 2 in a descriptor)
    if (LOG2B == 7) {
#pragma unroll
        for (int o = 0; o < 2; ++o) {                          // outputs 0 .. 63, 64 .. 127
#pragma unroll
            for (int s = 0; s < 8; ++s)                        // 16 inputs a step
                tile_mma(tmem + o * 64, x[s >> 2] + 2 * (s & 3), hd + ((s >> 2) & o) * (TILE_H_BYTES / 16) + 2 * (s & 3), tile_idesc(64), s > 0);
        }
    } else {
#pragma unroll
        for (int k = 0; k < 8; ++k) {                          // step of 16 channels of the piece
            const int s = k % (B / 16);
            tile_mma(tmem + (k / (B / 16)) * B, x[k >> 2] + 2 * (k & 3), hd + 2 * s, tile_idesc(B), s > 0);
        }
    }
}

// -------------------------------------------------------------------------------------------- exact sums

// Byte offset of channel c of piece r in a tile.
__device__ __forceinline__ uint32_t tile_at(uint32_t half_bytes, uint32_t r, uint32_t c)
{
    return (c >> 6) * half_bytes + r * 128u + ((((c >> 3) ^ r) & 7u) << 4) + (c & 7u) * 2u;
}

// Sums for the exact outputs of the block at column c of a piece, by one lane: by the place in eight adjacent inputs,
// signed by the eight's parity; the low three index bits of the output are left.  load(k): inputs k .. k + 7 of the block.
template <int LOG2B, int UNROLL, typename F>
__device__ __forceinline__ void tile_sums(uint32_t c, F load, double (&S)[8])
{
    constexpr uint32_t B = 1u << LOG2B;
    const uint32_t i = c & (B - 1u);
#pragma unroll
    for (int e = 0; e < 8; ++e) S[e] = 0.0;
#pragma unroll(B / 8 < UNROLL ? B / 8 : UNROLL)
    for (uint32_t k = 0; k < B; k += 8) {
        const uint4 v = load(k);
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
        const double f = __hiloint2double(((__popc(i & k) & 1) ? (int)0x80000000 : 0) | 0x77e00000, 0);          // +-2^896 / 2
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            S[2 * j] = fma(bf16_raw_f64(w[j] << 16), f, S[2 * j]);
            S[2 * j + 1] = fma(bf16_raw_f64(w[j]), f, S[2 * j + 1]);
        }
    }
}
template <int LOG2B>
__device__ __forceinline__ void tile_sums_global(const TileParams &p, uint32_t piece, uint32_t c, double (&S)[8])
{
    const uint4 *src = reinterpret_cast<const uint4 *>(p.x + (size_t)piece * 128 + (c & ~((1u << LOG2B) - 1u)));
    tile_sums<LOG2B, 16>(c, [&](uint32_t k) { return __ldg(src + k / 8); }, S);
}
// From the sums: the four exact outputs of a quad (c a multiple of 4), or the one at column c.
__device__ __forceinline__ void tile_quad_of(double (&S)[8], uint32_t c, double (&o)[4])
{
    const double s4 = (c & 4u) ? -1.0 : 1.0;
#pragma unroll
    for (int e = 0; e < 4; ++e) S[e] = fma(s4, S[e + 4], S[e]);
    const double a0 = S[0] + S[1], a1 = S[0] - S[1], a2 = S[2] + S[3], a3 = S[2] - S[3];
    o[0] = a0 + a2; o[1] = a1 + a3; o[2] = a0 - a2; o[3] = a1 - a3;
}
__device__ __forceinline__ double tile_output_of(double (&S)[8], uint32_t c)
{
    const double s1 = (c & 1u) ? -1.0 : 1.0, s2 = (c & 2u) ? -1.0 : 1.0, s4 = (c & 4u) ? -1.0 : 1.0;
#pragma unroll
    for (int e = 0; e < 4; ++e) S[e] = fma(s4, S[e + 4], S[e]);
    return fma(s2, fma(s1, S[3], S[2]), fma(s1, S[1], S[0])) + 0.0;        // (+0 for a sum of zeros of either sign)
}
__device__ __forceinline__ double tile_abs_max(const double (&o)[4]) { return fmax(fmax(fabs(o[0]), fabs(o[1])), fmax(fabs(o[2]), fabs(o[3]))); }

// All exact outputs of a piece, by a warp: lane l brings the inputs of columns 4 l .. 4 l + 3 and gets the outputs there
// (the butterfly in fp64).
template <int LOG2B>
__device__ __forceinline__ void tile_butterfly(uint32_t w0, uint32_t w1, int lane, double (&o)[4])
{
    const double x0 = bf16_raw_f64(w0 << 16), x1 = bf16_raw_f64(w0), x2 = bf16_raw_f64(w1 << 16), x3 = bf16_raw_f64(w1);
    const double a0 = x0 + x1, a1 = x0 - x1, a2 = x2 + x3, a3 = x2 - x3;
    o[0] = (a0 + a2) * 0x1p895; o[1] = (a1 + a3) * 0x1p895; o[2] = (a0 - a2) * 0x1p895; o[3] = (a1 - a3) * 0x1p895;
#pragma unroll
    for (int t = 0; t < LOG2B - 2; ++t) {
        const double sg = ((lane >> t) & 1) ? -1.0 : 1.0;
#pragma unroll
        for (int e = 0; e < 4; ++e) o[e] = fma(sg, o[e], __shfl_xor_sync(0xffffffffu, o[e], 1 << t));
    }
}
// Whether the fp32 outputs of a piece are exact (see RowSpan; the products are aligned to the largest of a step and none of
// their bits lies lower than the span), by one lane.
__device__ __noinline__ bool tile_lane_exact(const uint16_t *x)
{
    RowSpan s = {0.0f, 1 << 20};
#pragma unroll 8
    for (int k = 0; k < 16; ++k) {
        const uint4 v = __ldg(reinterpret_cast<const uint4 *>(x) + k);
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const uint32_t a = (w[e >> 1] >> (16 * (e & 1))) & 0x7fffu;
            s.sum += __uint_as_float(a << 16);
            if (a != 0u) s.low = min(s.low, a < 0x80u ? __ffs(a) : (int)(a >> 7) + __ffs((a & 0x7fu) | 0x80u) - 1);
        }
    }
    return row_span_exact(s);
}

// Largest exact magnitude among the outputs of piece r of a tile at the columns c0 + (set bits of want), by a warp.
template <int LOG2B>
__device__ __noinline__ double tile_exact_max(uint32_t tile, uint32_t half_bytes, uint32_t r, uint32_t c0, uint32_t want, int lane)
{
    double o[4], a = 0.0;
    uint32_t w[2];
    asm volatile("ld.shared.v2.b32 {%0,%1}, [%2];" : "=r"(w[0]), "=r"(w[1]) : "r"(tile + tile_at(half_bytes, r, 4u * (uint32_t)lane)) : "memory");
    tile_butterfly<LOG2B>(w[0], w[1], lane, o);
    const uint32_t c = 4u * (uint32_t)lane - c0;
    if (c < 32u) {
#pragma unroll
        for (int e = 0; e < 4; ++e)
            if ((want >> (c + e)) & 1u) a = fmax(a, fabs(o[e]));
    }
    return __longlong_as_double((long long)warp_max_u64((unsigned long long)__double_as_longlong(a)));
}

// -------------------------------------------------------------------------------------------- exact codes

// What the exact codes of a range or row depend on.
struct TileScale {
    double f;                // reciprocal of what an unnormalised value is divided by (a few roundings)
    double a, s64, z64;
    float mul;
    int E;
};
template <int MODE>
__device__ __forceinline__ TileScale tile_scale_max(const TileParams &p, double a)           // exact maximum: integers, E2M1 per token
{
    TileScale q = {0.0, a, 0.0, 0.0, 0.0f, 0};
    if (MODE == ROW_FP4) { q.s64 = a / p.sqrt_b / 7.0; q.f = a > 0.0 ? 7.0 / a : 0.0; }
    else q.mul = row_inverse((float)a);
    return q;
}
__device__ __forceinline__ TileScale tile_scale_asym(const TileParams &p, double hi, double lo)
{
    TileScale q = {0.0, 0.0, 0.0, 0.0, 0.0f, 0};
    q.s64 = (hi / p.sqrt_b - lo / p.sqrt_b) / 15.0;
    if (q.s64 != 0.0) {
        q.z64 = rint(lo / p.sqrt_b / q.s64);
        q.f = 15.0 / (hi - lo);
    }
    return q;
}
__device__ __forceinline__ TileScale tile_scale_mx(const TileParams &p, uint32_t exponent)
{
    TileScale q = {0.0, 0.0, 0.0, 0.0, 0.0f, (int)exponent - 127};
    q.f = __hiloint2double((1023 - q.E) << 20, 0) * p.inv_sqrt_b;
    return q;
}
// Code of the exact unnormalised value u: from a product, and where that is all but on a boundary from the operations of
// the definition.
template <int MODE>
__device__ __forceinline__ uint32_t tile_code(const TileParams &p, double u, const TileScale &q)
{
    if (MODE == ROW_TOKEN || MODE == ROW_GROUP) return q.a > 0.0 ? row_int4_code<true>(u, q.a, q.mul, p.sqrt_b) : 0u;
    const double t = u * q.f;
    if (MODE == ROW_ASYM) {
        if (q.s64 == 0.0) return 0u;
        const double k = rint(t);
        if (fabs(t - k) > 0.5 - 1.0e-9) return row_exact_code<ROW_ASYM>(u, p.sqrt_b, q.s64, q.z64, 0);
        return (uint32_t)((int)fmin(fmax(k - q.z64, 0.0), 15.0));
    }
    const uint32_t c = e2m1_code_exact(t * (1.0 - 1.0e-12), signbit(u));
    return c == e2m1_code_exact(t * (1.0 + 1.0e-12), signbit(u)) ? c : row_exact_code<MODE>(u, p.sqrt_b, q.s64, 0.0, q.E);
}
__device__ __forceinline__ void tile_mend(const TileParams &p, uint32_t piece, uint32_t job, uint32_t code)
{
    // (a correction, not a new value: nothing has to be read, and neighbours may be mended at the same time)
    const uint32_t c = (job >> 7) & 127u, diff = code ^ ((job >> 16) & 0xFu);
    if (diff) atomicXor(reinterpret_cast<uint32_t *>(p.out_codes + (size_t)piece * 64) + (c >> 3), diff << (4u * (c & 7u)));
}

// -------------------------------------------------------------------------------------------- quantising

// Codes of the lane's 32 values, and whether any of them is within the window of a tie (as row_quantise; integers are
// packed on the fp32 side: magic + k0 + 256 k2 and magic + k1 + 256 k3 are one packed fma).  TWO: the second half of the
// values by B.
template <int MODE, bool TWO>
__device__ __forceinline__ bool tile_quantise2(const f32x2 (&u)[16], const RowQuant &A, const RowQuant &B, uint32_t *cw)
{
    if (MODE == ROW_MX || MODE == ROW_FP4) {
        uint32_t h[8], diff = 0u;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const RowQuant &Q = TWO && j >= 4 ? B : A;
            const f32x2 m2 = pack2(Q.mul, Q.mul), tp = pack2(Q.tau, Q.tau), tm = pack2(0.0f - Q.tau, 0.0f - Q.tau);
            const f32x2 up0 = fma2(u[2 * j], m2, tp), up1 = fma2(u[2 * j + 1], m2, tp);
            const f32x2 dn0 = fma2(u[2 * j], m2, tm), dn1 = fma2(u[2 * j + 1], m2, tm);
            h[j] = cvt_e2m1x4_pair(up0.x, up0.y, up1.x, up1.y, dn0.x, dn0.y, dn1.x, dn1.y);
        }
#pragma unroll
        for (int w = 0; w < 4; ++w) {
            cw[w] = __byte_perm(h[2 * w], h[2 * w + 1], 0x5410);
            diff |= cw[w] ^ __byte_perm(h[2 * w], h[2 * w + 1], 0x7632);
        }
        return diff != 0u;
    }
    const f32x2 up = pack2(-256.0f, -256.0f);
    float far[2] = {0.0f, 0.0f}, far2[2] = {0.0f, 0.0f};
#pragma unroll
    for (int w = 0; w < 4; ++w) {
        const RowQuant &Q = TWO && w >= 2 ? B : A;
        const f32x2 m2 = pack2(Q.mul, Q.mul), mg = pack2(Q.magic, Q.magic);
        uint32_t h[2];
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const f32x2 v0 = u[4 * w + 2 * j], v1 = u[4 * w + 2 * j + 1];
            f32x2 r0 = fma2(v0, m2, mg), r1 = fma2(v1, m2, mg);
            f32x2 n0 = sub2(mg, r0), n1 = sub2(mg, r1);                      // minus the rounded values
            const f32x2 e0 = fma2(v0, m2, n0), e1 = fma2(v1, m2, n1);
            far[w >> 1] = max3abs(far[w >> 1], e0.x, e0.y);
            far2[w >> 1] = max3abs(far2[w >> 1], e1.x, e1.y);
            if (MODE == ROW_ASYM) {            // codes 0 .. 15: the magic number less z makes the sum 1.5 * 2^23 + code
                const float lo = 12582912.0f, hi = 12582927.0f;
                r0 = pack2(fminf(fmaxf(r0.x, lo), hi), fminf(fmaxf(r0.y, lo), hi));
                r1 = pack2(fminf(fmaxf(r1.x, lo), hi), fminf(fmaxf(r1.y, lo), hi));
                n1 = sub2(pack2(lo, lo), r1);
            }
            const f32x2 s = fma2(n1, up, r0);
            h[j] = __float_as_uint(s.y) * 16u + __float_as_uint(s.x);
        }
        cw[w] = __byte_perm(h[0], h[1], 0x5410);
        if (MODE != ROW_ASYM) cw[w] ^= 0x88888888u;
    }
    return fmaxf(far[0], far2[0]) > 0.5f - A.tau || fmaxf(far[1], far2[1]) > 0.5f - (TWO ? B : A).tau;
}
template <int MODE>
__device__ __forceinline__ bool tile_quantise(const f32x2 (&u)[16], const RowQuant &Q, uint32_t *cw) { return tile_quantise2<MODE, false>(u, Q, Q, cw); }

// Maximum magnitudes of the two halves of 32 values, and of all.
__device__ __forceinline__ void tile_half_max(const f32x2 (&u)[16], float &a, float &b)
{
    a = max3abs(fabsf(u[0].x), u[0].y, u[1].x);
    b = max3abs(fabsf(u[8].x), u[8].y, u[9].x);
    a = fmaxf(a, fabsf(u[1].y));
    b = fmaxf(b, fabsf(u[9].y));
#pragma unroll
    for (int m = 2; m < 8; ++m) { a = max3abs(a, u[m].x, u[m].y); b = max3abs(b, u[m + 8].x, u[m + 8].y); }
}
__device__ __forceinline__ float tile_max(const f32x2 (&u)[16])
{
    float a, b;
    tile_half_max(u, a, b);
    return fmaxf(a, b);
}

// Asymmetric: reciprocal step, zero point, and the rounding window (slack + per_ref * largest magnitude of the block) from
// the fp32 extremes of a row; true where rounding the zero point is a close call.
__device__ __forceinline__ bool tile_zero_point(float hr, float lr, float err, float &inv, float &z, float &slack, float &per_ref)
{
    const float a_row = fmaxf(fabsf(hr), fabsf(lr));
    inv = hr > lr ? fminf(__fdividef(1.875f, 0.125f * hr - 0.125f * lr), 3.0e38f) : 0.0f;         // (the range itself may overflow)
    const float ar = hr > lr ? fminf(a_row * inv, 3.0e38f) : 3.0e38f, v = lr * inv;
    z = rintf(v);
    // errors of an element, and of the step (2 err |y|max / range, relative)
    slack = (ar + 8.0f) * 6.0e-7f;
    per_ref = err * inv * (1.0f + ar * (2.0f / 15.0f));
    return !(fabsf(v - z) <= 0.5f - (err * ar * (1.0f + ar * (2.0f / 15.0f)) + slack));
}

// false: no room
__device__ __forceinline__ bool tile_note(TileNotes *notes, uint32_t job)
{
    const uint32_t at = atomicAdd(&notes->count, 1u);
    if (at < TILE_JOBS) notes->job[at] = job;
    return at < TILE_JOBS;
}

// ---- Flat rows, small integers: where a piece has many candidates or doubtful elements its fp32 outputs are as a rule exact,
// which a look at its inputs shows; sums only where they are not.  A piece per lane, all lanes at work.  (2048 x 9728 of
// integers -3 .. 3, b = 128, INT4 per token: 245 us, 856 with the pieces settled in turn by one warp, 270 in registers)

// The quads of 32 columns that hold candidates for a row's maximum.
__device__ __forceinline__ uint32_t tile_candidates(const f32x2 (&u)[16], float thr)
{
    uint32_t quads = 0u;
#pragma unroll
    for (int j = 0; j < 8; ++j) quads |= fmaxf(max3abs(fabsf(u[2 * j].x), u[2 * j].y, u[2 * j + 1].x), fabsf(u[2 * j + 1].y)) >= thr ? (1u << j) : 0u;
    return quads;
}

// Exact maximum of the lane's candidates (cmask: chunks that have some; 0: nothing to do) into its row's word.
template <int LOG2B>
__device__ __noinline__ void tile_put_maximum(const TileParams &p, uint32_t tmem, uint32_t piece, uint32_t cmask, float thr, TileNotes *notes, int ri)
{
    f32x2 u[16];
    int exact = -1;                                          // (asked for when there are several: a look costs as much as a sum)
    double a = 0.0;
    __syncwarp();
#pragma unroll 1
    for (int c = 0; c < 4; ++c) {
        if (!__any_sync(0xffffffffu, (cmask >> c) & 1u)) continue;
        tmem_load32(tmem + 32 * c, u);
        uint32_t quads = (cmask >> c) & 1u ? tile_candidates(u, thr) : 0u;
        if (exact < 0 && __popc(quads) > 2) exact = tile_lane_exact(p.x + (size_t)piece * 128);
        if (exact > 0 && quads) {
            quads = 0u;
            a = fmax(a, (double)tile_max(u));
        }
        while (quads) {
            double S[8], o[4];
            const uint32_t col = (uint32_t)(32 * c) + 4u * ((uint32_t)__ffs(quads) - 1u);
            quads &= quads - 1u;
            tile_sums_global<LOG2B>(p, piece, col, S);
            tile_quad_of(S, col, o);
            a = fmax(a, tile_abs_max(o));
        }
        __syncwarp();
    }
    if (cmask != 0u) atomicMax(&notes->ex[ri], (unsigned long long)__double_as_longlong(a));
    __syncwarp();
}

// Exact codes of the pieces of the lanes with `mine`: quantised again, by exact scales, and their doubtful elements settled here.
// aux: exponents (MX) or bits of the exact maximum (ranges); token rows have their maxima in the row's words.
template <int LOG2B, int MODE>
__device__ __noinline__ void tile_requantise(const TileParams &p, uint32_t tmem, uint32_t piece, bool mine, unsigned long long aux, TileNotes *notes, int w, int ri)
{
    f32x2 u[16];
    const int lane = (int)(threadIdx.x & 31u);
    const unsigned whose = __ballot_sync(0xffffffffu, mine);
    if (lane == 0) notes->settled[w] = whose;
    const bool exact = mine && tile_lane_exact(p.x + (size_t)piece * 128);
    const float err = exact ? 1.2e-7f : p.err;               // (exact elements: the fp32 maximum of an exact range)
    __syncwarp();
    float ref = 0.0f;                                        // (of the piece: not less than any block's)
#pragma unroll 1
    for (int c = 0; c < 4; ++c) { tmem_load32(tmem + 32 * c, u); ref = fmaxf(ref, tile_max(u)); }
    TileScale q = {0.0, 0.0, 0.0, 0.0, 0.0f, 0};
    RowQuant Q;
    Q.magic = 12584968.0f;
    Q.mul = Q.tau = 0.0f;
    if (MODE != ROW_MX) {
        q = tile_scale_max<MODE>(p, __longlong_as_double((long long)(MODE == ROW_GROUP ? aux : notes->ex[ri])));
        Q.mul = row_inverse((float)q.a);
        Q.tau = (err + 5.0e-7f) * Q.mul * ref + (MODE == ROW_FP4 ? 0.0f : 2.0e-7f);
    }
#pragma unroll 1
    for (int c = 0; c < 4; ++c) {
        tmem_load32(tmem + 32 * c, u);
        if (MODE == ROW_MX) {
            const int Eb = (int)(((uint32_t)aux >> (8 * c)) & 0xffu);
            q = tile_scale_mx(p, (uint32_t)Eb);
            Q.mul = __uint_as_float((uint32_t)min(max(255 - Eb - LOG2B / 2, 1), 254) << 23) * ((LOG2B & 1) ? 0.70710678118654752f : 1.0f);
            Q.tau = Eb == 0 ? 3.0e38f : err * ref * Q.mul + 2.0e-6f;          // (the lowest exponent: perhaps a group of zeros)
            // exact, and so is the product with a power of two: the conversion rounds ties to even (2048 x 9728 of integers, b = 16: 869 us
            // with every tie evaluated in fp64, 270)
            if ((LOG2B & 1) == 0 && exact) Q.tau = 0.0f;
        }
        uint32_t cw[4];
        const bool fl = tile_quantise<MODE>(u, Q, cw) && mine;
        uint32_t tie = fl ? row_tie_bits<MODE>(u, Q) : 0u;
        if (LOG2B <= 5 && (MODE == ROW_MX || MODE == ROW_FP4) && Q.tau < 0.2f) {        // (blocks of zeros have code 0, as stored)
            float a, b;
            tile_half_max(u, a, b);
            if (LOG2B == 5) a = b = fmaxf(a, b);
            tie &= (a > 0.0f ? 0xffffu : 0u) | (b > 0.0f ? 0xffff0000u : 0u);
        }
        if ((MODE == ROW_MX || MODE == ROW_FP4) && exact && Q.tau < 0.2f) {           // exact zeros have code 0, as stored
            uint32_t zero = 0u;
#pragma unroll
            for (int i = 0; i < 16; ++i) zero |= (u[i].x == 0.0f ? 1u << (2 * i) : 0u) | (u[i].y == 0.0f ? 2u << (2 * i) : 0u);
            tie &= ~zero;
        }
        // few lanes with many: an element per lane
        unsigned lanes = __ballot_sync(0xffffffffu, __popc(tie) > 2);
        if (__popc(lanes) > 4) lanes = 0u;
        while (lanes) {
            const int src = __ffs(lanes) - 1;
            lanes &= lanes - 1;
            const bool ex = __shfl_sync(0xffffffffu, (int)exact, src) != 0;
            const uint32_t pc = __shfl_sync(0xffffffffu, piece, src), ts = __shfl_sync(0xffffffffu, tie, src);
            float f = 0.0f;
#pragma unroll
            for (int i = 0; i < 16; ++i) {
                const float a = __shfl_sync(0xffffffffu, u[i].x, src), b = __shfl_sync(0xffffffffu, u[i].y, src);
                f = (lane >> 1) == i ? ((lane & 1) ? b : a) : f;
            }
            TileScale r;
            r.f = __shfl_sync(0xffffffffu, q.f, src);
            r.a = __shfl_sync(0xffffffffu, q.a, src);
            r.s64 = __shfl_sync(0xffffffffu, q.s64, src);
            r.z64 = __shfl_sync(0xffffffffu, q.z64, src);
            r.mul = __shfl_sync(0xffffffffu, q.mul, src);
            r.E = __shfl_sync(0xffffffffu, q.E, src);
            double v = (double)f + 0.0;
            if (!ex) {
                double S[8];
                tile_sums_global<LOG2B>(p, pc, (uint32_t)(32 * c + lane), S);
                v = tile_output_of(S, (uint32_t)(32 * c + lane));
            }
            uint32_t w = 0u, code = 0u;                        // the word of the lane's element as stored; its code
#pragma unroll
            for (int i = 0; i < 4; ++i) { const uint32_t t = __shfl_sync(0xffffffffu, cw[i], src); w = (lane >> 3) == i ? t : w; }
            const uint32_t sh = 4u * (uint32_t)(lane & 7);
            code = ((ts >> lane) & 1u) ? tile_code<MODE>(p, v, r) : (w >> sh) & 0xFu;
            code <<= sh;
#pragma unroll
            for (int o = 1; o < 8; o <<= 1) code |= __shfl_xor_sync(0xffffffffu, code, o);
#pragma unroll
            for (int i = 0; i < 4; ++i) { const uint32_t t = __shfl_sync(0xffffffffu, code, 8 * i); if (lane == src) cw[i] = t; }
            if (lane == src) tie = 0u;
        }
#pragma unroll 1
        while (tie) {
            const uint32_t e = (uint32_t)__ffs(tie) - 1u, col = (uint32_t)(32 * c) + e;
            tie &= tie - 1u;
            double v;
            if (exact) {
                float f = 0.0f;
#pragma unroll
                for (uint32_t i = 0; i < 16; ++i) f = (e >> 1) == i ? ((e & 1u) ? u[i].y : u[i].x) : f;
                v = (double)f + 0.0;                          // (+0 for a zero, as the sums give)
            } else {
                double S[8];
                tile_sums_global<LOG2B>(p, piece, col, S);
                v = tile_output_of(S, col);
            }
            const uint32_t sh = 4u * (e & 7u), code = tile_code<MODE>(p, v, q) << sh, keep = ~(0xFu << sh);
#pragma unroll
            for (uint32_t i = 0; i < 4; ++i) cw[i] = (e >> 3) == i ? (cw[i] & keep) | code : cw[i];
        }
        if (mine) *reinterpret_cast<uint4 *>(p.out_codes + (size_t)piece * 64 + 16 * c) = make_uint4(cw[0], cw[1], cw[2], cw[3]);
        __syncwarp();
    }
}

// A lane's place in the tiles: the same for all of them.
struct TileLane {
    int w, lane;             // warp of the four, lane
    int ri;                  // token row of the tile (its index in the exchange words)
    bool first, coupled, whole;      // first piece of its row; rows lie in several warps; the warp lies in one row
};

// A warp's 32 pieces of tile t.  tmem: its lanes of the accumulator; bar: the four warps' named barrier.  false: another of the four
// warps, which share rows, has given up.
template <int LOG2B, int MODE>
__device__ __forceinline__ bool tile_epilogue(const TileParams &p, const TileLane &L, uint32_t tmem, uint32_t tile, uint32_t half, uint32_t t, TileRows *rows,
                                              uint32_t par, int bar, TileNotes *notes)
{
    constexpr bool TOK = MODE == ROW_TOKEN || MODE == ROW_FP4;
    const int lane = L.lane, l = L.w * 32 + lane;
    const uint32_t piece = t * (uint32_t)p.tile_pieces + (uint32_t)l;
    const bool live = l < p.tile_pieces && piece < p.pieces;
    const float err = p.err;
    uint8_t *out = p.out_codes + (size_t)piece * 64;
    f32x2 ua[16], ub[16];
    RowQuant Q;
    Q.magic = 12584968.0f;                // 1.5 * 2^23 + 8 * 257: two nibbles of the sum are codes + 8
    float m[4] = {0.0f, 0.0f, 0.0f, 0.0f};                         // largest magnitude of each chunk of 32 columns
    float inv = 0.0f, lm = 0.0f, slack = 0.0f, per_ref = 0.0f, thr = 0.0f;
    uint32_t cmask = 0u;                                           // per token: chunks with candidates for the row's maximum
    bool many_max = false, many = false;                           // more candidates, doubtful elements than are worth a note each
    unsigned long long aux = 0ull;                                 // exact maximum (ranges)

    tmem_issue32(tmem, ua);
    if (MODE == ROW_GROUP) {
        // ---- the exact maximum of the lane's 128 outputs: the quads that reach the threshold (nearly always one)
        float qm[32];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            tmem_wait(ua);
#pragma unroll
            for (int j = 0; j < 8; ++j) qm[8 * c + j] = fmaxf(max3abs(fabsf(ua[2 * j].x), ua[2 * j].y, ua[2 * j + 1].x), fabsf(ua[2 * j + 1].y));
            if (c < 3) tmem_issue32(tmem + 32 * (c + 1), ua);
            m[c] = fmaxf(fmaxf(fmaxf(qm[8 * c], qm[8 * c + 1]), fmaxf(qm[8 * c + 2], qm[8 * c + 3])),
                         fmaxf(fmaxf(qm[8 * c + 4], qm[8 * c + 5]), fmaxf(qm[8 * c + 6], qm[8 * c + 7])));
        }
        lm = fmaxf(fmaxf(m[0], m[1]), fmaxf(m[2], m[3]));
        thr = lm - 2.0f * err * lm - lm * 2.4e-7f;
        uint32_t want = 0u;
#pragma unroll
        for (int j = 0; j < 32; ++j) want |= (qm[j] >= thr) ? (1u << j) : 0u;
        if (!live || !(lm > 0.0f)) want = 0u;
        double a_ex = 0.0;
        if (__popc(want) > 2 && tile_lane_exact(p.x + (size_t)piece * 128)) { a_ex = (double)lm; want = 0u; }
        __syncwarp();
        while (__any_sync(0xffffffffu, want != 0u)) {
            const uint32_t c = want ? 4u * ((uint32_t)__ffs(want) - 1u) : 0u, c0 = c & ~((1u << LOG2B) - 1u);
            double S[8], o[4];
            tile_sums<LOG2B, 4>(c, [&](uint32_t k) {
                uint4 v;
                asm volatile("ld.shared.v4.b32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(tile + tile_at(half, (uint32_t)l, c0 + k)) : "memory");
                return v;
            }, S);
            tile_quad_of(S, c, o);
            if (want) a_ex = fmax(a_ex, tile_abs_max(o));
            want &= want - 1u;
        }
        tmem_issue32(tmem, ua);
        if (live) reinterpret_cast<float *>(p.out_scales)[piece] = row_scale(a_ex, p.inv_7_sqrt_b, p.sqrt_b, 7.0);
        aux = (unsigned long long)__double_as_longlong(a_ex);
        notes->aux[l] = aux;
        inv = row_inverse((float)a_ex);
        // the element's error and the multiplier's (three roundings); the distance's own
        per_ref = (err + 5.0e-7f) * inv;
        slack = 2.0e-7f;
    } else if (TOK || LOG2B >= 6) {
        // ---- fp32 maxima of the chunks, then of the rows (MX inside longer blocks: the error reference)
#pragma unroll
        for (int c = 0; c < 4; c += 2) {
            tmem_wait(ua);
            tmem_issue32(tmem + 32 * (c + 1), ub);
            m[c] = tile_max(ua);
            tmem_wait(ub);
            tmem_issue32(tmem + (c ? 0 : 64), ua);                    // (in the end: the first chunk again, for the quantiser)
            m[c + 1] = tile_max(ub);
        }
        lm = fmaxf(fmaxf(m[0], m[1]), fmaxf(m[2], m[3]));
        if (TOK) {
            float hr = live ? lm : 0.0f;                              // the row's largest magnitude
            if (!L.coupled && p.row_pieces == 32) {
                hr = warp_max_f32(hr);
            } else if (!L.coupled) {
                for (int o = 1; o < p.row_pieces; o <<= 1) hr = fmaxf(hr, __shfl_xor_sync(0xffffffffu, hr, o));
            } else {
                if (L.whole) hr = warp_max_f32(hr);
                if (L.whole ? lane == 0 : live) atomicMax(&rows->mx[par][L.ri], __float_as_uint(hr));
                if (!named_barrier_all(bar, 128, true)) { tmem_wait(ua); return false; }
                hr = __uint_as_float(rows->mx[par][L.ri]);
                if (L.first) rows->mx[par ^ 1u][L.ri] = 0u;           // (the other tile's word: everybody has left that tile)
            }
            thr = hr - hr * (2.0f * err + 2.4e-7f);
#pragma unroll
            for (int c = 0; c < 4; ++c) cmask |= (m[c] >= thr) ? (1u << c) : 0u;
            if (!live || !(hr > 0.0f)) cmask = 0u;
            inv = row_inverse(hr);
            // the element's error and the multiplier's (the maximum's, three roundings); integers: the distance's own
            per_ref = (2.0f * err + 5.0e-7f) * inv;
            slack = MODE == ROW_FP4 ? 0.0f : 2.0e-7f;
        }
    }

    // ---- quantise and store, 64 columns at a time
    uint32_t exps = 0u;
#pragma unroll 1
    for (int h = 0; h < 2; ++h) {
        uint32_t cw[8];
        auto chunk = [&](const f32x2 (&u)[16], int k) {
            const float mh = h ? m[2 + k] : m[k];
            float hm[2] = {0.0f, 0.0f};                       // b = 16, E2M1: the chunk's two blocks
            int Eb = 0;
            if (MODE == ROW_MX) {
                float gm;
                if (LOG2B == 4) { tile_half_max(u, hm[0], hm[1]); gm = fmaxf(hm[0], hm[1]); }
                else gm = tile_max(u);
                const float ref = LOG2B <= 5 ? gm : LOG2B == 6 ? (h ? fmaxf(m[2], m[3]) : fmaxf(m[0], m[1])) : lm;
                // E + 127 with E = floor(log2(2 a / sqrt(b))) - 2; the distance of a to a value where the floor changes
                const uint32_t bits = __float_as_uint(gm);
                const int e8 = (int)(bits >> 23);
                float dist;
                if ((LOG2B & 1) == 0) {
                    const float lower = __uint_as_float(bits & 0x7f800000u);
                    dist = fminf(gm - lower, 2.0f * lower - gm);
                    Eb = e8 - LOG2B / 2 - 1;
                } else {
                    dist = fabsf(gm - __uint_as_float((bits & 0x7f800000u) | 0x3504f3u));
                    Eb = e8 - (LOG2B - 1) / 2 - 2 + ((bits & 0x7fffffu) >= 0x3504f4u ? 1 : 0);
                }
                const float tol = 2.0f * err * ref + gm * 4.8e-7f;
                // (a group inside a longer block can be zero in fp32 and not in truth)
                const bool near = live && (LOG2B <= 5 ? gm : ref) > 0.0f && (dist <= tol || e8 == 0);
                bool zero = !(gm > 0.0f);
                if (__any_sync(0xffffffffu, near)) {          // rare: the exact maximum of the group
                    uint32_t want = near ? row_reach(u, gm - tol) : 0u;
                    auto settle = [&](double best) {
                        int ex;
                        (void)frexp(best / p.sqrt_b, &ex);
                        Eb = ex - 3 + 127;
                        zero = best == 0.0;                   // (the fp32 values of a group that cancels exactly are rounding noise)
                    };
                    unsigned lanes = __ballot_sync(0xffffffffu, want != 0u);
                    if (__popc(lanes) > 4) {                  // flat rows, integers
                        if (want != 0u && tile_lane_exact(p.x + (size_t)piece * 128)) { settle((double)gm); want = 0u; }
                        lanes = __ballot_sync(0xffffffffu, want != 0u);
                    }
                    while (lanes) {
                        const int src = __ffs(lanes) - 1;
                        lanes &= lanes - 1;
                        const uint32_t ws = __shfl_sync(0xffffffffu, want, src);
                        const double best = tile_exact_max<LOG2B>(tile, half, (uint32_t)(L.w * 32 + src), (uint32_t)(64 * h + 32 * k), ws, lane);
                        if (lane == src) settle(best);
                    }
                }
                Eb = min(max(Eb, 0), 254);
                if ((LOG2B & 1) == 0) Q.mul = __uint_as_float((uint32_t)min(max(255 - Eb - LOG2B / 2, 1), 254) << 23);
                else Q.mul = __uint_as_float((uint32_t)min(max(255 - Eb - (LOG2B - 1) / 2, 1), 254) << 23) * 0.70710678118654752f;
                if (zero) { Eb = 0; Q.mul = 0.0f; }
                Q.tau = (ref > 0.0f && !(near && zero)) ? err * ref * Q.mul + 2.0e-6f : 0.0f;        // (the multiplier's and the product's rounding)
                exps |= (uint32_t)Eb << (16 * h + 8 * k);
            } else {
                const float ref = LOG2B <= 5 ? mh : LOG2B == 6 ? (h ? fmaxf(m[2], m[3]) : fmaxf(m[0], m[1])) : lm;
                Q.mul = inv;
                Q.tau = per_ref * ref + slack;
            }
            const uint32_t place = (uint32_t)(64 * h + 32 * k) << 7 | (uint32_t)l;
            if (TOK) {                                        // candidates for the row's maximum
                const bool cand = (cmask >> (2 * h + k)) & 1u;
                if (__any_sync(0xffffffffu, cand)) {
                    uint32_t quads = cand ? tile_candidates(u, thr) : 0u;
                    if (__popc(quads) > 2) { many_max = true; quads = 0u; }
                    while (quads) {
                        const uint32_t j = (uint32_t)__ffs(quads) - 1u;
                        quads &= quads - 1u;
                        if (!tile_note(notes, JOB_MAX | (uint32_t)L.ri << 20 | (place + (4u * j << 7)))) many_max = true;
                    }
                }
            }
            // b = 16: a block of zeros beside one that is not has no doubtful signs (4096 x 4096, FP4, such channels: 87 us without this, 18)
            constexpr bool HALVES = LOG2B == 4 && (MODE == ROW_MX || MODE == ROW_FP4);
            RowQuant QA = Q, QB = Q;
            if (HALVES) {
                if (MODE == ROW_FP4) tile_half_max(u, hm[0], hm[1]);
                if (!(hm[0] > 0.0f)) QA.tau = 0.0f;
                if (!(hm[1] > 0.0f)) QB.tau = 0.0f;
            }
            const bool fl = tile_quantise2<MODE, HALVES>(u, QA, QB, cw + 4 * k) && live;
            if (__any_sync(0xffffffffu, fl)) {
                uint32_t tie = fl ? row_tie_bits<MODE>(u, Q) : 0u;
                if (HALVES) tie &= (hm[0] > 0.0f ? 0xffffu : 0u) | (hm[1] > 0.0f ? 0xffff0000u : 0u);
                if (__popc(tie) > TILE_TIES) { many = true; tie = 0u; }
                while (tie) {
                    const uint32_t e = (uint32_t)__ffs(tie) - 1u;
                    tie &= tie - 1u;
                    const uint32_t w = e < 16 ? (e < 8 ? cw[4 * k] : cw[4 * k + 1]) : (e < 24 ? cw[4 * k + 2] : cw[4 * k + 3]);
                    if (!tile_note(notes, JOB_TIE | (uint32_t)(TOK ? L.ri : 0) << 20 | ((w >> (4 * (e & 7u))) & 0xFu) << 16 | (place + (e << 7)))) { many = true; break; }
                }
            }
        };
        tmem_wait(ua);
        tmem_issue32(tmem + 64 * h + 32, ub);
        chunk(ua, 0);
        tmem_wait(ub);
        if (h == 0) tmem_issue32(tmem + 64, ua);
        chunk(ub, 1);
        if (live) tile_store32(out + 32 * h, cw, p.wide_store);
    }
    if (MODE == ROW_MX) {
        if (live) reinterpret_cast<uint32_t *>(p.out_scales)[piece] = exps;
        aux = exps;
        notes->aux[l] = aux;
    }
    bool codes = __any_sync(0xffffffffu, many);
    if (TOK) {
        const bool ext = codes || __any_sync(0xffffffffu, many_max);
        if (ext && lane == 0) atomicOr(&notes->flat, codes ? FLAT_ROWS | FLAT_CODES : FLAT_ROWS);
        if (L.coupled) {                                              // (the four warps take this way together)
            named_barrier(bar, 128);
            codes = (*reinterpret_cast<volatile uint32_t *>(&notes->flat) & FLAT_CODES) != 0u;
        }
        if (ext || codes) tile_put_maximum<LOG2B>(p, tmem, piece, many_max || codes ? cmask : 0u, thr, notes, L.ri);
        if (codes && L.coupled) named_barrier(bar, 128);
    }
    if (codes) tile_requantise<LOG2B, MODE>(p, tmem, piece, many, aux, notes, L.w, L.ri);
    return true;
}

// -------------------------------------------------------------------------------------------- notes

// Up to 32 records, one per lane.
template <int LOG2B, int MODE>
__device__ __forceinline__ void tile_settle_records(const TileParams &p, const TileRecord *list, int n, int lane)
{
    constexpr bool TOK = MODE == ROW_TOKEN || MODE == ROW_FP4;
    if (lane >= n) return;
    const TileRecord rec = list[lane];
    const uint32_t c = (rec.job >> 7) & 127u;
    double S[8], u = 0.0;
    TileScale q = {0.0, 0.0, 0.0, 0.0, 0.0f, 0};
    const bool tie = !TOK || (rec.job >> 30) == (JOB_TIE >> 30);
    if (tie) {
        tile_sums_global<LOG2B>(p, rec.piece, c, S);
        u = tile_output_of(S, c);
    }
    if (TOK) {                                     // the row's maximum, from the quad that holds it
        double o[4];
        tile_sums_global<LOG2B>(p, rec.aux[0], rec.aux[1], S);
        tile_quad_of(S, rec.aux[1], o);
        q = tile_scale_max<MODE>(p, tile_abs_max(o));
        if (!tie) reinterpret_cast<float *>(p.out_scales)[rec.piece / (uint32_t)p.row_pieces] = row_scale(q.a, p.inv_7_sqrt_b, p.sqrt_b, 7.0);
    } else if (MODE == ROW_MX) {
        q = tile_scale_mx(p, rec.aux[0] >> (8 * (c >> 5)) & 0xffu);
    } else {
        q = tile_scale_max<MODE>(p, __hiloint2double((int)rec.aux[1], (int)rec.aux[0]));
    }
    if (tie) tile_mend(p, rec.piece, rec.job, tile_code<MODE>(p, u, q));
}

// Batches of records on their way from the warp that collects them to those that settle them: one each, filled in turn.
struct TileBatches {
    TileRecord rec[2][TILE_RECORDS];
    uint32_t count[2];
};
struct TileCollector {
    TileBatches *b;
    uint32_t full, free;     // barriers
    uint32_t turn;           // batches handed over
    int n, lane;
    __device__ __forceinline__ TileRecord *list() { return b->rec[turn & 1u]; }
    __device__ __forceinline__ void hand_over(uint32_t last)
    {
        if (lane == 0) b->count[turn & 1u] = (uint32_t)n | last;
        __syncwarp();
        if (lane == 0) mbar_arrive(full + (turn & 1u) * 8);
        ++turn;
        n = 0;
        if (turn >= 2u && !mbar_wait_fast(free + (turn & 1u) * 8, ((turn >> 1) - 1u) & 1u) && lane == 0) atomicOr(&g_perq_device_error, 1u);
    }
    // room for 32 more
    __device__ __forceinline__ void make_room() { if (n > TILE_RECORDS - 32) hand_over(0u); }
};

// The notes of a tile, by a warp.  Most become records; token rows with several candidates, or with maxima that have no note,
// are settled here: their exact maxima and scales, then the doubtful codes.
template <int LOG2B, int MODE>
__device__ __forceinline__ void tile_settle(const TileParams &p, uint32_t t, TileNotes *notes, TileCollector &to, int lane)
{
    constexpr bool TOK = MODE == ROW_TOKEN || MODE == ROW_FP4;
    const uint32_t piece0 = t * (uint32_t)p.tile_pieces, rp = (uint32_t)p.row_pieces;
    const uint32_t n = min(*reinterpret_cast<volatile uint32_t *>(&notes->count), (uint32_t)TILE_JOBS);
    if (!TOK && n == 0u) return;
    const uint32_t here = min((uint32_t)p.tile_pieces, p.pieces - piece0);              // pieces of the tile
    if (TOK && n <= 32u && *reinterpret_cast<volatile uint32_t *>(&notes->flat) == 0u) {
        const bool has = (uint32_t)lane < n;
        const uint32_t j = has ? notes->job[lane] : 0u, row = (j >> 20) & 31u;
        const bool cand = has && (j >> 30) == (JOB_MAX >> 30);
        const unsigned cands = __ballot_sync(0xffffffffu, cand);
        const unsigned mates = __match_any_sync(0xffffffffu, has ? row : 0x100u + (uint32_t)lane) & cands;      // its row's candidates
        const bool my_row = (uint32_t)lane * rp < here;
        const bool bad = has && __popc(mates) != 1;
        if (!__any_sync(0xffffffffu, bad)) {
            // rows without a candidate are rows of zeros
            const uint32_t rows = __reduce_or_sync(0xffffffffu, cand ? 1u << row : 0u);
            if (my_row && !((rows >> lane) & 1u)) reinterpret_cast<float *>(p.out_scales)[(size_t)(piece0 / rp) + lane] = 0.0f;
            const uint32_t j0 = __shfl_sync(0xffffffffu, j, mates ? __ffs(mates) - 1 : lane);
            const unsigned who = __ballot_sync(0xffffffffu, has);
            to.make_room();
            if (has) {
                TileRecord rec;
                rec.job = j;
                rec.piece = piece0 + (j & 127u);
                rec.aux[0] = piece0 + (j0 & 127u);
                rec.aux[1] = (j0 >> 7) & 127u;
                to.list()[to.n + __popc(who & ((1u << lane) - 1u))] = rec;
            }
            to.n += __popc(who);
            return;
        }
    }
    if (TOK) {
        for (uint32_t k = lane; k < n; k += 32) {
            const uint32_t j = notes->job[k], row = (j >> 20) & 31u, c = (j >> 7) & 127u;
            if ((j >> 30) == (JOB_MAX >> 30)) {
                double S[8], o[4];
                tile_sums_global<LOG2B>(p, piece0 + (j & 127u), c, S);
                tile_quad_of(S, c, o);
                atomicMax(&notes->ex[row], (unsigned long long)__double_as_longlong(tile_abs_max(o)));
            }
        }
        __syncwarp();
        // ---- scales: a row per lane
        if ((uint32_t)lane * rp < here)
            reinterpret_cast<float *>(p.out_scales)[(size_t)(piece0 / rp) + lane] = row_scale(__longlong_as_double((long long)notes->ex[lane]), p.inv_7_sqrt_b, p.sqrt_b, 7.0);
        __syncwarp();
    }
    // ---- doubtful codes
    // (not those of pieces that were quantised again: a correction would meet the new code)
    for (uint32_t k0 = 0; k0 < n; k0 += 32) {
        const uint32_t j = k0 + lane < n ? notes->job[k0 + lane] : 0u, r = j & 127u, c = (j >> 7) & 127u;
        const bool tie = k0 + lane < n && (j >> 30) == (JOB_TIE >> 30) && !((notes->settled[r >> 5] >> (r & 31u)) & 1u);
        if (TOK) {
            if (tie) {
                double S[8];
                tile_sums_global<LOG2B>(p, piece0 + r, c, S);
                const TileScale q = tile_scale_max<MODE>(p, __longlong_as_double((long long)notes->ex[(j >> 20) & 31u]));
                tile_mend(p, piece0 + r, j, tile_code<MODE>(p, tile_output_of(S, c), q));
            }
        } else {
            to.make_room();
            const unsigned who = __ballot_sync(0xffffffffu, tie);
            if (tie) {
                TileRecord rec;
                rec.job = j;
                rec.piece = piece0 + r;
                rec.aux[0] = (uint32_t)notes->aux[r];
                rec.aux[1] = (uint32_t)(notes->aux[r] >> 32);
                to.list()[to.n + __popc(who & ((1u << lane) - 1u))] = rec;
            }
            to.n += __popc(who);
        }
    }
    __syncwarp();
}

// -------------------------------------------------------------------------------------------- the kernel

constexpr int TILE_WGS = 3;                                   // groups of four warps, a tile each
constexpr int TILE_ACCS = 4;                                  // accumulators of 128 columns: one is rotated ahead
constexpr int TILE_STAGES = 6;
constexpr int TILE_NOTES = 6;
constexpr int TILE_SETTLERS = 2;
constexpr int TILE_WARPS = TILE_WGS * 4 + 2 + TILE_SETTLERS;  // one that loads and issues the contractions, one that collects notes, two that settle records
constexpr int TILE_THREADS = TILE_WARPS * 32;
constexpr int TILE_REGS = 128;

struct TileSmem {
    static constexpr uint32_t half = TILE_PIECES * 128;
    static constexpr uint32_t stages = 0;
    static constexpr uint32_t had = stages + TILE_STAGES * 2 * half;
    static constexpr uint32_t notes = had + 2 * TILE_H_BYTES;
    static constexpr uint32_t batches = notes + TILE_NOTES * (uint32_t)sizeof(TileNotes);
    static constexpr uint32_t rows = batches + (uint32_t)sizeof(TileBatches);
    // loaded, empty: of each stage; done, free: of each accumulator; written, free: of each tile's notes and each batch
    static constexpr uint32_t bars = rows + TILE_WGS * (uint32_t)sizeof(TileRows);
    static constexpr uint32_t n_bars = 2 * (TILE_STAGES + TILE_ACCS + TILE_NOTES + TILE_SETTLERS);
    static constexpr uint32_t slot = bars + n_bars * 8;
    static constexpr uint32_t total = slot + 16 + 1024;
};
static_assert(sizeof(TileNotes) % 8 == 0 && sizeof(TileBatches) % 8 == 0 && TileSmem::total <= 227 * 1024, "shared memory of the tile kernel");

// The words of a tile's notes as they are before it.
__device__ __forceinline__ void tile_clear_notes(TileNotes *notes, int lane)
{
    notes->ex[lane] = 0ull;
    if (lane < 4) notes->settled[lane] = 0u;
    if (lane == 0) notes->flat = notes->count = 0u;
}

template <int LOG2B, int MODE>
__global__ void __maxnreg__(TILE_REGS) perq_tile_kernel(const __grid_constant__ CUtensorMap map, const __grid_constant__ TileParams p)
{
    // the quantising warps read the tile (its stage is free when they have left it, otherwise as soon as it is rotated)
    constexpr bool IN_PLACE = MODE == ROW_GROUP || MODE == ROW_MX;
    extern __shared__ __align__(128) unsigned char tsmem_raw[];
    unsigned char *smem = tsmem_raw + ((1024u - (smem_u32(tsmem_raw) & 1023u)) & 1023u);
    const uint32_t base = smem_u32(smem);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t full = base + TileSmem::bars, empty = full + TILE_STAGES * 8, done = empty + TILE_STAGES * 8, avail = done + TILE_ACCS * 8;
    const uint32_t noted = avail + TILE_ACCS * 8, nfree = noted + TILE_NOTES * 8, bfull = nfree + TILE_NOTES * 8, bfree = bfull + TILE_SETTLERS * 8;
    TileNotes *notes = reinterpret_cast<TileNotes *>(smem + TileSmem::notes);

    if (tid < (int)TileSmem::n_bars) {
        const uint32_t bar = full + tid * 8;
        mbar_init(bar, bar >= avail && bar < nfree ? 4 : 1);
        mbar_init_fence();
    }
    if (warp < TILE_NOTES) tile_clear_notes(notes + warp, lane);
    if (warp < TILE_WGS) {
        TileRows *rows = reinterpret_cast<TileRows *>(smem + TileSmem::rows) + warp;
        rows->mx[0][lane] = rows->mx[1][lane] = 0u;
    }
    tile_write_hadamard<LOG2B>(smem + TileSmem::had, tid, TILE_THREADS);
    fence_async_smem();                       // (the operand was written by ordinary stores)
    if (warp == TILE_WGS * 4) tmem_alloc_all(base + TileSmem::slot);
    tmem_fence_before();
    __syncthreads();
    tmem_fence_after();
    griddep_wait();                           // nothing above reads or writes global memory
    griddep_launch();
    const uint32_t tmem = *reinterpret_cast<volatile uint32_t *>(smem + TileSmem::slot);
    const uint32_t first = blockIdx.x, n = first < p.tiles ? (p.tiles - first + gridDim.x - 1) / gridDim.x : 0u;
    auto stage_at = [&](uint32_t s) { return base + TileSmem::stages + s * 2 * TileSmem::half; };
    auto give_up = [&]() { if (lane == 0) atomicOr(&g_perq_device_error, 1u); };
    auto load = [&](uint32_t j) {
        const uint32_t s = j % TILE_STAGES;
        mbar_expect_tx(full + s * 8, (uint32_t)p.tile_pieces * 256u);
        const int y = (int)((first + j * gridDim.x) * (uint32_t)p.tile_pieces);
        tma_load_2d(stage_at(s), &map, 0, y, full + s * 8);
        tma_load_2d(stage_at(s) + TileSmem::half, &map, 64, y, full + s * 8);
    };

    // (a wait that runs out ends its warp's part; the others' waits run out too, and all meet at the end)
    if (warp == TILE_WGS * 4) {
        if (lane == 0) {
            uint32_t loads = 0, j = 0;
            for (; loads < n && loads < TILE_STAGES; ++loads) load(loads);
            for (; j < n; ++j) {
                const uint32_t s = j % TILE_STAGES, b = j % TILE_ACCS;
                bool ok = mbar_wait_fast(full + s * 8, (j / TILE_STAGES) & 1u);
                if (j >= TILE_ACCS) ok = mbar_wait_fast(avail + b * 8, ((j / TILE_ACCS) - 1u) & 1u) && ok;
                if (!ok) { give_up(); break; }
                tmem_fence_after();
                tile_rotate<LOG2B>(tmem + b * 128, stage_at(s), TileSmem::half, base + TileSmem::had);
                tile_commit(done + b * 8);
                if (!IN_PLACE) {
                    tile_commit(empty + s * 8);
                    if (j > 0 && loads < n) {                 // into the stage of the previous tile
                        if (!mbar_wait_fast(empty + (loads % TILE_STAGES) * 8, ((loads / TILE_STAGES) - 1u) & 1u)) { give_up(); break; }
                        load(loads++);
                    }
                }
            }
            // nothing is in flight when the CTA ends, also after a wait that ran out (in place: the collector's loads)
            for (uint32_t k = IN_PLACE ? loads : loads > TILE_STAGES ? loads - TILE_STAGES : 0u; k < loads; ++k)
                (void)mbar_wait_fast(full + (k % TILE_STAGES) * 8, (k / TILE_STAGES) & 1u);
            for (uint32_t k = j > TILE_ACCS ? j - TILE_ACCS : 0u; k < j; ++k) (void)mbar_wait_fast(done + (k % TILE_ACCS) * 8, (k / TILE_ACCS) & 1u);
        }
        __syncwarp();
    } else if (warp == TILE_WGS * 4 + 1) {
        TileCollector to = {reinterpret_cast<TileBatches *>(smem + TileSmem::batches), bfull, bfree, 0u, 0, lane};
        uint32_t loaded = min(n, (uint32_t)TILE_STAGES);       // tiles, of which the first are the other warp's
        for (uint32_t j = 0; j < n; ++j) {
            const uint32_t s = j % TILE_NOTES;
            if (!mbar_wait_fast(noted + s * 8, (j / TILE_NOTES) & 1u)) { give_up(); break; }
            if (IN_PLACE && loaded < n && j + TILE_STAGES == loaded) {                    // (its four warps have left the tile)
                if (lane == 0) load(loaded);
                ++loaded;
            }
            tile_settle<LOG2B, MODE>(p, first + j * gridDim.x, notes + s, to, lane);
            __syncwarp();
            tile_clear_notes(notes + s, lane);
            __syncwarp();
            if (lane == 0) mbar_arrive(nfree + s * 8);
            if (to.n >= 32) to.hand_over(0u);
        }
        to.hand_over(TILE_LAST);
        to.hand_over(TILE_LAST);
        if (IN_PLACE && lane == 0) {                           // (as above)
            for (uint32_t k = loaded > TILE_STAGES ? loaded - TILE_STAGES : 0u; k < loaded; ++k) (void)mbar_wait_fast(full + (k % TILE_STAGES) * 8, (k / TILE_STAGES) & 1u);
        }
        __syncwarp();
    } else if (warp > TILE_WGS * 4 + 1) {
        const TileBatches *batches = reinterpret_cast<const TileBatches *>(smem + TileSmem::batches);
        for (uint32_t k = (uint32_t)(warp - TILE_WGS * 4 - 2);; k += TILE_SETTLERS) {
            const uint32_t s = k & 1u;
            if (!mbar_wait_fast(bfull + s * 8, (k >> 1) & 1u)) { give_up(); break; }
            const uint32_t c = *reinterpret_cast<const volatile uint32_t *>(&batches->count[s]);
            const int m = (int)(c & 0xffffu);
            for (int i = 0; i < m; i += 32) tile_settle_records<LOG2B, MODE>(p, batches->rec[s] + i, m - i, lane);
            __syncwarp();
            if (lane == 0) mbar_arrive(bfree + s * 8);
            if (c & TILE_LAST) break;
        }
    } else {
        const int wg = warp >> 2;
        TileRows *rows = reinterpret_cast<TileRows *>(smem + TileSmem::rows) + wg;
        TileLane L;
        L.w = warp & 3;
        L.lane = lane;
        const int l = L.w * 32 + lane, rp = p.row_pieces;
        L.ri = min(l / rp, TILE_ROW_CAP - 1);
        L.first = l < p.tile_pieces && l % rp == 0;
        L.coupled = (rp & (rp - 1)) != 0 || rp > 32;
        L.whole = (L.w * 32) / rp == (L.w * 32 + 31) / rp && L.w * 32 + 31 < p.tile_pieces;
        for (uint32_t j = (uint32_t)wg; j < n; j += TILE_WGS) {
            const uint32_t s = j % TILE_STAGES, b = j % TILE_ACCS, m = j % TILE_NOTES;
            bool ok = mbar_wait_fast(done + b * 8, (j / TILE_ACCS) & 1u);
            if (IN_PLACE) ok = mbar_wait_fast(full + s * 8, (j / TILE_STAGES) & 1u) && ok;
            if (j >= TILE_NOTES) ok = mbar_wait_fast(nfree + m * 8, ((j / TILE_NOTES) - 1u) & 1u) && ok;
            if (!ok) {                                        // (warps that share rows leave together)
                if (MODE != ROW_GROUP && MODE != ROW_MX && L.coupled) (void)named_barrier_all(1 + wg, 128, false);
                give_up();
                break;
            }
            tmem_fence_after();
            ok = tile_epilogue<LOG2B, MODE>(p, L, tmem + b * 128 + ((uint32_t)(L.w * 32) << 16), stage_at(s), TileSmem::half, first + j * gridDim.x, rows,
                                            (j / TILE_WGS) & 1u, 1 + wg, notes + m);
            if (!ok) { give_up(); break; }
            tmem_fence_before();
            __syncwarp();
            if (lane == 0) {
                mbar_arrive(avail + b * 8);
                mbar_arrive(noted + m * 8);
            }
        }
    }
    tmem_fence_before();
    __syncthreads();
    if (warp == TILE_WGS * 4) {
        tmem_fence_after();
        tmem_free_all(tmem);
    }
}

}  // namespace perq
