// Column kernel: whole-row rotations (b = d = 2048 or 4096) with one scale per token, on the fifth-generation tensor cores.
//
// The rotation is H_d = H_(d/128) (x) H_128.  As in the tile kernel a tile is 128 pieces of 128 adjacent channels (four
// rows of 4096 or eight of 2048), but the operands change places: H_128 is the one with 128 rows, the pieces are the
// columns of the result.  A lane of tensor memory then holds output i of every piece of a row in adjacent columns, so
// that the remaining stages, over the pieces of the row, are butterflies on the 32 values that one load brings -- no trip
// through shared memory and no shuffle.  The outputs go back to tensor memory until the row's maximum is known (forming
// them again took 96 instructions per 1024 elements).  32 x 32 codes of a warp change places in ten shuffles.
//
// The row kernel, which makes a trip through an fp32 tile, spends 1160 warp instructions on 1024 elements and five
// barriers of a row's warps on a row; here two barriers serve four rows.
//
// Error bound.  What the tensor cores lose depends on the inputs: a step adds 16 products to the accumulator, cuts all of
// them at 2^(e-25), e the exponent of the largest, and the sum at 2^(e-23) (measured: a model of that gives the same bits
// on inputs of 4 to 26 binades).  Beside a large input tiny ones can be lost in every piece, to the same side: a bound that
// covers any inputs is 900 * 2^-24 of the row's largest output, and with it a row has six doubtful codes.  But only inputs
// 2^16 below their piece's l1 norm can be lost, and few rows have many: four warps count them (col_lost) while the tile waits
// for its group, 82 of 863 warp instructions on 1024 elements.  (16384 x 4096, INT4: 95 to 98 us; 129 with a bound of 208 * 2^-24 for all rows; 85 with one of 12 that some
// rows exceed.)
//
// Exact maxima and doubtful codes: sums over the whole row.  They are listed while the rows are quantised, and then a warp
// takes the sums of a row (or two): 16384 terms for each of the four.  Rows in which more is listed than fits (ties:
// one nonzero, few small integers; a zero point in doubt) are rotated again in fp64 by the four warps, where every output is
// exact.
#pragma once
#include "perq_tile.cuh"

namespace perq {

constexpr int COL_WGS = 3;
constexpr int COL_ACCS = 4;
constexpr int COL_STAGES = 5;
constexpr int COL_WARPS = COL_WGS * 4 + 4;                    // four that bound the rows' errors; one of them loads, one issues the contractions
constexpr int COL_THREADS = COL_WARPS * 32;
constexpr int COL_LIST = 8;                                   // listed places per row
constexpr int COL_ROWS = 8;                                   // rows per tile at most
constexpr float COL_LOST = 0x1p-12f;                          // of the largest output: where more may be lost the row is rotated in fp64
// The stages over the C pieces of a row round to nearest.  Those of one stage add up to 2^-24 * sqrt(values that meet in an
// output) of the row's largest output at most (Cauchy, Parseval): sqrt(C/2) + sqrt(C/4) + .. + 1.  In 2^-24 of that
// output, a little more than that:
__host__ __device__ constexpr float col_stage_err(int log2c) { return log2c == 5 ? 11.3f : 7.3f; }

struct ColNotes {                                             // of a tile; two per group, used in turn
    float hi[COL_ROWS][4], lo[COL_ROWS][4];                   // fp32 extremes by warp (symmetric: hi is the largest magnitude)
    uint32_t count[COL_ROWS];                                 // more than COL_LIST: the row is rotated again
    uint32_t list[COL_ROWS][COL_LIST];                        // position (12 bits), code as stored (4, from bit 16), doubtful (bit 31) or a candidate
};
struct ColGroup {
    ColNotes notes[2];
    double swap[4][8][32];                                    // exchange between the warps of an fp64 rotation
    unsigned long long ex_hi[4], ex_lo[4];
};

struct ColSmem {
    static constexpr uint32_t half = TILE_PIECES * 128;
    static constexpr uint32_t stages = 0;
    static constexpr uint32_t had = stages + COL_STAGES * 2 * half;
    static constexpr uint32_t groups = had + 2 * half;
    static constexpr uint32_t bars = groups + COL_WGS * (uint32_t)sizeof(ColGroup);
    // loaded, empty: of each stage; done, free: of each accumulator; scanned: of each stage
    static constexpr uint32_t n_bars = 3 * COL_STAGES + 2 * COL_ACCS;
    static constexpr uint32_t lost = bars + n_bars * 8;              // float[COL_ROWS] of each stage
    static constexpr uint32_t slot = lost + COL_STAGES * COL_ROWS * 4;
    static constexpr uint32_t total = slot + 16 + 1024;
};
static_assert(sizeof(ColGroup) % 8 == 0 && ColSmem::total <= 227 * 1024, "shared memory of the column kernel");

// D[i][piece] = H_128 X^T (one thread).
__device__ __forceinline__ void col_rotate(uint32_t tmem, uint32_t tile, uint32_t had)
{
    const uint32_t x = tile_desc(tile), h = tile_desc(had);
#pragma unroll
    for (int s = 0; s < 8; ++s)                               // 16 inputs a step
        tile_mma(tmem, h + (s >> 2) * (ColSmem::half / 16) + 2 * (s & 3), x + (s >> 2) * (ColSmem::half / 16) + 2 * (s & 3), tile_idesc(128), s > 0);
}

// Inputs 8 c .. 8 c + 7 of a piece.
__device__ __forceinline__ void col_words(uint32_t tile, uint32_t r, uint32_t c, uint32_t (&w)[4])
{
    asm volatile("ld.shared.v4.b32 {%0,%1,%2,%3}, [%4];" : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3]) : "r"(tile + tile_at(ColSmem::half, r, 8u * c)));
}
__device__ __forceinline__ uint32_t add_bf16x2(uint32_t a, uint32_t b)
{
    uint32_t r;
    asm("add.rn.bf16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
    return r;
}
__device__ __forceinline__ uint32_t above_bf16x2(uint32_t a, uint32_t b)      // all ones where a > b
{
    uint32_t r;
    asm("set.gt.u32.bf16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
    return r;
}
// -2^(e-16), twice (biased e)
__device__ __forceinline__ uint32_t col_limit(uint32_t e) { return ((e > 16u ? (e - 16u) << 7 : 0u) | 0x8000u) * 0x10001u; }
// Nonzero inputs below 2^(e-16).
__device__ __noinline__ float col_count(uint32_t tile, uint32_t r, uint32_t e)
{
    const uint32_t limit = col_limit(e);
    uint32_t n = 0u;
#pragma unroll 1
    for (uint32_t c = 0; c < 16; ++c) {
        uint32_t w[4];
        col_words(tile, r, c, w);
        // (x - 1 as bits; a zero becomes NaN)
#pragma unroll
        for (int k = 0; k < 4; ++k) n += __popc(above_bf16x2((w[k] | 0x80008000u) - 0x00010001u, limit));
    }
    return (float)(n / 16u);
}
// Bound of what the contraction loses in any output of piece r of a tile, by one lane.  With g = 2^(e-23) and 2^(e+1) above
// the sum of the piece's magnitudes, inputs of 2^7 g and more are multiples of g, every term and sum is below 2^(e+1), and
// all grids that a step cuts at divide g.  A step without smaller inputs only moves the accumulator's part below g, and only
// where its grid is coarser than any before: between two steps that have some, by less than g in all.  A step with n of
// them cuts these and the accumulator, by less than g / 4 each.
// guess: biased e of the lane's piece of the previous tile, plus one.  Inputs are counted against it while they are added
// up, zeros as well; again where it was too low, or there are many.
__device__ __forceinline__ float col_lost(uint32_t tile, uint32_t r, uint32_t &guess)
{
    constexpr float MANY = 12.0f;
    const uint32_t limit = col_limit(guess);
    float a = 0.0f, b = 0.0f;
    uint32_t count = 0u;
#pragma unroll 4
    for (uint32_t c = 0; c < 16; ++c) {
        uint32_t w[4];
        col_words(tile, r, c, w);
#pragma unroll
        for (int k = 0; k < 4; ++k) w[k] |= 0x80008000u;
        const uint32_t s = add_bf16x2(add_bf16x2(w[0], w[1]), add_bf16x2(w[2], w[3]));
        a += __uint_as_float(s);                              // (the lower half only adds to its magnitude)
        b += __uint_as_float(s << 16);
        count += above_bf16x2(w[0], limit) + above_bf16x2(w[1], limit);          // (each half takes off one)
        count += above_bf16x2(w[2], limit) + above_bf16x2(w[3], limit);
    }
    const uint32_t e = (__float_as_uint((a + b) * -1.01f) >> 23) & 0xffu;         // (two roundings to bf16, 17 to fp32)
    const uint32_t lo = (0u - count) & 0xffffu;                                   // (the lower halves' borrows: as many as they count)
    float n = (float)(lo + ((((0u - count) >> 16) + lo) & 0xffffu));
    if (e > guess || n > MANY) n = col_count(tile, r, e);
    guess = min(e, 253u) + 1u;
    return e >= 254u ? 3.0e38f : (n + 5.0f * fminf(n, 8.0f)) * (__uint_as_float(e << 23) * 0x1p-25f);          // (sums that might overflow)
}

// The stages over the pieces of a row: 32 values of one row (LOG2C 5), or 16 each of two (4).
template <int LOG2C>
__device__ __forceinline__ void col_stages(f32x2 (&u)[16])
{
#pragma unroll
    for (int m = 0; m < 16; ++m) u[m] = pack2(u[m].x + u[m].y, u[m].x - u[m].y);
#pragma unroll
    for (int t = 0; t < LOG2C - 1; ++t) {
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

// Exact unnormalised output at position pos of the row whose pieces start at piece r of the tile, by a warp.
template <int LOG2C>
__device__ __noinline__ double col_exact(uint32_t tile, uint32_t r, uint32_t pos, int lane)
{
    constexpr int STEPS = 1 << (LOG2C - 1);                   // of 32 groups of eight inputs: two pieces
    double S[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) S[e] = 0.0;
    // sign of a group: the lane's part of its index, and the step's (bits 8 on of the position)
    const uint32_t own = (uint32_t)__popc(pos & (8u * (uint32_t)lane)) << 31, p0 = (uint32_t)lane >> 4, c = (uint32_t)lane & 15u;
    const uint32_t at = tile + (c >> 3) * ColSmem::half + (r + p0) * 128u;
#pragma unroll 4
    for (int t = 0; t < STEPS; ++t) {
        uint32_t w[4];
        asm volatile("ld.shared.v4.b32 {%0,%1,%2,%3}, [%4];" : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3])
                     : "r"(at + (uint32_t)t * 256u + (((c ^ (r + p0 + 2u * (uint32_t)t)) & 7u) << 4)) : "memory");
        const double f = __hiloint2double((int)(0x77f00000u | (own ^ ((uint32_t)__popc((pos >> 8) & (uint32_t)t) << 31))), 0);          // +-2^896
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            S[2 * j] = fma(bf16_raw_f64(w[j] << 16), f, S[2 * j]);
            S[2 * j + 1] = fma(bf16_raw_f64(w[j]), f, S[2 * j + 1]);
        }
    }
    double v = tile_output_of(S, pos);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return __shfl_sync(0xffffffffu, v, 0) + 0.0;
}

template <int MODE>
__device__ __noinline__ uint32_t col_code(const TileParams &p, double u, const TileScale &q) { return tile_code<MODE>(p, u + 0.0, q); }

template <int MODE>
__device__ __forceinline__ void col_store_scale(const TileParams &p, size_t row, const TileScale &q)
{
    if (MODE == ROW_ASYM) reinterpret_cast<float2 *>(p.out_scales)[row] = make_float2((float)q.s64, (float)q.z64);
    else reinterpret_cast<float *>(p.out_scales)[row] = row_scale(q.a, p.inv_7_sqrt_b, p.sqrt_b, 7.0);
}

// Codes of a lane's column to a run of 32 adjacent positions each: lane l gets piece l of the warp's 32 positions.
__device__ __forceinline__ void col_store(uint8_t *row0, uint32_t row_bytes, int log2c, uint32_t (&cw)[4], int w, int lane, uint32_t rows_left)
{
    row_transpose_codes(cw, 1, lane);
    const uint32_t r = (uint32_t)lane >> log2c, c = (uint32_t)lane & ((1u << log2c) - 1u);
    if (r < rows_left) *reinterpret_cast<uint4 *>(row0 + (size_t)r * row_bytes + c * 64u + (uint32_t)w * 16u) = make_uint4(cw[0], cw[1], cw[2], cw[3]);
}

// A whole row in fp64, by the four warps: scale and codes.
template <int LOG2C, int MODE>
__device__ __noinline__ void col_exact_row(const TileParams &p, uint32_t tile, uint32_t r, size_t row, ColGroup *G, int w, int lane, int bar)
{
    constexpr int C = 1 << LOG2C;
    double v[C];
#pragma unroll
    for (int m = 0; m < C; ++m) v[m] = bf16_raw_f64(lds_u16(tile + tile_at(ColSmem::half, r + m, (uint32_t)(w * 32 + lane))) << 16);
#pragma unroll
    for (int t = 1; t < C; t <<= 1) {
#pragma unroll
        for (int m = 0; m < C; ++m) {
            if ((m & t) == 0) {
                const double a = v[m], c = v[m | t];
                v[m] = a + c;
                v[m | t] = a - c;
            }
        }
    }
#pragma unroll 1
    for (int o = 1; o < 32; o <<= 1) {
        const double sg = (lane & o) ? -1.0 : 1.0;
#pragma unroll
        for (int m = 0; m < C; ++m) v[m] = fma(sg, v[m], __shfl_xor_sync(0xffffffffu, v[m], o));
    }
    const double s1 = (w & 1) ? -1.0 : 1.0, s2 = (w & 2) ? -1.0 : 1.0;
#pragma unroll
    for (int m0 = 0; m0 < C; m0 += 8) {
#pragma unroll
        for (int m = 0; m < 8; ++m) G->swap[w][m][lane] = v[m0 + m];
        named_barrier(bar, 128);
#pragma unroll
        for (int m = 0; m < 8; ++m) {
            const double a = fma(s1, v[m0 + m], G->swap[w ^ 1][m][lane]), b = fma(s1, G->swap[w ^ 2][m][lane], G->swap[w ^ 3][m][lane]);
            v[m0 + m] = fma(s2, a, b) * 0x1p896;
        }
        named_barrier(bar, 128);
    }
    double hi = v[0], lo = v[0];
#pragma unroll
    for (int m = 1; m < C; ++m) { hi = fmax(hi, v[m]); lo = fmin(lo, v[m]); }
    const unsigned long long kh = warp_max_u64(order_key(hi)), kl = warp_max_u64(~order_key(lo));
    if (lane == 0) { G->ex_hi[w] = kh; G->ex_lo[w] = kl; }
    named_barrier(bar, 128);
    unsigned long long h = 0ull, l = 0ull;
#pragma unroll
    for (int k = 0; k < 4; ++k) { h = max(h, G->ex_hi[k]); l = max(l, G->ex_lo[k]); }
    hi = order_value(h);
    lo = order_value(~l);
    const TileScale q = MODE == ROW_ASYM ? tile_scale_asym(p, hi, lo) : tile_scale_max<MODE>(p, fmax(fabs(hi), fabs(lo)));
    if (w == 0 && lane == 0) col_store_scale<MODE>(p, row, q);
    uint32_t cw[4] = {0u, 0u, 0u, 0u};
#pragma unroll
    for (int m = 0; m < C; ++m) cw[m >> 3] |= col_code<MODE>(p, v[m], q) << (4 * (m & 7));
    col_store(p.out_codes + row * (size_t)(64 * C), 64u * C, LOG2C, cw, w, lane, 1u);
    named_barrier(bar, 128);
}

template <int LOG2C, int MODE>
__global__ void __maxnreg__(TILE_REGS) perq_col_kernel(const __grid_constant__ CUtensorMap map, const __grid_constant__ TileParams p)
{
    constexpr int C = 1 << LOG2C, R = TILE_PIECES / C, RU = 32 / C;          // pieces of a row, rows of a tile and of 32 columns
    extern __shared__ __align__(128) unsigned char csmem_raw[];
    unsigned char *smem = csmem_raw + ((1024u - (smem_u32(csmem_raw) & 1023u)) & 1023u);
    const uint32_t base = smem_u32(smem);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t full = base + ColSmem::bars, empty = full + COL_STAGES * 8, done = empty + COL_STAGES * 8, avail = done + COL_ACCS * 8;
    const uint32_t scanned = avail + COL_ACCS * 8;
    float *lost = reinterpret_cast<float *>(smem + ColSmem::lost);

    if (tid < (int)ColSmem::n_bars) {
        const uint32_t bar = full + tid * 8;
        mbar_init(bar, bar >= scanned || (bar >= empty && bar < done) || bar >= avail ? 4 : 1);
        mbar_init_fence();
    }
    for (int e = tid; e < COL_WGS * 2 * COL_ROWS; e += COL_THREADS)
        reinterpret_cast<ColGroup *>(smem + ColSmem::groups)[e / (2 * COL_ROWS)].notes[(e / COL_ROWS) & 1].count[e % COL_ROWS] = 0u;
    for (int e = tid; e < 128 * 64; e += COL_THREADS) {                      // H_128 as an operand
        const int n = e >> 6, k = 2 * (e & 63);
        *reinterpret_cast<uint32_t *>(smem + ColSmem::had + tile_at(ColSmem::half, (uint32_t)n, (uint32_t)k)) = hadamard_bf16(n, k) | (hadamard_bf16(n, k + 1) << 16);
    }
    fence_async_smem();                       // (the operand was written by ordinary stores)
    if (warp == COL_WGS * 4) tmem_alloc_all(base + ColSmem::slot);
    tmem_fence_before();
    __syncthreads();
    tmem_fence_after();
    griddep_wait();                           // nothing above reads or writes global memory
    griddep_launch();
    const uint32_t tmem = *reinterpret_cast<volatile uint32_t *>(smem + ColSmem::slot);
    const uint32_t first = blockIdx.x, n = first < p.tiles ? (p.tiles - first + gridDim.x - 1) / gridDim.x : 0u;
    auto stage_at = [&](uint32_t s) { return base + ColSmem::stages + s * 2 * ColSmem::half; };
    auto give_up = [&]() { if (lane == 0) atomicOr(&g_perq_device_error, 1u); };

    // (a wait that runs out ends its warp's part; the others' waits run out too, and all meet at the end)
    if (warp >= COL_WGS * 4) {
        // a quarter of every tile's pieces each, one per lane.  Tile j is looked at when tile j - 4 has been finished: the three
        // groups are at j - 3 .. j - 1 then, and none waits for this.
        const uint32_t q = (uint32_t)(warp - COL_WGS * 4);
        uint32_t j = 0, loads = 0, guess = 0u;
        bool ok = true;
        auto load = [&]() {
            const uint32_t s = loads % COL_STAGES;
            mbar_expect_tx(full + s * 8, 2 * ColSmem::half);
            const int y = (int)((first + loads * gridDim.x) * (uint32_t)TILE_PIECES);
            tma_load_2d(stage_at(s), &map, 0, y, full + s * 8);
            tma_load_2d(stage_at(s) + ColSmem::half, &map, 64, y, full + s * 8);
            ++loads;
        };
        if (q == 0u && lane == 0) while (loads < n && loads < COL_STAGES) load();
        for (; j < n && ok; ++j) {
            const uint32_t s = j % COL_STAGES, b = j % COL_ACCS;
            if (q == 0u && j >= 4u && j + 1u < n) {
                static_assert(COL_STAGES == 5, "tile j + 1 goes where tile j - 4 was");
                const uint32_t e = (j + 1u) % COL_STAGES;
                ok = mbar_wait_fast(empty + e * 8, ((j + 1u) / COL_STAGES - 1u) & 1u);
                if (ok && lane == 0) load();
            }
            ok = mbar_wait_fast(full + s * 8, (j / COL_STAGES) & 1u) && ok;
            if (q == 1u) {
                if (j >= COL_ACCS) ok = mbar_wait_fast(avail + b * 8, ((j / COL_ACCS) - 1u) & 1u) && ok;
                if (ok && lane == 0) {
                    tmem_fence_after();
                    col_rotate(tmem + b * 128, stage_at(s), base + ColSmem::had);
                    tile_commit(done + b * 8);
                }
            }
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) { give_up(); break; }
            const uint32_t r = 32u * q + (uint32_t)lane;
            float e = col_lost(stage_at(s), r, guess);
#pragma unroll
            for (int o = 1; o < C; o <<= 1) e += __shfl_xor_sync(0xffffffffu, e, o);
            if ((lane & (C - 1)) == 0) lost[s * COL_ROWS + r / C] = e;
            __syncwarp();
            if (lane == 0) mbar_arrive(scanned + s * 8);
        }
        // nothing is in flight when the CTA ends, also after a wait that ran out
        if (q == 0u && lane == 0) {
            for (uint32_t k = loads > COL_STAGES ? loads - COL_STAGES : 0u; k < loads; ++k) (void)mbar_wait_fast(full + (k % COL_STAGES) * 8, (k / COL_STAGES) & 1u);
        }
        if (q == 1u && lane == 0) {
            for (uint32_t k = j > COL_ACCS ? j - COL_ACCS : 0u; k < j; ++k) (void)mbar_wait_fast(done + (k % COL_ACCS) * 8, (k / COL_ACCS) & 1u);
        }
        __syncwarp();
    } else {
        const int wg = warp >> 2, w = warp & 3, bar = 1 + wg;
        ColGroup *G = reinterpret_cast<ColGroup *>(smem + ColSmem::groups) + wg;
        const uint32_t rows_all = p.pieces / C;
        f32x2 u[16];
        for (uint32_t j = (uint32_t)wg, it = 0; j < n; j += COL_WGS, ++it) {
            const uint32_t s = j % COL_STAGES, b = j % COL_ACCS, tile = stage_at(s), acc = tmem + b * 128 + ((uint32_t)(w * 32) << 16);
            const uint32_t row0 = (first + j * gridDim.x) * R, rows = min((uint32_t)R, rows_all - row0);
            ColNotes *N = &G->notes[it & 1u];
            bool ok = mbar_wait_fast(done + b * 8, (j / COL_ACCS) & 1u) && mbar_wait_fast(full + s * 8, (j / COL_STAGES) & 1u) &&
                      mbar_wait_fast(scanned + s * 8, (j / COL_STAGES) & 1u);
            tmem_fence_after();
            // this lane's extremes of row k of 32 columns (symmetric: the largest magnitude)
            auto extremes = [&](int k, float &hi, float &lo) {
                hi = lo = MODE == ROW_ASYM ? u[k * (C / 2)].x : 0.0f;
                float hi2 = hi, lo2 = lo;
#pragma unroll
                for (int m = k * (C / 2); m < (k + 1) * (C / 2); m += 2) {
                    if (MODE == ROW_ASYM) {
                        hi = fmaxf(fmaxf(hi, u[m].x), u[m].y);
                        lo = fminf(fminf(lo, u[m].x), u[m].y);
                        hi2 = fmaxf(fmaxf(hi2, u[m + 1].x), u[m + 1].y);
                        lo2 = fminf(fminf(lo2, u[m + 1].x), u[m + 1].y);
                    } else {
                        hi = max3abs(hi, u[m].x, u[m].y);
                        hi2 = max3abs(hi2, u[m + 1].x, u[m + 1].y);
                    }
                }
                hi = fmaxf(hi, hi2);
                lo = fminf(lo, lo2);
            };
            // ---- extremes of the rows (loops that are not unrolled: these kernels are short of instruction cache)
#pragma unroll 1
            for (int un = 0; un < 4 && ok; ++un) {
                tmem_load32(acc + 32 * un, u);
                col_stages<LOG2C>(u);
                tmem_store32(acc + 32 * un, u);                              // (kept for the codes)
#pragma unroll
                for (int k = 0; k < RU; ++k) {
                    float hi, lo;
                    extremes(k, hi, lo);
                    const int r = un * RU + k;
                    const float wh = warp_max_f32(hi);
                    const float wl = MODE == ROW_ASYM ? warp_min_f32(lo) : 0.0f;
                    if (lane == 0) { N->hi[r][w] = wh; N->lo[r][w] = wl; }
                }
            }
            if (!named_barrier_all(bar, 128, ok)) { give_up(); break; }             // (the four warps leave together)
            if (w == 0 && lane < COL_ROWS) G->notes[(it & 1u) ^ 1u].count[lane] = 0u;      // (everybody has left that tile)
            if (w == 1 && lane < R) {                                        // (much lost: the row again, in fp64)
                const float4 h4 = *reinterpret_cast<const float4 *>(N->hi[lane]), l4 = *reinterpret_cast<const float4 *>(N->lo[lane]);
                float a_row = fmaxf(fmaxf(h4.x, h4.y), fmaxf(h4.z, h4.w));
                if (MODE == ROW_ASYM) a_row = fmaxf(a_row, -fminf(fminf(l4.x, l4.y), fminf(l4.z, l4.w)));
                if (!(lost[s * COL_ROWS + lane] <= fminf(a_row, 3.0e38f) * COL_LOST)) atomicAdd(&N->count[lane], COL_LIST + 1u);
            }
            // ---- codes, by the fp32 extremes
#pragma unroll 1
            for (int un = 0; un < 4; ++un) {
                tmem_load32(acc + 32 * un, u);
                uint32_t cw[4];
                RowQuant Q[RU];
                uint32_t cand = 0u;
#pragma unroll
                for (int k = 0; k < RU; ++k) {
                    const int r = un * RU + k;
                    const float4 h4 = *reinterpret_cast<const float4 *>(N->hi[r]);
                    const float hr = fmaxf(fmaxf(h4.x, h4.y), fmaxf(h4.z, h4.w));
                    const float own_hi = N->hi[r][w], lost_r = lost[s * COL_ROWS + r];
                    if (MODE == ROW_ASYM) {
                        const float4 l4 = *reinterpret_cast<const float4 *>(N->lo[r]);
                        const float lr = fminf(fminf(l4.x, l4.y), fminf(l4.z, l4.w)), a_row = fmaxf(fabsf(hr), fabsf(lr));
                        const float e_row = fmaf(p.err, a_row, lost_r), e_abs = 2.0f * e_row + 2.4e-7f * a_row;
                        const float err = fminf(__fdividef(0.25f * e_row, 0.25f * a_row), 1.0f);
                        float inv, z, slack, per_ref;
                        const bool near = tile_zero_point(hr, lr, err, inv, z, slack, per_ref) && a_row > 0.0f;
                        if (!(a_row > 0.0f)) inv = z = slack = per_ref = 0.0f;
                        Q[k].mul = inv;
                        Q[k].tau = slack + per_ref * a_row;
                        Q[k].magic = 12582912.0f - z;
                        // (a zero point in doubt, extremes that are equal in fp32: the row again, in fp64)
                        if (near && w == 0 && lane == 0) atomicAdd(&N->count[r], COL_LIST + 1u);
                        if (a_row > 0.0f && !near && (own_hi >= hr - e_abs || N->lo[r][w] <= lr + e_abs)) {       // (the same for the warp)
#pragma unroll
                            for (int m = k * (C / 2); m < (k + 1) * (C / 2); ++m) {
                                cand |= (u[m].x >= hr - e_abs || u[m].x <= lr + e_abs ? 1u : 0u) << (2 * m);
                                cand |= (u[m].y >= hr - e_abs || u[m].y <= lr + e_abs ? 2u : 0u) << (2 * m);
                            }
                        }
                    } else {
                        const float e_row = fmaf(p.err, hr, lost_r), thr = hr - (2.0f * e_row + 2.4e-7f * hr), inv = row_inverse(hr);
                        Q[k].mul = inv;
                        Q[k].magic = 12584968.0f;
                        // an element's error and the maximum's; integers: the distance's own
                        Q[k].tau = (2.0f * e_row + 5.0e-7f * hr) * inv + (MODE == ROW_FP4 ? 0.0f : 2.0e-7f);
                        if (hr > 0.0f && own_hi >= thr) {                              // (the same for the warp)
#pragma unroll
                            for (int m = k * (C / 2); m < (k + 1) * (C / 2); ++m)
                                cand |= (fabsf(u[m].x) >= thr ? 1u : 0u) << (2 * m) | (fabsf(u[m].y) >= thr ? 2u : 0u) << (2 * m);
                        }
                    }
                }
                uint32_t tie = 0u;
                if (tile_quantise2<MODE, RU == 2>(u, Q[0], Q[RU - 1], cw)) {
                    tie = row_tie_bits<MODE>(u, Q[0]);
                    if (RU == 2) tie = (tie & 0xffffu) | (row_tie_bits<MODE>(u, Q[RU - 1]) & 0xffff0000u);
                }
                // ---- candidates and doubtful elements of the rows
                if (__any_sync(0xffffffffu, (cand | tie) != 0u)) {
#pragma unroll
                    for (int k = 0; k < RU; ++k) {
                        const int r = un * RU + k;
                        const uint32_t sel = RU == 1 ? 0xffffffffu : 0xffffu << (16 * k);
                        uint32_t cb = (uint32_t)r < rows ? cand & sel : 0u, tb = (uint32_t)r < rows ? tie & sel : 0u;
                        const uint32_t cnt = (uint32_t)(__popc(cb) + __popc(tb));
                        if (cnt != 0u) {
                            uint32_t at = atomicAdd(&N->count[r], cnt);
                            while ((cb | tb) != 0u && at < COL_LIST) {
                                const bool t = cb == 0u;
                                const uint32_t bits = t ? tb : cb, e = (uint32_t)__ffs(bits) - 1u;
                                if (t) tb &= tb - 1u; else cb &= cb - 1u;
                                const uint32_t word = e < 16u ? (e < 8u ? cw[0] : cw[1]) : (e < 24u ? cw[2] : cw[3]);
                                N->list[r][at++] = (t ? 0x80000000u : 0u) | ((word >> (4u * (e & 7u))) & 0xFu) << 16 | ((e & (C - 1u)) * 128u + (uint32_t)(w * 32 + lane));
                            }
                        }
                    }
                }
                const uint32_t r0 = (uint32_t)(un * RU);
                if (r0 < rows) col_store(p.out_codes + (size_t)(row0 + r0) * (64 * C), 64u * C, LOG2C, cw, w, lane, rows - r0);
            }
            tmem_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(avail + b * 8);
            named_barrier(bar, 128);
            // ---- exact sums: a warp the lists of a row, or of two
            uint32_t again = 0u;
#pragma unroll
            for (int r = 0; r < R; ++r)
                if ((uint32_t)r < rows && *reinterpret_cast<volatile uint32_t *>(&N->count[r]) > COL_LIST) again |= 1u << r;
            for (uint32_t r = (uint32_t)(w * (R / 4)); r < (uint32_t)((w + 1) * (R / 4)); ++r) {
                if (r >= rows || ((again >> r) & 1u)) continue;
                const uint32_t cnt = *reinterpret_cast<volatile uint32_t *>(&N->count[r]);
                double a = 0.0, hi = -1.7976931348623157e308, lo = 1.7976931348623157e308;
                uint32_t ties = 0u;
                for (uint32_t k = 0; k < cnt; ++k) {
                    const uint32_t e = N->list[r][k];
                    if (e >> 31) { ties |= 1u << k; continue; }
                    const double v = col_exact<LOG2C>(tile, r * C, e & 0xfffu, lane);
                    a = fmax(a, fabs(v));
                    hi = fmax(hi, v);
                    lo = fmin(lo, v);
                }
                if (MODE == ROW_ASYM && !(hi >= lo)) hi = lo = 0.0;        // (no candidates: a row of zeros)
                if (lane == 0 || ties != 0u) {
                    const TileScale q = MODE == ROW_ASYM ? tile_scale_asym(p, hi, lo) : tile_scale_max<MODE>(p, a);
                    if (lane == 0) col_store_scale<MODE>(p, row0 + r, q);
                    while (ties) {
                        const uint32_t k = (uint32_t)__ffs(ties) - 1u, e = N->list[r][k], pos = e & 0xfffu;
                        ties &= ties - 1u;
                        const double v = col_exact<LOG2C>(tile, r * C, pos, lane);
                        if (lane == 0) {
                            const uint32_t diff = col_code<MODE>(p, v, q) ^ ((e >> 16) & 0xFu);
                            if (diff) atomicXor(reinterpret_cast<uint32_t *>(p.out_codes + (size_t)(row0 + r) * (64 * C)) + (pos >> 3), diff << (4u * (pos & 7u)));
                        }
                    }
                }
                __syncwarp();
            }
            while (again) {
                const uint32_t r = (uint32_t)__ffs(again) - 1u;
                again &= again - 1u;
                col_exact_row<LOG2C, MODE>(p, tile, r * C, (size_t)row0 + r, G, w, lane, bar);
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(empty + s * 8);
        }
    }
    tmem_fence_before();
    __syncthreads();
    if (warp == COL_WGS * 4) {
        tmem_fence_after();
        tmem_free_all(tmem);
    }
}

}  // namespace perq
