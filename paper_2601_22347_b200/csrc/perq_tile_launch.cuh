// Host side of the tile kernels: which calls they take, tensor maps, launches.  Included by perq_api.cu inside its
// anonymous namespace (uses its sm_count, allow_smem, ilog2, is_pow2).
#pragma once

// The driver's encoder of tensor maps, asked for once (the library does not link against libcuda).
typedef CUresult (*TensorMapEncode)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *, const cuuint64_t *, const cuuint32_t *,
                                    const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
TensorMapEncode tensor_map_encode()
{
    static std::atomic<void *> cached{nullptr};
    void *fn = cached.load();
    if (fn == nullptr) {
        cudaDriverEntryPointQueryResult found;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &found) != cudaSuccess ||
            found != cudaDriverEntryPointSuccess) {
            (void)cudaGetLastError();
            return nullptr;
        }
        cached.store(fn);
    }
    return reinterpret_cast<TensorMapEncode>(fn);
}

// x as rows of 128 channels, read in boxes of 64 channels by `rows`, 128-byte swizzle.
bool tile_tensor_map(CUtensorMap *map, const void *x, uint64_t pieces, int rows)
{
    TensorMapEncode encode = tensor_map_encode();
    if (encode == nullptr) return false;
    const cuuint64_t dims[2] = {128, pieces}, strides[1] = {256};
    const cuuint32_t box[2] = {64, (cuuint32_t)rows}, step[2] = {1, 1};
    return encode(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(x), dims, strides, box, step, CU_TENSOR_MAP_INTERLEAVE_NONE,
                  CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// As launch_overlapped, for kernels with a tensor map.
template <typename P>
int launch_with_map(void (*kernel)(CUtensorMap, P), int grid, int threads, size_t smem, cudaStream_t st, const CUtensorMap &map, const P &p)
{
    if (int rc = allow_smem(kernel, smem)) return rc;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (cudaLaunchKernelEx(&cfg, kernel, map, p) != cudaSuccess) {
        (void)cudaGetLastError();
        return PERQ_ERR_CUDA;
    }
    return PERQ_OK;
}

template <int MODE>
int launch_tile_b(int log2b, const CUtensorMap &map, const perq::TileParams &p, int grid, cudaStream_t st)
{
    constexpr int threads = perq::TILE_THREADS;
    constexpr size_t smem = perq::TileSmem::total;
    switch (log2b) {
    case 4: return launch_with_map(perq::perq_tile_kernel<4, MODE>, grid, threads, smem, st, map, p);
    case 5: return launch_with_map(perq::perq_tile_kernel<5, MODE>, grid, threads, smem, st, map, p);
    case 6: return launch_with_map(perq::perq_tile_kernel<6, MODE>, grid, threads, smem, st, map, p);
    default: return launch_with_map(perq::perq_tile_kernel<7, MODE>, grid, threads, smem, st, map, p);
    }
}

// Where the tile kernel is the better one.  It pays 3 to 5 us more than the kernels that rotate in registers (tensor
// memory, operand, the last tile and batch), so calls have to be large; how large depends on what those kernels need, on how
// many lanes of a tile whole rows fill, and on the doubtful codes, which grow with the error bound of b (tile_err).  Both
// sides in us (CUDA graphs, others / tile; laplace and, after a comma, swiglu values), 2^20 elements unless stated:
//   widths that are no multiple of 1024 (row kernel), 9728, 4 / 16: MXFP4 b = 32 10.6 / 8.5, 24 / 13, b = 128 12.1 / 10.7, 27 / 19; per
//     128 b = 32 13 / 8.7, 31 / 15 (2: 8.4 / 7.8); INT4 per token b = 32 10.0 / 9.7, 23 / 18, b = 128 11.9 / 12.7, 27 / 23; FP4 b = 64
//     13.0 / 11.4, 32 / 23, b = 128 12.8 / 13.9, 32 / 26; 8320, whose rows fill half a tile: INT4 b = 64 10.7 / 10.8, 27 / 21
//   MXFP4, 4096, 16: b = 32 13.9 / 12.4, b = 64 15.2 / 14.6; 64: 40 / 34, 42 / 38; b = 128 46 / 55; b = 16 45 / 41, but 8 x 2^22 values of
//     four significant bits 84 / 227
//   per 128, 4096, 16: b = 16 15.9 / 13.9, b = 64 18.6 / 16.0; b = 128 21.2 / 20.7, at 24 28.9 / 27.2
//   INT4 per token, 8 (64): 4096, b = 64 12.7 / 11.9 (43 / 38); b = 128 13.1 / 15.0 (53 / 57); 2048, b = 64 (39 / 48)
//     other widths, 32: b = 32 6144 25.1 / 24.9, 29 / 25, 14336 26 / 22; b = 16 6144 22.4 / 25.2, 14336 23.3 / 21.5; 16: b = 64 3072 17.0 / 16.7,
//     14336 18 / 16; b = 128 12288 22.5 / 20.8, 6144 21.8 / 22.1 (61 / 64)
//   FP4, 1 (16): 4096, b = 32 9.4 / 8.0 (21 / 15), b = 64 10.9 / 8.8 (25 / 18), at 200 161 / 142, 154 / 161; 2048, b = 32 at 32 29.9 / 23.6, at 64
//     51 / 45, 48 / 48, b = 64 at 24 27 / 25, at 48 45 / 50; b = 128, 4096, 64: 60 / 71
//     other widths, 8: b = 32 3072 11.8 / 11.2, 14336 12.5 / 11.7; 16: b = 64 6144 20 / 19, 3072 at 64 56 / 62; b = 128 12288 27 / 23, 6144 25.2 / 24.6 (73 / 81)
// Asymmetric rows are not taken: a zero point in doubt has to be settled while its tile waits, 10 us for the first one; 4096 channels,
// b = 16 at 64 53 / 70, 9728 at 4 12 / 21.
bool tile_is_better(int mode, int d, int b, long long pieces)
{
    const long long M = 8192;                                // pieces of 2^20 elements
    if (d % perq::SEG_ELEMS != 0) return pieces >= (mode == perq::ROW_GROUP ? 2 : b == 128 && mode != perq::ROW_MX ? 16 : 4) * M;
    const bool lean = d == 2048 || d == 4096 || d == 8192;  // (per token: these have a kernel of their own up to b = 128)
    switch (mode) {
    case perq::ROW_MX: return (b == 32 || b == 64) && pieces >= 16 * M;
    case perq::ROW_GROUP: return pieces >= (b == 128 ? 24 : 16) * M;
    case perq::ROW_TOKEN:
        if (lean) return d >= 4096 && b == 64 && pieces >= 8 * M;
        return b >= 64 ? d >= (b == 128 ? 12288 : 3072) && pieces >= 16 * M : d > (b == 16 ? 12288 : 2048) && pieces >= 32 * M;
    default:
        if (lean) return b <= 64 && pieces >= M && pieces <= (d == 2048 ? b == 64 ? 24 : 32 : d == 4096 && b == 64 ? 128 : 1 << 17) * M;
        return b >= 64 ? d >= (b == 128 ? 12288 : 6144) && pieces >= 16 * M : d >= 3072 && pieces >= 8 * M;
    }
}

// Returns -1 if the tile kernel does not take the call.
int try_launch_tile(const void *x, const int32_t *perm, int64_t T, int32_t d, int32_t b, int32_t fmt, int g, void *out_codes, void *out_scales,
                    cudaStream_t st)
{
    if (perm != nullptr || d % 128 != 0 || !is_pow2(b) || b < 16 || b > 128) return -1;
    int mode;
    if (fmt == PERQ_FMT_MXFP4) mode = perq::ROW_MX;
    else if (fmt == PERQ_FMT_FP4) mode = perq::ROW_FP4;
    else if (fmt == PERQ_FMT_INT4 && g == 128) mode = perq::ROW_GROUP;
    else if (fmt == PERQ_FMT_INT4 && g == d) mode = perq::ROW_TOKEN;
    else return -1;
    const bool rows = mode != perq::ROW_MX && mode != perq::ROW_GROUP;
    const int row_pieces = d / 128, row_cap = rows ? perq::TILE_PIECES / row_pieces : 0;
    if (rows && (row_cap < 1 || row_cap > perq::TILE_ROW_CAP)) return -1;
    const long long pieces = (long long)T * row_pieces;
    if (pieces >= (1ll << 31) - perq::TILE_PIECES) return -1;
    if (!tile_is_better(mode, d, b, pieces)) return -1;
    perq::TileParams p;
    std::memset(&p, 0, sizeof(p));
    p.x = static_cast<const uint16_t *>(x);
    p.out_codes = static_cast<uint8_t *>(out_codes);
    p.out_scales = out_scales;
    p.pieces = (uint32_t)pieces;
    p.tile_pieces = rows ? row_cap * row_pieces : perq::TILE_PIECES;
    p.tiles = (uint32_t)((pieces + p.tile_pieces - 1) / p.tile_pieces);
    p.row_pieces = row_pieces;
    p.wide_store = (reinterpret_cast<uintptr_t>(out_codes) & 31u) == 0;
    const int log2b = ilog2(b);
    p.err = perq::tile_err(log2b);
    p.sqrt_b = 0.5 * std::sqrt((double)b);
    p.inv_sqrt_b = 1.0 / p.sqrt_b;
    p.inv_7_sqrt_b = 1.0 / (7.0 * p.sqrt_b);
    const int sms = sm_count();
    if (sms <= 0) return PERQ_ERR_CUDA;
    CUtensorMap map;
    if (!tile_tensor_map(&map, x, (uint64_t)pieces, p.tile_pieces)) return -1;
    const int grid = (int)std::min<long long>(p.tiles, sms);
    switch (mode) {
    case perq::ROW_MX: return launch_tile_b<perq::ROW_MX>(log2b, map, p, grid, st);
    case perq::ROW_FP4: return launch_tile_b<perq::ROW_FP4>(log2b, map, p, grid, st);
    case perq::ROW_GROUP: return launch_tile_b<perq::ROW_GROUP>(log2b, map, p, grid, st);
    default: return launch_tile_b<perq::ROW_TOKEN>(log2b, map, p, grid, st);
    }
}

// x as boxes of eight rows by 512 channels: 64 channels, the rows, blocks of 64 channels.
bool perm_tensor_map(CUtensorMap *map, const void *x, uint64_t T, int d)
{
    TensorMapEncode encode = tensor_map_encode();
    if (encode == nullptr) return false;
    const cuuint64_t dims[3] = {64, T, (cuuint64_t)d / 64}, strides[2] = {(cuuint64_t)d * 2, 128};
    const cuuint32_t box[3] = {64, perq::PERM_ROWS, perq::PERM_BOX / 64}, step[3] = {1, 1, 1};
    return encode(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void *>(x), dims, strides, box, step, CU_TENSOR_MAP_INTERLEAVE_NONE,
                  CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <int MODE>
int launch_perm_b(int log2b, const CUtensorMap &map, const perq::PermParams &p, int grid, size_t smem, cudaStream_t st)
{
    constexpr int threads = perq::PERM_THREADS;
    switch (log2b) {
    case 4: return launch_with_map(perq::perq_perm_kernel<4, MODE>, grid, threads, smem, st, map, p);
    case 5: return launch_with_map(perq::perq_perm_kernel<5, MODE>, grid, threads, smem, st, map, p);
    case 6: return launch_with_map(perq::perq_perm_kernel<6, MODE>, grid, threads, smem, st, map, p);
    default: return launch_with_map(perq::perq_perm_kernel<7, MODE>, grid, threads, smem, st, map, p);
    }
}

// Where the kernel for many permuted rows is the better one: widths that are no multiple of 1024, whose permuted rows were the row kernel's
// (us, others / this one; gaussian and, after a comma, swiglu values).  A set of eight rows to every second SM at least; fewer rows
// at 9728 are better spread by the row kernel (148 rows, MXFP4 b = 32: 7.7 / 10.3; 300 rows, b = 128: 13.5 / 14.5).
//   MXFP4, 9728: b = 16, 592 rows 24 / 17, 8192 rows 240 / 103; b = 32, 1200 rows 44 / 27, 33.5 / 23.1, 8192 rows 176 / 82; b = 128, 592 rows 20.4 / 18.0,
//     8192 rows 195 / 121; 4736: b = 32, 592 rows 11.0 / 7.8, 2368 rows 25.5 / 17.4; 640 and 1152: 592 rows 6.1 .. 8.4 / 5.9 .. 6.5
//   INT4 per 128, 9728: b = 16, 592 rows 22.9 / 15.5; b = 128, 1200 rows 50.7 / 27.6, 8192 rows 282 / 106; 1152: b = 128, 8192 rows 40 / 25
//   One nonzero, integers, few nonzeros, equal values, zeros, eight shapes from 592 x 640 to 2368 x 4736: 0.07 .. 1.0 of the row kernel's time, but up to
//     1.2 for small integers and 2 % of nonzeros in MXFP4, b = 16 .. 64 (592 x 640, 2 % of nonzeros, b = 64: 1.7)
// Widths of 1024 k stay with the group kernel, which has no ragged segments: 4096 x 8192, MXFP4, b = 32 37.6 / 41.8; per 128, b = 128 48.0 / 49.9.
// (Here a set's rows are interleaved while no unit is being rotated: a third of the time at 8192 channels, whose interleaved rows fill
// half of the shared memory.)
bool perm_is_better(int d, long long T) { return d % perq::SEG_ELEMS != 0 && T >= 592; }

// Returns -1 if that kernel does not take the call.
int try_launch_perm(const void *x, const int32_t *perm, int64_t T, int32_t d, int32_t b, int32_t fmt, int g, void *out_codes, void *out_scales,
                    cudaStream_t st)
{
    if (perm == nullptr || d % 128 != 0 || !is_pow2(b) || b < 16 || b > 128) return -1;
    int mode;
    if (fmt == PERQ_FMT_MXFP4) mode = perq::ROW_MX;
    else if (fmt == PERQ_FMT_INT4 && g == 128) mode = perq::ROW_GROUP;
    else return -1;
    if (T >= (1ll << 31) - perq::PERM_ROWS || !perm_is_better(d, T)) return -1;
    const int boxes = (d + perq::PERM_BOX - 1) / perq::PERM_BOX;
    const perq::PermLayout lay(d, boxes, (uint32_t)kMaxSmem);
    if (lay.stages < 4) return -1;
    perq::PermParams p;
    std::memset(&p, 0, sizeof(p));
    p.perm = perm;
    p.out_codes = static_cast<uint8_t *>(out_codes);
    p.out_scales = out_scales;
    p.T = (uint32_t)T;
    p.sets = (uint32_t)((T + perq::PERM_ROWS - 1) / perq::PERM_ROWS);
    p.d = d;
    p.units = d / 128;
    p.boxes = boxes;
    p.stages = lay.stages;
    p.off_ring = lay.ring;
    p.off_tab = lay.tab;
    p.off_bars = lay.bars;
    p.sqrt_b = std::sqrt((double)b);
    p.inv_7_sqrt_b = 1.0 / (7.0 * p.sqrt_b);
    const int sms = sm_count();
    if (sms <= 0) return PERQ_ERR_CUDA;
    CUtensorMap map;
    if (!perm_tensor_map(&map, x, (uint64_t)T, d)) return -1;
    const int tail = (int)(p.sets % (uint32_t)sms);
    p.parts = tail > 0 ? std::min(sms / tail, (p.units + perq::PERM_WARPS - 1) / perq::PERM_WARPS) : 1;
    const int grid = p.sets >= (uint32_t)sms ? sms : tail * p.parts;
    return mode == perq::ROW_MX ? launch_perm_b<perq::ROW_MX>(ilog2(b), map, p, grid, lay.total, st)
                                : launch_perm_b<perq::ROW_GROUP>(ilog2(b), map, p, grid, lay.total, st);
}

// Where the column kernel is better than the row kernel (us, CUDA graphs, row / column, laplace and swiglu values): 4096
// channels, 2048 rows 18.4 / 21.9, 18.6 / 21.4, 4096 rows 31.3 / 30.0, 30.9 / 29.8, 8192 rows 58.5 / 53.0, 58.9 / 53.7, 16384 rows 113 / 98,
// 113 / 99; FP4 62.0 / 56.1 and 117 / 99; asymmetric, 4096 rows 51 / 40, 16384 rows 191 / 134.  2048 channels, 8192 rows 30.8 / 31.6, 16384
// rows 58.0 / 54.9; FP4 59.4 / 55.8, asymmetric 95 / 80.
bool col_is_better(int mode, int d, long long pieces)
{
    return pieces >= (d == 2048 ? 16 * 16384 : 32 * (mode == perq::ROW_ASYM ? 4096 : 8192));
}

// Whole-row rotations of 2048 and 4096 channels with one scale per token.  Returns -1 if the column kernel does not take
// the call.
int try_launch_col(const void *x, const int32_t *perm, int64_t T, int32_t d, int32_t b, int32_t fmt, int g, void *out_codes, void *out_scales,
                   cudaStream_t st)
{
    if (perm != nullptr || b != d || (d != 2048 && d != 4096)) return -1;
    int mode;
    if (fmt == PERQ_FMT_FP4) mode = perq::ROW_FP4;
    else if (fmt == PERQ_FMT_INT4_ASYM) mode = perq::ROW_ASYM;
    else if (fmt == PERQ_FMT_INT4 && g == d) mode = perq::ROW_TOKEN;
    else return -1;
    const long long pieces = (long long)T * (d / 128);
    if (pieces >= (1ll << 31) - perq::TILE_PIECES) return -1;
    if (!col_is_better(mode, d, pieces)) return -1;
    perq::TileParams p;
    std::memset(&p, 0, sizeof(p));
    p.x = static_cast<const uint16_t *>(x);
    p.out_codes = static_cast<uint8_t *>(out_codes);
    p.out_scales = out_scales;
    p.pieces = (uint32_t)pieces;
    p.tile_pieces = perq::TILE_PIECES;
    p.tiles = (uint32_t)((pieces + perq::TILE_PIECES - 1) / perq::TILE_PIECES);
    p.row_pieces = d / 128;
    p.err = perq::col_stage_err(ilog2(d) - 7) * perq::TWO_M24;      // (what the contraction loses is added row by row)
    p.sqrt_b = std::sqrt((double)b);
    p.inv_sqrt_b = 1.0 / p.sqrt_b;
    p.inv_7_sqrt_b = 1.0 / (7.0 * p.sqrt_b);
    const int sms = sm_count();
    if (sms <= 0) return PERQ_ERR_CUDA;
    CUtensorMap map;
    if (!tile_tensor_map(&map, x, (uint64_t)pieces, perq::TILE_PIECES)) return -1;
    const int grid = (int)std::min<long long>(p.tiles, sms);
    constexpr int threads = perq::COL_THREADS;
    constexpr size_t smem = perq::ColSmem::total;
    const bool wide = d == 4096;
    switch (mode) {
    case perq::ROW_FP4: return launch_with_map(wide ? perq::perq_col_kernel<5, perq::ROW_FP4> : perq::perq_col_kernel<4, perq::ROW_FP4>, grid, threads, smem, st, map, p);
    case perq::ROW_ASYM: return launch_with_map(wide ? perq::perq_col_kernel<5, perq::ROW_ASYM> : perq::perq_col_kernel<4, perq::ROW_ASYM>, grid, threads, smem, st, map, p);
    default: return launch_with_map(wide ? perq::perq_col_kernel<5, perq::ROW_TOKEN> : perq::perq_col_kernel<4, perq::ROW_TOKEN>, grid, threads, smem, st, map, p);
    }
}
