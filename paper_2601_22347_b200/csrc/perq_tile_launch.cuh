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
// memory, operand, the last tile and batch), so calls have to be large; how large depends on what those kernels need.  Both
// sides in us (CUDA graphs, others / tile), 2^20 elements unless stated:
//   widths that are no multiple of 1024 (row kernel), 9728, b = 32, 4 / 16: MXFP4 9.4 / 7.3, 22 / 12; per 128 12 / 7.5, 30 / 13;
//     INT4 per token 9.4 / 8.5, 24 / 16; FP4 11 / 8.6, 29 / 16; asymmetric 12 / 10, 31 / 23.  (2: 0.8 .. 1.1 of the others' rate.)
//   MXFP4, 4096, 16: b = 32 13.9 / 12.4, 64 14.5 / 13.9, 128 15.1 / 14.8; b = 16 13.7 / 14.1, at 32 21.5 / 21.0
//   per 128, 4096, 16 (8): b = 16 15.0 / 13.1 (9.5 / 9.3), b = 128 20.1 / 18.0 (12.7 / 12.7)
//   INT4 per token, 4096, 8: b = 32 9.2 / 9.5, 64 11.4 / 10.0, 128 12.5 / 11.4; 2048, 16: 64 15.9 / 13.2, but 64: 38.7 / 44.2;
//     14336, 16 (4): b = 16 13.9 / 12.5 (6.0 / 7.5), 128 22.1 / 15.3 (8.8 / 9.4)
//   FP4, 4096, 1: b = 32 8.6 / 6.7, 64 9.4 / 7.0; 128 7.3 / 8.1, at 8 14.2 / 11.5; 14336, 8: 12.4 / 9.4, 14.8 / 11.6
//   asymmetric, 4096, 16: b = 32 21.5 / 17.9, 64 24 / 18.4, 128 26.8 / 22.2, b = 16 20.7 / 18.4, but 64: 52.4 / 54.6
bool tile_is_better(int mode, int d, int b, long long pieces)
{
    const long long M = 8192;                                // pieces of 2^20 elements
    if (d % perq::SEG_ELEMS != 0) return pieces >= (mode == perq::ROW_GROUP ? 2 : 4) * M;
    const bool lean = d == 2048 || d == 4096 || d == 8192;  // (per token: these have a kernel of their own up to b = 64)
    switch (mode) {
    case perq::ROW_MX: return pieces >= (b == 16 ? 32 : 16) * M;
    case perq::ROW_GROUP: return pieces >= 16 * M;
    case perq::ROW_TOKEN: return lean ? d >= 4096 && b >= 64 && pieces >= 8 * M : d >= 3072 && pieces >= 16 * M;
    case perq::ROW_FP4: return lean && b <= 64 ? pieces >= M : d >= 3072 && pieces >= 8 * M;
    default: return d >= 3072 && (b >= 32 || !lean) && pieces >= 16 * M;
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
    else if (fmt == PERQ_FMT_INT4_ASYM) mode = perq::ROW_ASYM;
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
    p.err = perq::FAST_ERR_K * (float)log2b * perq::TWO_M24;
    p.sqrt_b = std::sqrt((double)b);
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
    case perq::ROW_ASYM: return launch_tile_b<perq::ROW_ASYM>(log2b, map, p, grid, st);
    case perq::ROW_GROUP: return launch_tile_b<perq::ROW_GROUP>(log2b, map, p, grid, st);
    default: return launch_tile_b<perq::ROW_TOKEN>(log2b, map, p, grid, st);
    }
}

// Where the column kernel is better than the row kernel (us, CUDA graphs, row / column, laplace and swiglu values): 4096
// channels, 2048 rows 18.4 / 21.9 and 18.6 / 21.4, 4096 rows 31.3 / 30.0 and 30.9 / 29.8, 16384 rows 113 / 98 and 113 / 99;
// FP4 33.0 / 31.0, 117 / 99; asymmetric 51 / 40, 191 / 134.  2048 channels, 8192 rows 30.8 / 31.6, 16384 rows 58.0 / 54.9;
// FP4 59.4 / 55.8, asymmetric 95 / 80.
bool col_is_better(int d, long long pieces) { return pieces >= (d == 2048 ? 16 * 16384 : 32 * 4096); }

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
    if (!col_is_better(d, pieces)) return -1;
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
