// Algorithm 1 (MassDiff) on the device, so that a calibration pass (statistic -> permutation -> permuted
// rotate+quantize) never leaves the GPU.  Same rules as the host function: channels in descending mass
// (equal masses: lower channel first), each to the open block with the smallest running sum (equal sums:
// lower block first), running sums in double, perm = the blocks concatenated.
//
// Two kernels.  Ranks by counting: d^2 comparisons spread over the grid (32 channels per CTA, its eight warps
// share the d comparisons of a channel), two instructions each.  Then the greedy itself, one CTA, in BATCHES:
//
//   The open blocks are kept in a list sorted by (running sum, block).  If the next channels were handed to
//   the blocks of the list in order, block i would reach new_i = s_i + c_i.  That is what the one-by-one
//   greedy does as long as no block that has received a channel has become the lightest again.  Let M be the
//   smallest (new_i, block).  new_i >= s_i, so every list entry above M comes after M's own entry: the entries
//   up to M are exactly the prefix that the greedy serves before it returns to a block.  That prefix is served
//   at once, and its new sums are merged into the list.
//
// Sums differ by about one channel mass, so a batch serves most of the blocks: 66 batches for 8192 channels of a
// real statistic in 256 blocks, 176 us (one channel at a time, one warp scanning all running sums: 2316 us).  Up to 256
// blocks the batches are formed by another kernel (below).
// Masses that fall steeply make small batches, and few blocks small ones anyway.  Channels are then served one by one by
// one warp: 32 channels reach no more than the first 32 entries of the list, so a lane holds one entry in registers and a
// channel costs three warp reductions; afterwards the entries are merged back like a batch.  (By all threads, a barrier
// and an insertion into the list per channel, 8192 steeply falling masses took 2593 us, 4096 channels in four blocks 2813;
// this way 1030 and 594.  The scan: 2303 and 860.)
// Zero masses (padded channels) change no sum, and a last open block takes what is left: no greedy is needed then.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "perq_fast.cuh"

namespace perq {

constexpr int MD_RANK_THREADS = 256;
constexpr int MD_RANK_CHANNELS = 32;     // channels per CTA of the ranking
constexpr int MD_TILE = 8192;            // masses staged at a time
constexpr int MD_MAX_BLOCKS = 4096;      // the list lives in shared memory
constexpr int MD_MAX_THREADS = 1024;
constexpr int MD_WINDOW = 2048;          // ordered channels staged at a time by the greedy

struct MassdiffParams {
    const float *a;          // [d] channel masses
    int32_t *order;          // [d] channels by rank
    int32_t *perm;           // [d]
    int d, b;
};

// Shared memory of the greedy: two lists (sum; block and its fill count in one word), the new sums, fp32 distances,
// the channel window, and a few words of reduction space.
struct MdSmem {
    size_t sum0, sum1, fresh, key, key_old, id0, id1, place, crowded, doubtful, chan, mass, red, total;
    __host__ __device__ explicit MdSmem(int n)
    {
        const size_t m = ((size_t)n + 3) & ~(size_t)3;
        size_t o = 0;
        sum0 = o;  o += m * 8;
        sum1 = o;  o += m * 8;
        fresh = o; o += m * 8;
        key = o;   o += m * 4;
        key_old = o; o += m * 4;
        id0 = o;   o += m * 4;
        id1 = o;   o += m * 4;
        place = o; o += m * 4;
        crowded = o; o += m;
        doubtful = o; o += m * 2;
        o = (o + 15) & ~(size_t)15;
        chan = o;  o += (size_t)MD_WINDOW * 4;
        mass = o;  o += (size_t)MD_WINDOW * 4;
        red = o;   o += 32 * 16;
        total = o;
    }
};

// A mass as both kernels see it: NaN and negative values count as 0, infinity as the largest float.  The entry point asks
// for finite non-negative masses; with others in the list, places would collide without being noticed (NaN compares
// with nothing, negative sums order the wrong way round as bit patterns), and a place that nobody has written holds
// no block.
__device__ __forceinline__ float md_mass(float a) { return fminf(fmaxf(a, 0.0f), 3.4028234663852886e38f); }

// Counting by packed fp32 adds: 1.0 for every comparison that holds, two per add (1.5 instructions a comparison
// where an integer count took 3; counts stay below 2^24, so they are exact).
__device__ __forceinline__ float md_gt(float a, float b) { float r; asm("set.gt.f32.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b)); return r; }
__device__ __forceinline__ float md_ge(float a, float b) { float r; asm("set.ge.f32.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b)); return r; }

// order[r] = the channel of rank r (rank = number of channels that come before it).  A lane counts for one
// channel; the staged masses are read four at a time, the same ones by every lane.  Before the CTA's own 32
// channels an equal mass comes first, after them it does not: one comparison per mass except among the 32.
__global__ void __launch_bounds__(MD_RANK_THREADS) perq_massdiff_rank_kernel(MassdiffParams p)
{
    __shared__ __align__(16) float tile[MD_TILE];
    __shared__ int part[MD_RANK_THREADS];
    griddep_wait();
    griddep_launch();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int i0 = blockIdx.x * MD_RANK_CHANNELS, i = i0 + lane;
    const float ai = (i < p.d) ? md_mass(p.a[i]) : 0.0f;
    const float nan = __int_as_float(0x7fffffff);        // padding: no comparison holds
    int rank = 0;
    f32x2 c0 = pack2(0.0f, 0.0f), c1 = c0;
    for (int k0 = 0; k0 < p.d; k0 += MD_TILE) {
        const int kn = min(MD_TILE, p.d - k0);
        const int per = ((kn + 255) / 256) * 32;         // masses per warp: a multiple of 32
        __syncthreads();
        for (int k = threadIdx.x; k < per * 8; k += MD_RANK_THREADS) tile[k] = (k < kn) ? md_mass(p.a[k0 + k]) : nan;
        __syncthreads();
        const int lo = warp * per, hi = lo + per, own = i0 - k0;       // all multiples of 32
        const float4 *t4 = reinterpret_cast<const float4 *>(tile);
        const int before = min(hi, own);
#pragma unroll 8
        for (int k = lo; k < before; k += 4) {
            const float4 v = t4[k >> 2];
            c0 = add2(c0, pack2(md_ge(v.x, ai), md_ge(v.y, ai)));
            c1 = add2(c1, pack2(md_ge(v.z, ai), md_ge(v.w, ai)));
        }
        if (own >= lo && own < hi) {
            for (int k = own; k < own + 32; ++k) {
                const float ak = tile[k];
                rank += (ak > ai || (ak == ai && k0 + k < i)) ? 1 : 0;
            }
        }
#pragma unroll 8
        for (int k = max(lo, own + 32); k < hi; k += 4) {
            const float4 v = t4[k >> 2];
            c0 = add2(c0, pack2(md_gt(v.x, ai), md_gt(v.y, ai)));
            c1 = add2(c1, pack2(md_gt(v.z, ai), md_gt(v.w, ai)));
        }
    }
    rank += (int)((c0.x + c0.y) + (c1.x + c1.y));
    part[threadIdx.x] = rank;
    __syncthreads();
    if (warp == 0 && i < p.d) {
#pragma unroll
        for (int w = 1; w < MD_RANK_THREADS / 32; ++w) rank += part[w * 32 + lane];
        p.order[min(rank, p.d - 1)] = i;
    }
}

// Running sums are non-negative doubles, so their bit patterns order like the values.  An entry's second word:
// block in the low MD_ID_BITS bits, channels it has received above them.
constexpr int MD_ID_BITS = 13;
constexpr int MD_ID_MASK = (1 << MD_ID_BITS) - 1;
__device__ __forceinline__ bool md_less(unsigned long long s, int i, unsigned long long t, int j)
{
    return s < t || (s == t && (i & MD_ID_MASK) < (j & MD_ID_MASK));
}

// A batch costs as much as 16 channels one by one.  Below 6 channels it is followed by 32 of those, by two and four
// times 32 if the next batches are small again; up to 16 blocks (in the kernel below) all channels go one by one.  (Whenever 32 blocks or
// fewer are open: 244 against 176 us for the 8192 channels above, whose last blocks fill in large batches.)
constexpr int MD_FEW_BLOCKS = 16;
constexpr int MD_SERIAL_K = 6;
constexpr int MD_SERIAL_RUNS = 4;

// The smallest (sum, block) of a warp's lanes.
__device__ __forceinline__ void md_warp_min(unsigned long long v, int blk, unsigned long long &m, int &m_blk)
{
    const uint32_t hi = (uint32_t)(v >> 32), lo = (uint32_t)v;
    const uint32_t mhi = __reduce_min_sync(0xffffffffu, hi);
    const uint32_t mlo = __reduce_min_sync(0xffffffffu, hi == mhi ? lo : 0xffffffffu);
    m_blk = (int)__reduce_min_sync(0xffffffffu, (hi == mhi && lo == mlo) ? (uint32_t)blk : (uint32_t)MD_ID_MASK);
    m = ((unsigned long long)mhi << 32) | mlo;
}

__global__ void __launch_bounds__(MD_MAX_THREADS, 1) perq_massdiff_greedy_kernel(MassdiffParams p)
{
    extern __shared__ __align__(16) unsigned char md_smem[];
    const int d = p.d, b = p.b, n = d / b;
    const MdSmem lay(n);
    unsigned long long *sum = (unsigned long long *)(md_smem + lay.sum0), *sum_next = (unsigned long long *)(md_smem + lay.sum1);
    unsigned long long *fresh = (unsigned long long *)(md_smem + lay.fresh);
    float *key = (float *)(md_smem + lay.key), *key_old = (float *)(md_smem + lay.key_old);
    int *id = (int *)(md_smem + lay.id0), *id_next = (int *)(md_smem + lay.id1);
    int *place = (int *)(md_smem + lay.place), *chan = (int *)(md_smem + lay.chan);
    unsigned char *crowded = md_smem + lay.crowded;
    unsigned short *doubtful = (unsigned short *)(md_smem + lay.doubtful);
    float *mass = (float *)(md_smem + lay.mass);
    unsigned long long *red_sum = (unsigned long long *)(md_smem + lay.red);
    int *red_id = (int *)(md_smem + lay.red + 32 * 8), *red_open = (int *)(md_smem + lay.red + 32 * 12);
    const int tid = threadIdx.x, nthr = blockDim.x, lane = tid & 31, warp = tid >> 5;
    const unsigned long long INF = 0x7ff0000000000000ull;
    auto swap_lists = [&]() {
        unsigned long long *t = sum; sum = sum_next; sum_next = t;
        int *u = id; id = id_next; id_next = u;
    };

    for (int j = tid; j < n; j += nthr) { sum[j] = 0ull; id[j] = j; crowded[j] = 0; }
    if (tid < 32) { red_sum[tid] = INF; red_id[tid] = MD_ID_MASK; red_open[tid] = 0; }
    griddep_wait();             // nothing above reads or writes global memory
    griddep_launch();
    int split = 0;              // log2 of the threads that count for one entry
    while (split < 1 && (n << (split + 1)) <= nthr) ++split;
    int m = n;                  // open blocks: list entries [0, m)
    int s = 0, w0 = 0, w1 = 0;  // next rank; staged window of ranks [w0, w1)
    int serial = 0, runs = 1;   // runs of 32 channels still to be served one by one; after the next small batch
    uint32_t batch = 0;
    while (s < d) {
        if (s >= w1) {
            __syncthreads();    // everybody has read the last window
            w0 = s;
            w1 = min(d, s + MD_WINDOW);
            for (int k = tid; k < w1 - w0; k += nthr) {
                const int c = min(max(p.order[w0 + k], 0), d - 1);
                chan[k] = c;
                mass[k] = md_mass(p.a[c]);
            }
            __syncthreads();
        }
        if (m == 1 || mass[s - w0] == 0.0f) break;          // one block or only zero masses are left: below
        const bool one_by_one = serial > 0;
        unsigned long long M;                     // the smallest new sum
        int M_id = MD_ID_MASK, K, q, steps, given;
        if (one_by_one) {
            // ---- 32 channels one by one: lane j of warp 0 has entry j
            --serial;
            if (warp == 0) {
                const int room = min(32, w1 - s);
                unsigned long long v = lane < m ? sum[lane] : ~0ull;
                int e = lane < m ? id[lane] : MD_ID_MASK, t = 0;
                const int e0 = e;
                for (; t < room; ++t) {
                    const float a = mass[s - w0 + t];
                    if (a == 0.0f) break;
                    unsigned long long least;
                    int blk;
                    md_warp_min(v, e & MD_ID_MASK, least, blk);
                    if (v == least && (e & MD_ID_MASK) == blk && lane < m) {
                        const int f = e >> MD_ID_BITS;
                        p.perm[(size_t)blk * b + f] = chan[s - w0 + t];
                        const double ns = __longlong_as_double((long long)v) + (double)a;
                        v = f + 1 < b ? (unsigned long long)__double_as_longlong(ns) : INF;
                        e += 1 << MD_ID_BITS;
                    }
                }
                if (lane < m) { fresh[lane] = v; id[lane] = e; }
                // (the entries that were served are a prefix of the list)
                const unsigned touched = __ballot_sync(0xffffffffu, e != e0);
                md_warp_min(e != e0 ? v : INF, e & MD_ID_MASK, M, M_id);
                if (lane == 0) { red_sum[0] = M; red_open[3] = t; red_open[4] = max(1, 32 - __clz((int)touched)); }
            }
            __syncthreads();
            M = red_sum[0];
            steps = red_open[3];
            K = q = red_open[4];
            given = 0;                            // (the entries' fill counts and perm are written)
        } else {
            // ---- the sums that the next q blocks of the list would reach, and the smallest of them
            q = min(m, w1 - s);
            unsigned long long best = INF;
            int best_id = MD_ID_MASK;
            for (int j = tid; j < q; j += nthr) {
                const double ns = __longlong_as_double((long long)sum[j]) + (double)mass[s - w0 + j];
                const unsigned long long v = ((id[j] >> MD_ID_BITS) + 1 < b) ? (unsigned long long)__double_as_longlong(ns) : INF;
                fresh[j] = v;
                if (v != INF && md_less(v, id[j], best, best_id)) { best = v; best_id = id[j] & MD_ID_MASK; }
            }
            md_warp_min(best, best_id, M, M_id);
            if (lane == 0) { red_sum[warp] = M; red_id[warp] = M_id; }
            __syncthreads();
            md_warp_min(red_sum[lane], red_id[lane], M, M_id);
            K = steps = 0;
            given = 1 << MD_ID_BITS;
        }
        // ---- K: the list entries up to M.  Distances of all sums to M in fp32 (sums within a batch are close
        // to each other: the difference, not the sum, is what fp32 resolves)
        const double m64 = __longlong_as_double((long long)M);
        for (int j = tid; j < m; j += nthr) {
            key_old[j] = (float)(__longlong_as_double((long long)sum[j]) - m64);
            if (j < q) key[j] = (fresh[j] != INF) ? (float)(__longlong_as_double((long long)fresh[j]) - m64) : __int_as_float(0x7f800000);
        }
        if (one_by_one) {
            __syncthreads();
        } else {
            for (int j0 = 0; j0 < q; j0 += nthr) {
                const int j = j0 + tid;
                K += __syncthreads_count(j < q && !md_less(M, M_id, sum[min(j, q - 1)], id[min(j, q - 1)]));
            }
            K = steps = max(K, 1);
            if (K < MD_SERIAL_K && K < q) { serial = runs; runs = min(2 * runs, MD_SERIAL_RUNS); }
            else if (K < q) runs = 1;
        }
        // ---- serve them; every entry's place in the merged list: new sums below it (counted, 2^split threads
        // to an entry), and for a new sum the untouched entries below it (searched).  fp32 distances to M
        // decide; equal ones (masses are sums of bf16: equal sums do occur, a few per batch) show as entries that
        // took one place.
        int *closed = red_open + (batch & 1u), *closed_next = red_open + ((batch + 1) & 1u);
        for (int j0 = 0; j0 < m; j0 += nthr >> split) {
            const int j = j0 + (tid >> split), sub = tid & ((1 << split) - 1);
            const bool in = j < m, served = in && j < K;
            const float v = in ? (served ? key[j] : key_old[j]) : 0.0f;
            f32x2 c0 = pack2(0.0f, 0.0f), c1 = c0;
            const int k4 = K >> 2;
#pragma unroll 4
            for (int k = sub; k < k4; k += 1 << split) {
                const float4 x = reinterpret_cast<const float4 *>(key)[k];
                c0 = add2(c0, pack2(md_gt(v, x.x), md_gt(v, x.y)));
                c1 = add2(c1, pack2(md_gt(v, x.z), md_gt(v, x.w)));
            }
            float c = (c0.x + c0.y) + (c1.x + c1.y);
            if (sub == 0) {
                for (int k = 4 * k4; k < K; ++k) c += md_gt(v, key[k]);
            }
            for (int o = 1; o < (1 << split); o <<= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
            if (!in || sub != 0) continue;
            int blk = id[j];
            const unsigned long long v64 = served ? fresh[j] : sum[j];
            if (served) {
                if (given) p.perm[(size_t)(blk & MD_ID_MASK) * b + (blk >> MD_ID_BITS)] = chan[s - w0 + j];
                blk += given;
                if (v64 == INF) { place[j] = -1; atomicAdd(closed, 1); continue; }
            }
            // (untouched entries are in order; equal distances among them share the first one's place)
            int lo = K, hi = served ? m : j;
            if (served || (j > K && !(key_old[j - 1] < v))) {
                while (lo < hi) {
                    const int mid = (lo + hi) >> 1;
                    if (key_old[mid] < v) lo = mid + 1; else hi = mid;
                }
            } else {
                lo = j;
            }
            const int pos = (int)c + lo - K;
            sum_next[pos] = v64;
            id_next[pos] = blk;
            place[j] = pos;
        }
        __syncthreads();
        // ---- entries that took one place are put in their order by (sum, block), one warp to an entry
        int clash = 0;
        for (int j = tid; j < m; j += nthr) {
            const int pj = place[j];
            if (pj >= 0 && ((id_next[pj] ^ id[j]) & MD_ID_MASK) != 0) { crowded[pj] = 1; clash = 1; }
        }
        if (__syncthreads_or(clash)) {
            for (int j = tid; j < m; j += nthr)
                if (place[j] >= 0 && crowded[place[j]]) doubtful[atomicAdd(&red_open[2], 1)] = (unsigned short)j;
            __syncthreads();
            const int nd = red_open[2];
            for (int e = warp; e < nd; e += nthr >> 5) {
                const int j = doubtful[e], pj = place[j], blk = id[j];
                const unsigned long long v64 = j < K ? fresh[j] : sum[j];
                int before = 0;
                for (int k = lane; k < m; k += 32)
                    before += (place[k] == pj && md_less(k < K ? fresh[k] : sum[k], id[k], v64, blk)) ? 1 : 0;
                before = __reduce_add_sync(0xffffffffu, before);
                if (lane == 0) { sum_next[pj + before] = v64; id_next[pj + before] = blk + (j < K ? given : 0); }
            }
            __syncthreads();
            for (int e = tid; e < nd; e += nthr) crowded[place[doubtful[e]]] = 0;
            if (tid == 0) red_open[2] = 0;
        }
        if (tid == 0) *closed_next = 0;
        __syncthreads();
        m -= *closed;
        s += steps;
        ++batch;
        swap_lists();
    }
    // ---- zero masses change no sum: the blocks of the list take what they have room for, one after the other (so does
    // the last open block)
    if (s < d) {
        for (int r = s + tid; r < d; r += nthr) {
            const int c = min(max(p.order[r], 0), d - 1);
            int left = r - s, j = 0;
            while (j < m && left >= b - (id[j] >> MD_ID_BITS)) { left -= b - (id[j] >> MD_ID_BITS); ++j; }
            if (j < m) p.perm[(size_t)(id[j] & MD_ID_MASK) * b + (id[j] >> MD_ID_BITS) + left] = c;
        }
    }
}

// ---------------------------------------------------------------- up to 256 blocks: a block to a lane
//
// The same batches in fewer dependent steps.  Above, places in the merged list are counted and searched (11000 warp instructions and
// five barriers a batch, 5000 cycles).  Here the list is one 32-bit word a block and is sorted anew after every batch: by warps
// (bitonic), then every word looks for its place in the other warps' runs.  A word is the block below 23 bits of the sum's distance to
// the list's smallest one, in units of a little more than the next mass: a batch ends before its smallest new sum, which is at
// most one mass away, so that sums further away need no order yet.  Sums and fill counts stay in shared memory by block, masses
// and the place of every rank as well; the permutation is stored in the end.  Neighbours that their words do not tell apart are
// looked at when the list is read.  Small batches (steep masses) are followed by runs of 32 channels one by one, as above; these need
// the 32 smallest entries, for which the distances beyond that reach keep their leading bits (3 % of the words: with half of them 17 instead of 8 of
// 75 steps found neighbours to put in order, 120 us instead of 106).  Without them a run ended with its first block wherever fewer than
// 32 entries were within reach: 256 blocks of 16, lognormal(0, 2) masses 246 -> 172 us, u^-3 681 -> 519.
// 8192 channels of a real statistic in 256 blocks: 106 us (175 as above), 2800 cycles a batch (the sort in the warps 560, the places 750).
// What it did not gain: all of it in one warp, eight words a lane and no barrier (151 us: one warp's issue), the places by fours
// with 16-byte loads (116).  Other masses (heavy-tailed, steep, equal, subnormal, too small to change a sum; 20 to 256 blocks of 8 to 128
// channels): 0.1 to 0.94 of the time above.
constexpr int MD_SORT_BLOCKS = 256;
constexpr int MD_SORT_SLOTS = 512;                       // (entries of the tables by block: a word without a block has the last one)
constexpr int MD_SORT_THREADS = 512;
constexpr uint32_t MD_ID = MD_SORT_SLOTS - 1;            // block in the low 9 bits
constexpr uint32_t MD_FAR = 0x7c0000u << 9;              // far: in order by ten bits of the distance's mantissa
constexpr uint32_t MD_NONE = 0xffffffffu;                // full block, or none

struct MdSortSmem {
    size_t sum, lows, fill, list, runs, red, place, mass, total;
    __host__ __device__ explicit MdSortSmem(int d)
    {
        size_t o = 0;
        sum = o;   o += (size_t)MD_SORT_SLOTS * 8;
        lows = o;  o += 16 * 8;
        fill = o;  o += (size_t)MD_SORT_SLOTS * 4;
        list = o;  o += (size_t)MD_SORT_BLOCKS * 4;
        runs = o;  o += (size_t)MD_SORT_BLOCKS * 4;
        red = o;   o += 32 * 4;
        place = o; o += ((size_t)d * 2 + 15) & ~(size_t)15;
        mass = o;  o += (size_t)d * 4;
        total = o;
    }
};

// A barrier of the warps that sort, with a count or a disjunction over their threads.
__device__ __forceinline__ int md_barrier_count(int threads, bool v)
{
    uint32_t c;
    asm volatile("{ .reg .pred p; setp.ne.u32 p, %1, 0; bar.red.popc.u32 %0, 1, %2, p; }" : "=r"(c) : "r"((uint32_t)v), "r"(threads) : "memory");
    return (int)c;
}
__device__ __forceinline__ bool md_barrier_any(int threads, bool v)
{
    uint32_t any;
    asm volatile("{ .reg .pred p, q; setp.ne.u32 p, %1, 0; bar.red.or.pred q, 1, %2, p; selp.u32 %0, 1, 0, q; }"
                 : "=r"(any) : "r"((uint32_t)v), "r"(threads) : "memory");
    return any != 0u;
}

// Up to `room` channels from rank s on, one by one (a warp): lane j has entry j of the list.  Returns how many (a mass of zero ends it).
// 32 channels reach no more than the 32 smallest entries.  These are the first ones of the list where all of them are near, where the next one's
// word tells it apart from them, or where there is none.  Elsewhere only near entries are looked at, and the first one must not become
// full before the last channel: until then no block that is served is further from where the first one was than the masses served,
// so that all of them are near if the list reaches 32 masses beyond its first entry.
__device__ __noinline__ int md_warp_serial(uint32_t *list, unsigned long long *sum, int *fill, uint16_t *place, const float *mass, int s, int room, int b,
                                           uint32_t beyond, int lane)
{
    const uint32_t own = list[lane], last = __shfl_sync(0xffffffffu, own, 31);
    const bool known = last < MD_FAR || last == MD_NONE || (last >> 9) < (beyond >> 9);
    const bool has = own != MD_NONE && (known || lane == 0 || own < MD_FAR);      // (the first entry is near)
    const int mine = has ? (int)(own & MD_ID) : MD_ID_MASK;
    unsigned long long w = has ? sum[mine] : ~0ull;
    int f = has ? fill[mine] : 0, t = 0;
    const int first_room = b - __shfl_sync(0xffffffffu, f, 0);
    if (!known) room = min(room, first_room);
#pragma unroll 1
    for (; t < room; ++t) {
        const float a = mass[s + t];
        if (a == 0.0f) break;
        unsigned long long lowest;
        int blk;
        md_warp_min(w, mine, lowest, blk);
        if (w == lowest && mine == blk) {
            place[s + t] = (uint16_t)(blk * b + f);
            w = (unsigned long long)__double_as_longlong(__longlong_as_double((long long)w) + (double)a);
            if (++f == b) w = ~0ull;
        }
    }
    if (has) {
        fill[mine] = f;
        if (w != ~0ull) sum[mine] = w; else list[lane] = MD_NONE;
    }
    __syncwarp();
    return t;
}

// W warps sort (32 W blocks at most).
template <int W>
__global__ void __launch_bounds__(MD_SORT_THREADS, 1) perq_massdiff_sort_kernel(MassdiffParams p)
{
    extern __shared__ __align__(16) unsigned char md_smem[];
    const int d = p.d, b = p.b, n = d / b;
    constexpr int SERIAL_BELOW = W <= 4 ? 4 : 6;              // (about the channels one by one that a batch costs)
    const MdSortSmem lay(d);
    double *sum = (double *)(md_smem + lay.sum);
    unsigned long long *sum_bits = (unsigned long long *)sum, *lows = (unsigned long long *)(md_smem + lay.lows);
    int *fill = (int *)(md_smem + lay.fill);
    uint32_t *list = (uint32_t *)(md_smem + lay.list), *runs = (uint32_t *)(md_smem + lay.runs), *red = (uint32_t *)(md_smem + lay.red);
    int *full = (int *)(red + 16);                           // [3] blocks that became full; three steps in turn, so that one can be cleared
    int *served_one = full + 3, *left = full + 4;            // channels of a run one by one; rank and open blocks in the end
    uint16_t *place = (uint16_t *)(md_smem + lay.place);
    float *mass = (float *)(md_smem + lay.mass);
    int tid;
    asm volatile("mov.u32 %0, %%tid.x;" : "=r"(tid));
    const int lane = tid & 31, warp = tid >> 5;

    for (int j = tid; j < MD_SORT_SLOTS; j += MD_SORT_THREADS) {
        sum[j] = 0.0;
        fill[j] = 0;
        if (j < MD_SORT_BLOCKS) list[j] = j < n ? (uint32_t)j : MD_NONE;
    }
    if (tid < 32) red[tid] = 0u;
    griddep_wait();             // nothing above reads or writes global memory
    griddep_launch();
#pragma unroll 4
    for (int r = tid; r < d; r += MD_SORT_THREADS) mass[r] = md_mass(p.a[min(max(p.order[r], 0), d - 1)]);
    __syncthreads();
    if (tid < 32 * W) {
        int m = n, s = 0, serial = 0, length = 1;            // open blocks; next rank; runs one by one to come, after the next small batch
        int now = 0;                                         // step modulo 3
#pragma unroll 1
        while (s < d) {
            const float unit = mass[s];
            if (m == 1 || unit == 0.0f) break;               // one block or only zero masses are left: below
            const int next = now < 2 ? now + 1 : 0;
            // ---- sums, and those that the next channels would reach in the order of the list
            uint32_t k = list[tid];
            const double base = sum[list[0] & MD_ID];        // (the smallest)
            double v = sum[k & MD_ID];
            const uint32_t k1 = tid + 1 < 32 * W ? list[tid + 1] : MD_NONE;
            const double v1 = sum[k1 & MD_ID], w = v + (double)mass[min(s + tid, d - 1)];
            const int blk = (int)(k & MD_ID), f = fill[blk];
            const float at = (float)(v - base), to = (float)(w - base);
            const float step = unit + (float)(base * 1.2e-16);               // what a channel adds at most: the sum is rounded
            const bool near = k < MD_FAR;
            // (sums further away can not be the smallest)
            const uint32_t low = __reduce_min_sync(0xffffffffu, near && f + 1 < b ? __float_as_uint(to) : 0x7f800000u);
            if (lane == 0) red[warp] = low;
            const bool wrong = k1 < MD_FAR && (v1 < v || (v1 == v && (int)(k1 & MD_ID) < blk));
            if (md_barrier_any(32 * W, wrong)) {
                // neighbours change places until all near entries are in order (an even round settles the even pairs)
#pragma unroll 1
                for (int r = 0; r < 64 * W + 2; ++r) {
                    bool swapped = false;
                    if (((tid ^ r) & 1) == 0 && tid + 1 < 32 * W) {
                        const uint32_t e0 = list[tid], e1 = list[tid + 1];
                        const int b0 = (int)(e0 & MD_ID), b1 = (int)(e1 & MD_ID);
                        if (e1 < MD_FAR && md_less(sum_bits[b1], b1, sum_bits[b0], b0)) { list[tid] = e1; list[tid + 1] = e0; swapped = true; }
                    }
                    if (!md_barrier_any(32 * W, swapped) && (r & 1)) break;
                }
                continue;
            }
            double from = base;
            float reach, lift, scale;
            auto reach_to = [&](float r) {
                lift = r < 0x1p-60f ? 0x1p64f : 1.0f;        // (the reach has an inverse in fp32)
                reach = fminf(r * lift, 3.4e38f);
                scale = __fdividef(8126400.0f / 256.0f, reach * 0.00390625f);
            };
            int K;
            bool anew;                                       // the new smallest sum may be anywhere: to be looked for
            if (n <= MD_FEW_BLOCKS || serial > 0) {
                if (warp == 0) {
                    const int t = md_warp_serial(list, sum_bits, fill, place, mass, s, n <= MD_FEW_BLOCKS ? d - s : min(32, d - s), b, W > 1 ? list[32] : MD_NONE, lane);
                    if (lane == 0) *served_one = t;
                }
                named_barrier(1, 32 * W);
                if (serial > 0) --serial;
                const uint32_t before = k;
                k = list[tid];
                v = sum[k & MD_ID];
                if (k == MD_NONE && before != MD_NONE) atomicAdd(&full[now], 1);
                K = *served_one;
                // (while the first block is open, the smallest sum is at most 32 masses above the old one, from which distances count)
                anew = list[0] == MD_NONE;
                reach_to((serial > 0 && !anew ? 67.0f : 34.0f) * step);
            } else {
                // ---- serve the entries below the smallest of them (the first one always)
                uint32_t least_bits = red[0];
#pragma unroll
                for (int j = 1; j < W; ++j) least_bits = min(least_bits, red[j]);
                const float least = __uint_as_float(least_bits);
                const bool served = tid == 0 || (near && at < least);
                if (served) {
                    place[s + tid] = (uint16_t)(blk * b + f);
                    fill[blk] = f + 1;
                    sum[blk] = w;
                    v = w;
                    if (f + 1 == b) { k = MD_NONE; atomicAdd(&full[now], 1); }
                }
                // (at most two masses away where the first block stays open)
                anew = !(least < 3.0e38f && least <= 2.0f * unit);
                if (!anew) from = base + (double)(least * 0.9999998f);
                // (whether runs one by one follow, and need a longer reach, is known when the served entries are counted; the reach of the
                // largest masses would leave fp32)
                reach_to(1.05f * unit);
                K = md_barrier_count(32 * W, served);
                if (K < SERIAL_BELOW && K < m && unit < 1.0e36f) { serial = length; length = min(2 * length, MD_SERIAL_RUNS); reach_to(34.0f * step); }
                else if (K < m) length = 1;
            }
            if (anew) {
                // ---- the first block is full, and the next one may be anywhere: distances count from the smallest sum there is.  (From the old
                // one, entries that a run one by one needs would lie beyond its reach.)
                unsigned long long lowest;
                int unused;
                md_warp_min(k != MD_NONE ? (unsigned long long)__double_as_longlong(v) : ~0ull, blk, lowest, unused);
                if (lane == 0) lows[warp] = lowest;
                named_barrier(1, 32 * W);
                lowest = lows[0];
#pragma unroll
                for (int j = 1; j < W; ++j) lowest = min(lowest, lows[j]);
                from = __longlong_as_double((long long)lowest);
            }
            // ---- words of the new list, sorted by warps
            const float away = fmaxf((float)(v - from), 0.0f) * lift, q = fminf(away * scale, 8126463.0f);
            const uint32_t beyond = MD_FAR + ((__float_as_uint(away) - __float_as_uint(reach)) >> 13 << 9);
            k = k == MD_NONE ? MD_NONE : (away < reach ? __float_as_uint(q + 8388608.0f) << 9 : beyond) | (k & MD_ID);
#pragma unroll
            for (int size = 2; size <= 32; size *= 2) {
#pragma unroll
                for (int stride = size / 2; stride > 0; stride /= 2) {
                    // (the first step of a size compares mirrored lanes, so that all are ascending)
                    const uint32_t o = __shfl_xor_sync(0xffffffffu, k, stride == size / 2 ? size - 1 : stride);
                    k = (lane & stride) == 0 ? min(k, o) : max(k, o);
                }
            }
            int at_place = lane;
            if (W > 1) {
                runs[tid] = k;
                named_barrier(1, 32 * W);
                // ---- places: words before the own one in the other warps' runs
#pragma unroll
                for (int j = 1; j < W; ++j) {
                    const uint32_t *run = runs + ((warp + j) % W) * 32;
                    int c = 0;
#pragma unroll
                    for (int step = 16; step > 0; step /= 2) c += run[c + step - 1] < k ? step : 0;
                    at_place += c + (run[c] < k ? 1 : 0);
                }
            } else {
                __syncwarp();
            }
            m -= full[now];
            if (tid == 0) full[next] = 0;
            if (k != MD_NONE) list[at_place] = k;
            if (tid >= m) list[tid] = MD_NONE;
            s += K;
            now = next;
            named_barrier(1, 32 * W);
        }
        if (tid == 0) { left[0] = s; left[1] = m; }
    }
    __syncthreads();
    const int s = left[0], m = left[1];
    if (s < d) {
        // ---- zero masses change no sum: the open blocks take what they have room for, in the order of their sums (so does the last
        // open block).  Their order by counting.
        const uint32_t mine = tid < m ? list[tid] & MD_ID : 0u;
        int before = 0;
        if (tid < m)
#pragma unroll 1
            for (int j = 0; j < m; ++j) {
                const uint32_t o = list[j] & MD_ID;
                before += md_less(sum_bits[o], (int)o, sum_bits[mine], (int)mine) ? 1 : 0;
            }
        if (tid < m) runs[before] = mine;
        __syncthreads();
#pragma unroll 1
        for (int r = s + tid; r < d; r += MD_SORT_THREADS) {
            int rest = r - s, j = 0;
            while (j < m && rest >= b - fill[runs[j]]) { rest -= b - fill[runs[j]]; ++j; }
            if (j < m) place[r] = (uint16_t)((int)runs[j] * b + fill[runs[j]] + rest);
        }
        __syncthreads();
    }
#pragma unroll 4
    for (int r = tid; r < d; r += MD_SORT_THREADS) p.perm[place[r]] = min(max(p.order[r], 0), d - 1);
}

}  // namespace perq
