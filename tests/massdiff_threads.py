"""The device MassDiff up to 256 blocks on the CPU: its kernel's source, compiled with every thread as a coroutine.

Threads run one after the other up to the next warp operation or barrier.  A policy says which of the warps that can run goes next, so
that a warp can be far ahead of the others wherever no barrier holds it.  Warps that meet at different barriers (which would
wait for each other on a GPU) end the run with a status."""
import ctypes
import functools
import os
import re
import subprocess
import tempfile

import numpy as np

SOURCE = os.path.join(os.path.dirname(os.path.abspath(__file__)), "..", "paper_2601_22347_b200", "csrc", "perq_massdiff.cuh")
FIRST, LAST, RANDOM = 0, 1, 2           # the warp that goes next: the lowest, the highest, any (from RANDOM on: seeds)

HARNESS = r"""
#include <algorithm>
#include <csetjmp>
#include <cstdint>
#include <cstdlib>
#include <cstring>
#include <cmath>
#include <ucontext.h>
#include <vector>
using std::min; using std::max;
#define __device__
#define __host__
#define __global__
#define __forceinline__ inline
#define __noinline__
#define __launch_bounds__(...)
struct float2 { float x, y; };
static const int THREADS = 512, STACK = 32768;
struct Thread { jmp_buf at; ucontext_t start; bool started, done; int on_bar; unsigned bar_gen; };   // on_bar: the barrier it waits for, or -1
struct Warp { unsigned gen, arrived, done; int op; uint64_t v[32], out; bool flag; };
struct Barrier { unsigned gen; int count, kind; uint32_t acc; uint32_t out; };
static Thread T[THREADS]; static Warp W_[16]; static Barrier B_[2];
static unsigned char *stacks; static jmp_buf scheduler; static int cur, status;
static unsigned char *md_smem_base;
static void (*entry)();
static void yield() { if (_setjmp(T[cur].at) == 0) _longjmp(scheduler, 1); }
static void fail(int s) { if (!status) status = s; _longjmp(scheduler, 2); }
// all lanes of the warp: their values, of which `reduce` makes one (the last lane to come does)
template <typename F> static uint64_t meet(int op, uint64_t v, F reduce)
{
    Warp &w = W_[cur >> 5];
    if (w.arrived == 0) w.op = op;
    else if (w.op != op) fail(2);
    w.v[cur & 31] = v;
    if (++w.arrived == 32) { w.arrived = 0; w.out = reduce(w.v); ++w.gen; return w.out; }
    const unsigned g = w.gen;
    while (w.gen == g) yield();
    return w.out;
}
static uint32_t barrier(int id, int threads, int line, uint32_t v)
{
    Barrier &b = B_[id];
    if (b.count == 0) { b.kind = line * 4096 + threads; b.acc = 0; }
    else if (b.kind != line * 4096 + threads) fail(3);
    b.acc += v;
    if (++b.count == threads) { b.count = 0; b.out = b.acc; ++b.gen; }
    else { T[cur].on_bar = id; T[cur].bar_gen = b.gen; const unsigned g = b.gen; while (b.gen == g) yield(); T[cur].on_bar = -1; }
    return b.out;
}
#define __syncthreads() barrier(0, THREADS, __LINE__, 0)
#define named_barrier(id, threads) barrier(id, threads, __LINE__, 0)
#define md_barrier_count(threads, v) ((int)barrier(1, threads, __LINE__, v))
#define md_barrier_any(threads, v) (barrier(1, threads, __LINE__, v) != 0)
static uint32_t f2u(float f) { uint32_t u; memcpy(&u, &f, 4); return u; }
#define __float_as_uint f2u
static float __uint_as_float(uint32_t u) { float f; memcpy(&f, &u, 4); return f; }
static double __longlong_as_double(long long u) { double f; memcpy(&f, &u, 8); return f; }
static long long __double_as_longlong(double f) { long long u; memcpy(&u, &f, 8); return u; }
static float __fdividef(float a, float b) { return a * (1.0f / b); }
static void __syncwarp() { meet(1, 0, [](uint64_t *) { return 0ull; }); }
static uint32_t __reduce_min_sync(unsigned, uint32_t v) { return (uint32_t)meet(2, v, [](uint64_t *a) { return *std::min_element(a, a + 32); }); }
static uint32_t __reduce_max_sync(unsigned, uint32_t v) { return (uint32_t)meet(3, v, [](uint64_t *a) { return *std::max_element(a, a + 32); }); }
static bool __any_sync(unsigned, bool v) { return meet(4, v, [](uint64_t *a) { return *std::max_element(a, a + 32); }) != 0; }
// (a lane reads another's value before any lane can come to the next operation: the copies alternate)
static uint64_t shuffled[2][16][32];
template <typename V> static V __shfl_sync(unsigned, V v, int src)
{
    const int w = cur >> 5, side = (W_[w].gen) & 1;
    shuffled[side][w][cur & 31] = (uint32_t)v;
    meet(5, 0, [](uint64_t *) { return 0ull; });
    return (V)shuffled[side][w][src & 31];
}
template <typename V> static V __shfl_xor_sync(unsigned m, V v, int o) { return __shfl_sync(m, v, (cur & 31) ^ o); }
static int atomicAdd(int *p, int v) { const int o = *p; *p += v; return o; }
static void griddep_wait() {}
static void griddep_launch() {}
namespace perq {
//SOURCE
}
static perq::MassdiffParams params;
template <int N> static void kernel() { perq::perq_massdiff_sort_kernel<N>(params); }
static void run() { entry(); T[cur].done = true; _longjmp(scheduler, 1); }
extern "C" int massdiff(const float *a, int *order, int *perm, int d, int b, int policy)
{
    const int n = d / b;
    params = perq::MassdiffParams{a, order, perm, d, b};
    entry = n <= 32 ? kernel<1> : n <= 64 ? kernel<2> : n <= 128 ? kernel<4> : kernel<8>;
    std::vector<double> smem(perq::MdSortSmem(d).total / 8 + 2, -1.0);
    md_smem_base = (unsigned char *)(((uintptr_t)smem.data() + 15) & ~(uintptr_t)15);
    if (!stacks) stacks = (unsigned char *)malloc((size_t)THREADS * STACK);
    memset(W_, 0, sizeof W_); memset(B_, 0, sizeof B_);
    status = 0;
    for (int i = 0; i < THREADS; ++i) { T[i].started = T[i].done = false; T[i].on_bar = -1; }
    uint64_t rnd = 0x9E3779B97F4A7C15ull * (uint64_t)(policy + 1);
    auto blocked = [](int i) { return T[i].done || (T[i].on_bar >= 0 && B_[T[i].on_bar].gen == T[i].bar_gen); };
    for (;;) {
        int able[16], k = 0, open = 0;
        for (int w = 0; w < 16; ++w) {
            bool can = false;
            for (int l = 0; l < 32; ++l) { const int i = 32 * w + l; can |= !blocked(i); open += !T[i].done; }
            if (can) able[k++] = w;
        }
        if (!open) return 0;
        if (!k) return 4;                                       // they wait for each other
        rnd ^= rnd << 13; rnd ^= rnd >> 7; rnd ^= rnd << 17;
        const int w = able[policy == 0 ? 0 : policy == 1 ? k - 1 : (int)(rnd % (uint64_t)k)];
        // the warp, as far as it comes (RANDOM: now and then as far as its next operation)
        for (int turn = 0;; ++turn) {
            bool any = false;
            for (int l = 0; l < 32; ++l) {
                const int i = 32 * w + l;
                if (blocked(i)) continue;
                any = true;
                cur = i;
                if (_setjmp(scheduler) == 0) {
                    if (T[i].started) _longjmp(T[i].at, 1);
                    T[i].started = true;
                    getcontext(&T[i].start);
                    T[i].start.uc_stack.ss_sp = stacks + (size_t)i * STACK;
                    T[i].start.uc_stack.ss_size = STACK;
                    T[i].start.uc_link = nullptr;
                    makecontext(&T[i].start, run, 0);
                    setcontext(&T[i].start);
                }
                if (status) return status;
            }
            if (!any || (policy >= 2 && (rnd >> (8 + turn % 40) & 15) == 0)) break;
        }
    }
}
"""


def _block(text, head):
    """From `head` to the end of its braces."""
    i = text.index(head)
    depth = 0
    for j in range(text.index("{", i), len(text)):
        depth += {"{": 1, "}": -1}.get(text[j], 0)
        if depth == 0:
            return text[i:j + 1]
    raise ValueError(head)


@functools.lru_cache(None)
def _lib():
    with open(SOURCE) as f:
        text = f.read()
    text = text[text.index("namespace perq {") + len("namespace perq {"):text.rindex("}")]
    for head in ("__global__ void __launch_bounds__(MD_RANK_THREADS) perq_massdiff_rank_kernel",
                 "__global__ void __launch_bounds__(MD_MAX_THREADS, 1) perq_massdiff_greedy_kernel"):
        text = text.replace(_block(text, head), "")
    text = re.sub(r"__device__ __forceinline__ float md_g[te]\(.*\n", "", text)
    for head in ("__device__ __forceinline__ int md_barrier_count(int threads, bool v)",
                 "__device__ __forceinline__ bool md_barrier_any(int threads, bool v)"):
        text = text.replace(_block(text, head), "")
    text = text.replace('asm volatile("mov.u32 %0, %%tid.x;" : "=r"(tid));', "tid = cur;")
    text = text.replace("extern __shared__ __align__(16) unsigned char md_smem[];", "unsigned char *const md_smem = md_smem_base;")
    assert "asm" not in text and "__shared__" not in text
    d = tempfile.mkdtemp()
    src, lib = os.path.join(d, "threads.cpp"), os.path.join(d, "threads.so")
    with open(src, "w") as f:
        f.write(HARNESS.replace("//SOURCE", text))
    subprocess.run(["g++", "-std=c++17", "-O2", "-w", "-U_FORTIFY_SOURCE", "-fno-strict-aliasing", "-ffp-contract=off", "-shared", "-fPIC", "-o", lib, src], check=True)
    return ctypes.CDLL(lib)


def massdiff(a, b, policy=FIRST):
    """(status, perm): 0, or 2: lanes of a warp at different operations, 3: warps at different barriers, 4: all wait."""
    a = np.ascontiguousarray(a, np.float32)
    d = a.size
    clean = np.minimum(np.where(a > 0, a, 0), np.finfo(np.float32).max)
    order = np.argsort(-clean, kind="stable").astype(np.int32)
    perm = np.full(d, -1, np.int32)
    status = _lib().massdiff(a.ctypes.data_as(ctypes.c_void_p), order.ctypes.data_as(ctypes.c_void_p),
                             perm.ctypes.data_as(ctypes.c_void_p), d, b, policy)
    return status, perm


KINDS = ("lognormal2", "lognormal3", "power", "outliers", "graded", "rounded", "largest")


def far_apart(kind, n, b, seed):
    """Masses after which the next block to be served is far from the one that has just become full: heavy tails; graded masses, one to a
    block, above light ones; masses that a running sum rounds up to its last place; the upper end of fp32."""
    d = n * b
    rng = np.random.default_rng(seed)
    if kind.startswith("lognormal"):
        return rng.lognormal(0, int(kind[-1]), d).astype(np.float32)
    if kind == "power":
        a = rng.random(d) ** -3.0
    elif kind == "outliers":
        a = rng.random(d) * np.where(rng.random(d) < 0.01, 1e5, 1.0)
    elif kind == "graded":
        a = 1.0 + 10.0 ** -rng.integers(1, 9) * rng.random(d)
        k = rng.integers(1, n)
        a[:k] = rng.uniform(1, 4 * b, k)
    elif kind == "rounded":
        a = rng.uniform(0.3, 3, d) * 2.0 ** -53
        a[:n] = 1 + rng.integers(0, 60, n) * 2.0 ** -23
    else:
        a = np.full(d, 3e36)
        a[:n] = rng.uniform(0, 3.4e38, n)
    return rng.permutation(a.astype(np.float32))
