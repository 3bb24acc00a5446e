// Index work shared by the pack and the two unpack directions: where a routed copy or a received row goes.
//
// All three are the same problem.  A plan gives, step by step, runs of rows for one bucket (a destination or a sender
// rank); items (routed copies, received rows) fall into buckets or keys by a stable counting sort; the position of an item
// among the items of its bucket, looked up in that bucket's runs, is the row it goes to or comes from.
//
// Two forms of each call are built from the functions here:
//  * small problems (kSmallItems items at most): ONE launch in which every CTA builds the run table and counts the items
//    before its own by itself, then moves its own rows.  Nothing is shared between CTAs, so nothing has to be zeroed,
//    published or waited for.
//  * larger ones: a count kernel (one histogram per chunk of items), a map kernel (a chunk's base is the sum of the
//    histograms before it) and the row copy, chained by programmatic dependent launch: a kernel's CTAs are resident
//    before the one ahead has finished and wait for its results in griddepcontrol.wait.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "chunks.h"
#include "vp_internal.h"

namespace {

constexpr int kIdxWarps = kIdxThreads / 32;
constexpr int kMaxKeys = 1024;                      // experts_per_rank x N
// Items up to which one self-contained launch is used.  Its last CTA counts every item itself, and the rows move by plain loads
// and stores (10 % behind the bulk copy).  Pack of 16 ranks, top-8, one launch | chunked, us: rows of 256 B 6,144 copies 15.4 | 17.4,
// 8,192 17.4 | 17.4, 16,384 21.5 | 19.4; rows of 14,336 B 6,144 copies 28.7 | 33.8, 8,192 33.9 | 35.9, 12,288 48.1 | 46.1.
constexpr int kSmallItems = 8192;
constexpr int kSmallSteps = 1024;                   // plan arrays longer than this do not fit its run table
constexpr int kSmallOwn = 1024;                     // rows or copies one CTA may own there
constexpr int64_t kSmallRow = (int64_t)1 << 30;     // bytes per row: up to here 32 bits number the vectors of a row

// Division by the row size without a divide sequence: plan offsets are below 2^52, so the product with the rounded
// reciprocal is off by one at most.
struct RowDiv {
    int64_t d;
    double inv;
    __device__ __forceinline__ int64_t div(int64_t x, int64_t& rem) const {
        int64_t q = __double2ll_rz((double)x * inv), r = x - q * d;
        if (r < 0) { q--; r += d; }
        else if (r >= d) { q++; r -= d; }
        rem = r;
        return q;
    }
};
inline RowDiv row_div(int64_t d) { return RowDiv{d, 1.0 / (double)d}; }
// Division by the experts per rank: unsigned division by an invariant integer after Granlund and Montgomery ("Division by Invariant
// Integers using Multiplication", PLDI 1994, Section 4).  With l = ceil(log2 d) and m = floor(2^32 (2^l - d) / d) + 1 the quotient is
// (mulhi(m, x) + x) >> l; the sum needs 33 bits in general, 32 for the expert ids here, which are below 2^31.
struct SmallDiv {
    uint32_t m;
    int shift;
    __device__ __forceinline__ int div(int x) const { return (int)((__umulhi(m, (uint32_t)x) + (uint32_t)x) >> shift); }
};
inline SmallDiv small_div(int d) {
    int l = 0;
    while (((int64_t)1 << l) < d) l++;
    return SmallDiv{(uint32_t)((((uint64_t)1 << 32) * (((uint64_t)1 << l) - (uint64_t)d)) / (uint64_t)d + 1), l};
}

// SMs of the current device, asked once per device.
inline int sm_count_of_device() {
    static int s_sms[64] = {0};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 0;
    const bool cached = dev >= 0 && dev < 64;
    int sms = cached ? __atomic_load_n(&s_sms[dev], __ATOMIC_RELAXED) : 0;
    if (!sms) {
        if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
        if (cached) __atomic_store_n(&s_sms[dev], sms, __ATOMIC_RELAXED);
    }
    return sms;
}

// Launch that may start while the kernel ahead of it in the stream drains (its griddepcontrol.wait holds it back).
template <typename... P, typename... A>
inline cudaError_t launch_after(void (*fn)(P...), int grid, int threads, size_t smem, cudaStream_t stream, A... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    g_vp_launches++;
    return cudaLaunchKernelEx(&cfg, fn, P(args)...);
}

// The same for kernels whose shared memory may exceed the default limit of 48 KB.  The limit is raised to one constant,
// never to the launch's own size: it belongs to the function, and another thread may be about to launch with more.
constexpr size_t kSmemLimit = 220 * 1024;
template <typename... P, typename... A>
inline cudaError_t launch_wide(void (*fn)(P...), int grid, size_t smem, cudaStream_t stream, A... args) {
    if (smem > 48 * 1024) {
        const cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemLimit);
        if (e != cudaSuccess) return e;
    }
    return launch_after(fn, grid, kIdxThreads, smem, stream, args...);
}

// First statement of every kernel launched that way: nothing of an earlier kernel is read or overwritten before it, and the
// kernel behind may start launching.
__device__ __forceinline__ void grid_wait() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;");
}

// The runs of one rank, grouped by bucket: run s of bucket j (ptr[j] <= s < ptr[j + 1]) starts at position start[s] of the
// bucket's stream and at row row[s]; total[j] rows in all.
struct Runs {
    int *start, *row, *ptr, *total;
};

// Exclusive scan of v over the CTA (kIdxThreads threads); sum receives the total.  wsum: kIdxWarps + 1 ints of shared memory.
__device__ __forceinline__ int cta_exclusive_scan(int v, int* wsum, int& sum) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
    }
    if (lane == 31) wsum[warp] = incl;
    __syncthreads();
    int before = 0, all = 0;
#pragma unroll
    for (int w = 0; w < kIdxWarps; w++) {
        const int x = wsum[w];
        before += w < warp ? x : 0;
        all += x;
    }
    __syncthreads();
    sum = all;
    return before + incl - v;
}

// Scratch of build_runs: counts and rows per (warp, bucket).
__host__ __device__ inline int runs_scratch_ints(int N) { return 2 * kIdxWarps * N + kIdxWarps + 1; }

// One step of the plan as the rank sees it: bucket (-1: none), rows, first row.
struct Step { int j, rows, row0; };

// Builds the run table from the steps step(k), k < K.  `first` is step(threadIdx.x), which the caller fetches before it knows K
// (the plan arrays have k_max rows, and a trip to L2 is saved); what lies beyond K is ignored here.  out.* may be shared or global memory (each element is written once, by one thread); cnt is [N] ints of shared memory.
template <typename StepFn>
__device__ __forceinline__ void build_runs(int K, int N, Step first, StepFn step, Runs out, int* cnt, int* scratch) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    int* wcnt = scratch;
    int* wrow = scratch + kIdxWarps * N;
    int* wsum = scratch + 2 * kIdxWarps * N;
    for (int j = tid; j < N; j += kIdxThreads) cnt[j] = 0;
    for (int e = tid; e < 2 * kIdxWarps * N; e += kIdxThreads) scratch[e] = 0;
    __syncthreads();
    if (tid >= K) first.j = -1;
    if (first.j >= 0) atomicAdd(&cnt[first.j], 1);
    for (int k = tid + kIdxThreads; k < K; k += kIdxThreads) {
        const int j = step(k).j;
        if (j >= 0) atomicAdd(&cnt[j], 1);
    }
    __syncthreads();
    int all;
    const int mine = tid < N ? cnt[tid] : 0;                       // (N <= 256 <= kIdxThreads)
    const int ptr = cta_exclusive_scan(mine, wsum, all);
    if (tid < N) { out.ptr[tid] = ptr; cnt[tid] = ptr; }       // from here on: next free run of every bucket
    if (tid == 0) out.ptr[N] = all;
    __syncthreads();
    int run_rows = 0;                                              // rows of bucket tid in the tiles before
    for (int k0 = 0; k0 < K; k0 += kIdxThreads) {
        Step s = first;
        if (k0) s = k0 + tid < K ? step(k0 + tid) : Step{-1, 0, 0};
        const int j = s.j, rows = s.rows;
        // inside the warp: runs and rows of the same bucket in lower lanes
        const unsigned peers = __match_any_sync(0xffffffffu, j >= 0 ? j : -1 - lane);
        const unsigned lower = peers & ((1u << lane) - 1);
        int pre = 0;
        for (unsigned m = lower; __any_sync(0xffffffffu, m != 0); ) {
            const int v = __shfl_sync(0xffffffffu, rows, m ? __ffs(m) - 1 : 0);
            if (m) { pre += v; m &= m - 1; }
        }
        if (j >= 0 && (peers >> lane) == 1u) { wcnt[warp * N + j] = __popc(peers); wrow[warp * N + j] = pre + rows; }   // highest lane
        __syncthreads();
        // bucket tid: exclusive prefix over the warps, carried on from the tiles before
        if (tid < N) {
            int c = cnt[tid], r = run_rows;
#pragma unroll 4
            for (int w = 0; w < kIdxWarps; w++) {
                const int cw = wcnt[w * N + tid], rw = wrow[w * N + tid];
                wcnt[w * N + tid] = c; wrow[w * N + tid] = r;
                c += cw; r += rw;
            }
            cnt[tid] = c; run_rows = r;
        }
        __syncthreads();
        if (j >= 0) {
            const int at = wcnt[warp * N + j] + __popc(lower);
            out.start[at] = wrow[warp * N + j] + pre;
            out.row[at] = s.row0;
        }
        if (k0 + kIdxThreads < K) {
            __syncthreads();
            for (int e = tid; e < 2 * kIdxWarps * N; e += kIdxThreads) scratch[e] = 0;
            __syncthreads();
        }
    }
    if (tid < N) out.total[tid] = run_rows;
    __syncthreads();
}

// The run table of n buckets copied to shared memory (2 n_runs + 2 n + 1 words at `to`) if its runs fit `most`; all threads, no
// barrier.  A look-up is half a dozen dependent reads: 30 cycles each there, ten times that in L2.
__device__ __forceinline__ Runs runs_to_shared(const Runs& t, int n, int most, int* to) {
    const int n_runs = t.ptr[n];
    if (n_runs > most) return t;
    const Runs s{to + 2 * n + 1, to + 2 * n + 1 + n_runs, to, to + n + 1};
    for (int i = threadIdx.x; i < n_runs; i += kIdxThreads) { s.start[i] = t.start[i]; s.row[i] = t.row[i]; }
    for (int i = threadIdx.x; i <= n; i += kIdxThreads) s.ptr[i] = t.ptr[i];
    for (int i = threadIdx.x; i < n; i += kIdxThreads) s.total[i] = t.total[i];
    return s;
}

// Row of position p in bucket j's stream, -1 beyond the plan.
__device__ __forceinline__ int run_lookup(const Runs& t, int j, int p) {
    if (p >= t.total[j]) return -1;
    int lo = t.ptr[j], hi = t.ptr[j + 1] - 1;
    while (lo < hi) {                                              // last run starting at or before p
        const int mid = (lo + hi + 1) >> 1;
        if (t.start[mid] <= p) lo = mid; else hi = mid - 1;
    }
    return t.row[lo] + (p - t.start[lo]);
}

// peer[k] = the (highest) source rank whose lane of step k goes to `rank`, -1 if none, for the steps k0 <= k < k1.
// peer is shared memory; all threads of the CTA.
__device__ __forceinline__ void find_senders(const int16_t* __restrict__ lane_dst, int N, int rank, int k0, int k1, int* peer) {
    for (int k = k0 + threadIdx.x; k < k1; k += kIdxThreads) peer[k - k0] = -1;
    __syncthreads();
    const int16_t* base = lane_dst + (size_t)k0 * N;
    const long long cells = (long long)(k1 - k0) * N;
    if (N % 8 == 0 && ((uintptr_t)base & 15) == 0) {
#pragma unroll 4
        for (long long v = threadIdx.x; v < cells / 8; v += kIdxThreads) {
            const uint4 x = __ldg((const uint4*)base + v);
            const uint32_t w[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
            for (int q = 0; q < 8; q++)
                if ((int)((w[q >> 1] >> (16 * (q & 1))) & 0xffffu) == rank) {
                    const long long e = v * 8 + q;
                    atomicMax(&peer[e / N], (int)(e % N));
                }
        }
    } else {
        for (long long e = threadIdx.x; e < cells; e += kIdxThreads)
            if (base[e] == rank) atomicMax(&peer[e / N], (int)(e % N));
    }
    __syncthreads();
}

// Calls f(x[i]) for lo <= i < hi over the CTA, sixteen loads of four values in flight per thread where x is 16-byte aligned.
template <typename F>
__device__ __forceinline__ void for_each_item(const int32_t* __restrict__ x, int lo, int hi, F f) {
    const bool vec = ((uintptr_t)x & 15) == 0;
    const int v0 = vec ? (lo + 3) & ~3 : hi, v1 = vec ? hi & ~3 : hi;
    if (hi - lo >= 4 * kIdxThreads && v0 < v1) {     // (fewer: one value per thread spreads the work better)
#pragma unroll 4
        for (int v = v0 / 4 + threadIdx.x; v < v1 / 4; v += kIdxThreads) {
            const int4 q = __ldg((const int4*)x + v);
            f(4 * v, q.x); f(4 * v + 1, q.y); f(4 * v + 2, q.z); f(4 * v + 3, q.w);
        }
        if ((int)threadIdx.x < v0 - lo) f(lo + threadIdx.x, x[lo + threadIdx.x]);
        if ((int)threadIdx.x < hi - v1) f(v1 + threadIdx.x, x[v1 + threadIdx.x]);
    } else {
#pragma unroll 4
        for (int i = lo + threadIdx.x; i < hi; i += kIdxThreads) f(i, x[i]);
    }
}

// Stable positions of the items lo <= i < hi, taken 32 at a time by ONE warp: key(i) names an item's key (-1: none),
// next[] holds the position of the next item of every key and is carried on; put(i, key, position) is called for every
// item, with position -1 where there is no key.
template <typename Key, typename Put>
__device__ __forceinline__ void warp_positions(long long lo, long long hi, int* next, Key key, Put put) {
    const int lane = threadIdx.x & 31;
    for (long long i0 = lo; i0 < hi; i0 += 32) {
        const long long i = i0 + lane;
        const int k = i < hi ? key(i) : -1;
        const unsigned peers = __match_any_sync(0xffffffffu, k >= 0 ? k : -1 - lane);
        const unsigned lower = peers & ((1u << lane) - 1);
        const int p = k >= 0 ? next[k] + __popc(lower) : -1;
        __syncwarp();
        if (k >= 0 && lower == 0) next[k] += __popc(peers);
        __syncwarp();
        if (i < hi) put(i, k, p);
    }
}

// ---- moving the rows a CTA owns (the one-launch form) ------------------------------------------------------------

template <typename V> struct PieceOf { static constexpr int U = sizeof(V) == 16 ? 4 : 8; };   // vectors in flight per lane

// Own rows i < n: source row src[i] (-1: skip), destination rows dst[i * fanout + f] (-1: none).  Vectors v_lo <= v < v_hi
// of every row; a warp takes 32 U of them at a time, all loads in flight before the first store.
template <typename V>
__device__ __forceinline__ void move_rows(const char* __restrict__ rows, char* __restrict__ out, long long row_bytes, int n, int fanout,
                                          const int* src, const int* dst, int v_lo, int v_hi) {
    constexpr int U = PieceOf<V>::U;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int pieces = (v_hi - v_lo + 32 * U - 1) / (32 * U);
    for (int it = warp; it < n * pieces; it += kIdxWarps) {
        const int i = it / pieces, v0 = v_lo + (it - i * pieces) * 32 * U + lane;
        const int s = src[i];
        if (s < 0) continue;
        const V* from = (const V*)(rows + (long long)s * row_bytes);
        V x[U];
#pragma unroll
        for (int u = 0; u < U; u++)
            if (v0 + 32 * u < v_hi) x[u] = __ldg(from + v0 + 32 * u);
        for (int f = 0; f < fanout; f++) {
            const int d = dst[i * fanout + f];
            if (d < 0) continue;
            V* to = (V*)(out + (long long)d * row_bytes);
#pragma unroll
            for (int u = 0; u < U; u++)
                if (v0 + 32 * u < v_hi) to[v0 + 32 * u] = x[u];
        }
    }
}

// How a small problem of `n` source rows is dealt: `pieces` CTAs per row while there are fewer rows than SMs, then up to two
// CTAs per SM with contiguous row ranges.
struct SmallSplit { int grid, pieces; };
inline SmallSplit small_split(int n, int sms) {
    SmallSplit s;
    s.pieces = n >= sms ? 1 : (2 * sms / n < 8 ? 2 * sms / n : 8);
    s.grid = n >= sms ? (n < 2 * sms ? n : 2 * sms) : n * s.pieces;
    return s;
}

}  // namespace
