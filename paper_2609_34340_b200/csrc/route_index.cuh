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

#include "bulk_copy.cuh"
#include "chunks.h"
#include "vp_internal.h"

namespace {

constexpr int kIdxWarps = kIdxThreads / 32;
constexpr int kMaxKeys = 1024;                      // experts_per_rank x N
// Items up to which one self-contained launch is used: every CTA counts the items before its own, 0.15 to 0.3 us per 1,024 of them,
// which the two launches ahead of a copy that they replace (4 to 6 us) pay for up to here.  One launch | chunked, us, 16 ranks, rows of
// 14,336 B: pack of 8,192 copies 24.1 | 29.8, 12,288 35.6 | 39.4, 16,384 46.9 | 49.0; unpack 19.5 | 25.8, 26.9 | 32.7, 34.5 | 39.7; return
// 43.3 | 47.5, 63.5 | 64.6, 82.5 | 81.2.  Rows of 4,096 B, 16,384 items: 18.6 | 21.8, 17.3 | 20.5, 35.6 | 34.3; of 1,536 B 11.4 | 13.9,
// 11.4 | 14.6, 17.1 | 21.3; of 96 B with 16 and 64 ranks against the chunked form as it was then, 8,704 items: pack 7.9 | 11.3 and 9.7 | 11.8,
// return 8.5 | 16.1 and 10.5 | 18.6; 16,384 items: pack 9.5 | 11.9 and 11.3 | 13.4.  (The return counts twice, for both sides of its own range, over more keys: its line lies lower.)
constexpr int kSmallItems = 16384;
constexpr int kSmallReturn = 12288;
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


__device__ __forceinline__ void clear_runs_scratch(int N, int* scratch) {
    for (int e = threadIdx.x; e < 2 * kIdxWarps * N; e += kIdxThreads) scratch[e] = 0;
}

// One step of the plan as the rank sees it: bucket (-1: none), rows, first row.
struct Step { int j, rows, row0; };

// Inside a warp: the lanes whose step has the same bucket, and the rows of those below.
struct SameBucket { unsigned peers, lower; int pre; };
__device__ __forceinline__ SameBucket same_bucket(int j, int rows) {
    const int lane = threadIdx.x & 31;
    const unsigned peers = __match_any_sync(0xffffffffu, j >= 0 ? j : -1 - lane), lower = peers & ((1u << lane) - 1);
    int pre = 0;
    for (unsigned m = lower; __any_sync(0xffffffffu, m != 0); ) {
        const int v = __shfl_sync(0xffffffffu, rows, m ? __ffs(m) - 1 : 0);
        if (m) { pre += v; m &= m - 1; }
    }
    return SameBucket{peers, lower, pre};
}

// build_runs for K <= kIdxThreads, a step per thread.  Counts and rows per (warp, bucket) are gathered in one pass, over the warps that
// hold steps: 1,500 cycles for 44 steps, 3,600 by the tiles below, in front of everything else a call does.  `cleared`: the scratch
// holds zeros, behind a barrier.
__device__ __forceinline__ void build_runs_at_once(int K, int N, Step s, Runs out, int* cnt, int* scratch, bool cleared) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, warps = (K + 31) / 32;
    int *const wcnt = scratch, *const wrow = scratch + kIdxWarps * N, *const wsum = scratch + 2 * kIdxWarps * N;
    if (!cleared) {
        for (int e = tid; e < warps * N; e += kIdxThreads) wcnt[e] = wrow[e] = 0;
        __syncthreads();
    }
    if (tid >= K) s.j = -1;
    SameBucket b{};
    if (warp < warps) {
        b = same_bucket(s.j, s.rows);
        if (s.j >= 0 && (b.peers >> lane) == 1u) { wcnt[warp * N + s.j] = __popc(b.peers); wrow[warp * N + s.j] = b.pre + s.rows; }   // highest lane
    }
    __syncthreads();
    int c = 0, r = 0;                                              // bucket tid: exclusive prefix over the warps
    if (tid < N)
        for (int w = 0; w < warps; w += 4) {
            int cw[4], rw[4];
#pragma unroll
            for (int u = 0; u < 4; u++) {
                cw[u] = w + u < warps ? wcnt[(w + u) * N + tid] : 0;
                rw[u] = w + u < warps ? wrow[(w + u) * N + tid] : 0;
            }
#pragma unroll
            for (int u = 0; u < 4; u++) {
                if (w + u < warps) { wcnt[(w + u) * N + tid] = c; wrow[(w + u) * N + tid] = r; }
                c += cw[u]; r += rw[u];
            }
        }
    int all, ptr;
    if (N <= 32) {                                                 // (one warp's buckets)
        int incl = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += t;
        }
        ptr = incl - c; all = incl;
    } else {
        ptr = cta_exclusive_scan(c, wsum, all);
    }
    if (tid < N) {
        out.ptr[tid] = cnt[tid] = ptr; out.total[tid] = r;
        if (tid == N - 1) out.ptr[N] = ptr + c;
    }
    __syncthreads();
    if (s.j >= 0) {
        const int at = cnt[s.j] + wcnt[warp * N + s.j] + __popc(b.lower);
        out.start[at] = wrow[warp * N + s.j] + b.pre;
        out.row[at] = s.row0;
    }
    __syncthreads();
}

// Builds the run table from the steps step(k), k < K.  `first` is step(threadIdx.x), which the caller fetches before it knows K
// (the plan arrays have k_max rows, and a trip to L2 is saved); what lies beyond K is ignored here.  out.* may be shared or global memory (each element is written once, by one thread); cnt is [N] ints of shared memory.
template <typename StepFn>
__device__ __forceinline__ void build_runs(int K, int N, Step first, StepFn step, Runs out, int* cnt, int* scratch, bool cleared = false) {
    if (K <= kIdxThreads) { build_runs_at_once(K, N, first, out, cnt, scratch, cleared); return; }
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
        const SameBucket b = same_bucket(j, rows);
        if (j >= 0 && (b.peers >> lane) == 1u) { wcnt[warp * N + j] = __popc(b.peers); wrow[warp * N + j] = b.pre + rows; }   // highest lane
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
            const int at = wcnt[warp * N + j] + __popc(b.lower);
            out.start[at] = wrow[warp * N + j] + b.pre;
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

// peer[k - k0] = the (highest) source rank whose lane of step k goes to `rank`, for the steps k0 <= k < k1; peer is shared memory and
// holds -1 before, behind a barrier; all threads of the CTA.  Cells are read as vectors of eight where they can be; sender_cells is
// the thread's first vector, which a caller that does not know k1 yet asks for ahead of it (the plan has k_max steps; a trip to
// L2 is saved).
__device__ __forceinline__ bool sender_vectors(const int16_t* base, int N) { return N % 8 == 0 && ((uintptr_t)base & 15) == 0; }
__device__ __forceinline__ uint4 sender_cells(const int16_t* __restrict__ base, int N, int steps) {
    return sender_vectors(base, N) && (long long)threadIdx.x * 8 < (long long)steps * N ? __ldg((const uint4*)base + threadIdx.x) : make_uint4(0, 0, 0, 0);
}
__device__ __forceinline__ void find_senders(const int16_t* __restrict__ lane_dst, int N, int rank, int k0, int k1, uint4 first, int* peer) {
    const int16_t* base = lane_dst + (size_t)k0 * N;
    const unsigned cells = (unsigned)(k1 - k0) * (unsigned)N;      // (at most kInlineCells, or a tile of 32 steps)
    if (sender_vectors(base, N)) {
#pragma unroll 4
        for (unsigned v = threadIdx.x; v < cells / 8; v += kIdxThreads) {
            const uint4 x = v == threadIdx.x ? first : __ldg((const uint4*)base + v);
            const uint32_t w[4] = {x.x, x.y, x.z, x.w};
            int high = -1;                                         // (a vector is one step's: its highest rank is all that counts)
#pragma unroll
            for (int q = 0; q < 8; q++) high = (int)((w[q >> 1] >> (16 * (q & 1))) & 0xffffu) == rank ? q : high;
            if (high >= 0) {
                const unsigned k = v / ((unsigned)N / 8);
                atomicMax(&peer[k], (int)(v * 8 - k * (unsigned)N) + high);
            }
        }
    } else {
        for (unsigned e = threadIdx.x; e < cells; e += kIdxThreads)
            if (base[e] == rank) {
                const unsigned k = e / (unsigned)N;
                atomicMax(&peer[k], (int)(e - k * (unsigned)N));
            }
    }
    __syncthreads();
}
// The same with everything that has to come before it.
__device__ __forceinline__ void find_senders(const int16_t* __restrict__ lane_dst, int N, int rank, int k0, int k1, int* peer) {
    for (int k = k0 + threadIdx.x; k < k1; k += kIdxThreads) peer[k - k0] = -1;
    const uint4 first = sender_cells(lane_dst + (size_t)k0 * N, N, k1 - k0);
    __syncthreads();
    find_senders(lane_dst, N, rank, k0, k1, first, peer);
}

// Calls f(i, x[i]) for lo <= i < hi over the CTA, four loads (of four values where x is 16-byte aligned) in flight per thread.  They
// are written out: f has atomics, which the compiler moves no load across (an item then took a trip to L2 of its own).
template <typename F>
__device__ __forceinline__ void for_each_item(const int32_t* __restrict__ x, int lo, int hi, F f) {
    const bool vec = ((uintptr_t)x & 15) == 0;
    int v0 = vec ? (lo + 3) & ~3 : hi, v1 = vec ? hi & ~3 : hi;
    if (hi - lo < 4 * kIdxThreads || v0 >= v1) v0 = v1 = hi;       // (fewer: one value per thread spreads the work better)
    for (int i0 = lo + threadIdx.x; i0 < v0; i0 += 4 * kIdxThreads) {
        int y[4];
#pragma unroll
        for (int u = 0; u < 4; u++) y[u] = i0 + u * kIdxThreads < v0 ? __ldg(x + i0 + u * kIdxThreads) : 0;
#pragma unroll
        for (int u = 0; u < 4; u++)
            if (i0 + u * kIdxThreads < v0) f(i0 + u * kIdxThreads, y[u]);
    }
    for (int w0 = v0 / 4 + threadIdx.x; w0 < v1 / 4; w0 += 4 * kIdxThreads) {
        int4 y[4];
#pragma unroll
        for (int u = 0; u < 4; u++) y[u] = w0 + u * kIdxThreads < v1 / 4 ? __ldg((const int4*)x + w0 + u * kIdxThreads) : make_int4(0, 0, 0, 0);
#pragma unroll
        for (int u = 0; u < 4; u++) {
            const int i = 4 * (w0 + u * kIdxThreads);
            if (i >= v1) break;
            f(i, y[u].x); f(i + 1, y[u].y); f(i + 2, y[u].z); f(i + 3, y[u].w);
        }
    }
    for (int i = v1 + threadIdx.x; i < hi; i += kIdxThreads) f(i, __ldg(x + i));
}

// Counts of the warps' slices, count[w * stride], to the first position of each, starting at `run`; returns where the last one ends.
// (Eight read before the first of them is written: one after the other each read waits for the write ahead of it.  All sixteen at once
// cost the pack's map 62 registers instead of 40, so that its grid of up to 256 CTAs and the launches beside it no longer fit: 120,000
// copies of 96 B from 8, 16 and 64 ranks 34.9, 36.8 and 42.5 us by sixteen, 28.6, 30.8 and 38.1 by eight; of 1,536 B from 64 ranks 51.0, 52.7.)
__device__ __forceinline__ int slices_prefix(int* count, int stride, int run) {
    constexpr int U = 8;
    static_assert(kIdxWarps % U == 0, "whole batches");
#pragma unroll 1
    for (int w0 = 0; w0 < kIdxWarps; w0 += U) {
        int x[U];
#pragma unroll
        for (int u = 0; u < U; u++) x[u] = count[(w0 + u) * stride];
#pragma unroll
        for (int u = 0; u < U; u++) { count[(w0 + u) * stride] = run; run += x[u]; }
    }
    return run;
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

// Positions of the items a CTA owns: key[i] is own item i's key (-1: none; 16-byte aligned shared memory), next[] the position of the
// first own item of every key.  An item's position counts the equal keys before it: an item per thread, four keys per read, no
// chain (__match_any_sync takes 570 cycles, and a warp that carries next[] on waits for it per 32 items).
template <typename Put>
__device__ __forceinline__ void own_positions(const int* key, int own, const int* next, Put put) {
    for (int i = threadIdx.x; i < own; i += kIdxThreads) {
        const int k = key[i];
        int p = -1;
        if (k >= 0) {
            p = next[k];
            for (int q = 0; q < i; q += 4) {
                const int4 x = *(const int4*)(key + q);
                p += (x.x == k) + (q + 1 < i && x.y == k) + (q + 2 < i && x.z == k) + (q + 3 < i && x.w == k);
            }
        }
        put(i, k, p);
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

// The same by bulk asynchronous copies (TMA): rows of at least kMinOwnBulk (return: kMinReturnBulk) bytes at 16-byte addresses.  A unit is one piece of one
// own row; warp w < kOwnWarps drives every kOwnWarps-th unit through a ring of its own.  Loads need no index where the source rows
// are known before it (pack, unpack): they are in flight while it is worked out, and what follows it is the stores alone.  (They start
// behind the loads that the index waits for: ahead of them they keep those waiting, 4 us with six stages full on every SM.)  Pack of
// 16 ranks, 8,192 copies of 14,336 B, by plain loads and two CTAs per SM 33.9 us, so 24.1; 1,024 copies 8.2, so 6.8, of which 2.5 are
// the stores, at 5.6 TB/s.
constexpr int kOwnWarps = 2;
constexpr int kOwnStages = 6;
constexpr int kOwnPiece = 16384;                    // bytes per unit, at most
constexpr int kMinOwnBulk = 2048;
// The return knows its source rows behind the index only, and two warps issue a unit per row: rows below 7 KB move faster by plain
// loads (8,192 copies, by rings | plain, us, 16 ranks: rows of 2,048 B 18.3 | 11.1, 4,096 20.7 | 18.0, 6,144 24.3 | 23.5, 7,392 26.8 | 26.8,
// 8,192 27.9 | 28.4, 14,336 43.8 | 45.4; 64 ranks 20.2 | 13.3, 22.6 | 20.3, 26.3 | 25.9, 28.8 | 29.3, 30.0 | 31.0, 46.9 | 48.5).
constexpr int kMinReturnBulk = 7168;
constexpr unsigned kOwnSpins = 1u << 22;            // bounded mbarrier wait

// How a small problem is dealt, and what a one-launch kernel is told about it.
struct SmallLaunch {
    int grid, pieces, own;                          // CTAs, CTAs per row, places in dst (and src) per CTA
    int ring, stages, stage_bytes, piece;           // the rings' place in shared memory, stages of each, bytes of a stage and of a unit
    size_t smem;
    bool bulk;
};

template <unsigned SPINS>
struct OwnRingOf {
    const char* rows;
    char* out;
    long long row_bytes;
    int col0, cols, piece, pieces, units;           // this CTA's bytes of every row, of a unit, units per row, this warp's units
    unsigned ring, bars, stage_bytes;               // shared memory addresses
    unsigned loaded, phase;                         // per stage: holds a load; parity

    __device__ __forceinline__ void init(const SmallLaunch& z, const char* rows_, char* out_, long long row_bytes_, int v_lo, int v_hi, void* smem,
                                         unsigned long long* bars_) {
        const int w = threadIdx.x >> 5;
        rows = rows_; out = out_; row_bytes = row_bytes_;
        col0 = v_lo * 16; cols = (v_hi - v_lo) * 16; piece = z.piece; pieces = (cols + piece - 1) / piece; units = 0;
        stage_bytes = (unsigned)z.stage_bytes;
        ring = smem_u32((unsigned char*)smem + z.ring) + w * z.stages * stage_bytes; bars = smem_u32(bars_ + w * kOwnStages);
        loaded = phase = 0;
        if ((threadIdx.x & 31) == 0) {
            for (int s = 0; s < kOwnStages; s++) mbar_init(bars + 8 * s, 1);
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        }
        __syncwarp();
    }
    struct Unit { int row, at; };                   // own row, first byte
    __device__ __forceinline__ Unit unit(int u) const {
        const int g = u * kOwnWarps + (int)(threadIdx.x >> 5);
        if (pieces == 1) return Unit{g, 0};
        const int row = g / pieces;
        return Unit{row, (g - row * pieces) * piece};
    }
    template <typename Src>
    __device__ __forceinline__ bool issue(int u, Src src) const {  // one thread: the load of unit u < units; false: none
        const Unit n = unit(u);
        const int s = u % kOwnStages, from = src(n.row);
        if (from < 0) return false;
        const unsigned bytes = (unsigned)min(piece, cols - n.at), bar = bars + 8 * s;
        mbar_expect_tx(bar, bytes);
        bulk_load(ring + s * stage_bytes, rows + from * row_bytes + col0 + n.at, bytes, bar);
        return true;
    }
    // Loads in flight land before the CTA's shared memory is another's.
    __device__ __forceinline__ bool drain() {
        bool ok = true;
        for (int s = 0; s < kOwnStages; s++)
            if (loaded >> s & 1) ok &= mbar_wait_bounded(bars + 8 * s, phase >> s & 1u, SPINS);
        loaded = 0;
        return ok;
    }
    // Loads of the first units; src(i) is the source row of own row i < own, -1: none.
    template <typename Src>
    __device__ __forceinline__ void start(int own, Src src) {
        const int lane = threadIdx.x & 31;          // (a unit per lane: one after the other they take 330 cycles each)
        units = (own * pieces + kOwnWarps - 1 - (int)(threadIdx.x >> 5)) / kOwnWarps;
        const bool mine = lane < min(units, kOwnStages) && issue(lane, src);
        loaded = __ballot_sync(0xffffffffu, mine);
    }
    // Unit u by plain loads and stores, the whole warp.
    template <typename Src>
    __device__ __forceinline__ void move_plain(int u, int fanout, const int* dst, Src src) const {
        const Unit n = unit(u);
        const int from = src(n.row), vecs = min(piece, cols - n.at) / 16;
        if (from < 0) return;
        const uint4* const x = (const uint4*)(rows + from * row_bytes + col0 + n.at);
#pragma unroll 1
        for (int f = 0; f < fanout; f++) {
            const int d = dst[n.row * fanout + f];
            if (d < 0) continue;
            uint4* const to = (uint4*)(out + d * row_bytes + col0 + n.at);
#pragma unroll 1
            for (int v = threadIdx.x & 31; v < vecs; v += 32) to[v] = x[v];
        }
    }
    // Stores every unit to its destination rows dst[i * fanout + f] (-1: none) and loads the others; false: a wait gave up.  All units
    // are stored either way, those that are left then by plain loads: the caller reports it by a bit in the status word, which another CTA
    // writes by a plain store, so the bit may be lost, and no output may depend on it.
    template <typename Src>
    __device__ __forceinline__ bool finish(int fanout, const int* dst, Src src) {
        constexpr int S = kOwnStages, D = S / 2;    // a stage is loaded again D units after its stores
        const int lane = threadIdx.x & 31;
        bool failed = false;
        int u = 0;
        for (; u < units; u++) {
            const int s = u % S;
            const Unit n = unit(u);
            if (loaded >> s & 1) {
                failed = __any_sync(0xffffffffu, !mbar_wait_bounded(bars + 8 * s, phase >> s & 1u, SPINS));
                if (failed) break;
                loaded &= ~(1u << s);
                phase ^= 1u << s;
                const unsigned bytes = (unsigned)min(piece, cols - n.at);
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                for (int f = lane; f < fanout; f += 32) {
                    const int d = dst[n.row * fanout + f];
                    if (d >= 0) bulk_store(out + d * row_bytes + col0 + n.at, ring + s * stage_bytes, bytes);
                }
            }
            bulk_commit();                          // one group per unit from every lane, empty or not
            if (u >= D && u + S - D < units) {
                bulk_wait_read<D>();
                __syncwarp();
                const bool mine = lane == 0 && issue(u + S - D, src);
                if (__any_sync(0xffffffffu, mine)) loaded |= 1u << (u + S - D) % S;
            }
        }
        if (__builtin_expect(failed, 0)) {          // (no load is in flight otherwise)
#pragma unroll 1
            for (; u < units; u++) move_plain(u, fanout, dst, src);
            drain();
        }
        bulk_wait_read<0>();                        // the stores have read shared memory
        return !failed;
    }
};
using OwnRing = OwnRingOf<kOwnSpins>;

// Copies of `width` bytes, by rings from rows of min_bulk bytes on; ints(own) words of index in shared memory when a CTA owns up to `own` of the n rows.  With rings one CTA
// per SM, as a CTA's index costs the same however many rows it owns; by plain loads two, for the loads in flight.  While there are
// fewer rows than that, up to eight CTAs take a row's columns: with rings 74 rows are 148 CTAs and 75 rows 75 (pack of 74, 75, 96, 128, 147 and
// 148 tokens x 8 of 14,336 B 5.9, 6.3, 6.5, 6.7, 6.8, 7.0 us; by plain loads and up to 296 CTAs 7.4, 7.4, 7.5, 8.3, 8.4, 8.4 before).
template <typename Ints>
inline SmallLaunch small_launch(int n, int sms, int fanout, long long row_bytes, int width, int min_bulk, Ints ints) {
    SmallLaunch z{};
    for (int per_sm = width == 16 && row_bytes >= min_bulk ? 1 : 2; per_sm <= 2; per_sm++) {
        const int most = per_sm * sms;
        z.pieces = n >= sms ? 1 : (most / n < 8 ? most / n : 8);
        z.grid = n >= sms ? (n < most ? n : most) : n * z.pieces;
        const int n_cta = z.grid / z.pieces, own = (n + n_cta - 1) / n_cta, words = ints(own);
        z.own = own * fanout;
        z.smem = (size_t)words * 4;
        if (per_sm == 2) break;
        const long long cols = (row_bytes / 16 + z.pieces - 1) / z.pieces * 16;
        const long long split = own >= kOwnWarps ? cols : (cols / 16 + kOwnWarps - 1) / kOwnWarps * 16;   // (a unit for every warp)
        z.piece = split < kOwnPiece ? (int)split : kOwnPiece;
        z.stage_bytes = (z.piece + 127) & ~127;
        const long long units = (own * ((cols + z.piece - 1) / z.piece) + kOwnWarps - 1) / kOwnWarps;
        z.stages = units < kOwnStages ? (int)units : kOwnStages;
        z.ring = (words * 4 + 127) & ~127;
        const size_t with_rings = (size_t)z.ring + (size_t)kOwnWarps * z.stages * z.stage_bytes;
        if (with_rings <= kSmemLimit) { z.smem = with_rings; z.bulk = true; break; }
    }
    return z;
}

}  // namespace
