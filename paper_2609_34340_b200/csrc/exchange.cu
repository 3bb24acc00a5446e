// Plan execution over peer memory (Section 5, "Device-resident buffer layout"): the step between vp_pack and vp_unpack.
//
// A rank's staged send buffer holds one contiguous chunk per activation; the chunk of step k goes to the step's
// destination j = lane_dst[k][rank] and lands at j's running receive offset recv_off[k][j].  vp_exchange_put is the
// sender side: stores through pointers to the receivers' buffers -- ordinary device memory when the ranks share
// a GPU, peer-mapped memory of other GPUs over NVLink otherwise -- followed by a system-wide fence and, per CTA and destination,
// an addition to the receiver's device-resident arrival counter.  vp_exchange_wait is the receiver side: a bounded
// wait until the counter has reached the bytes the plan sends this rank, which is what replaces a global barrier.
// Double buffering is the caller's: two receive buffers and two counters per rank, alternated between invocations.
//
// No multicast and no cluster-scope copies: every byte moves by a bulk copy of this CTA or by an ordinary load and store, so
// the same code is valid for local and for peer destinations.
#include <cuda_runtime.h>

#include "announce.h"
#include "row_copy.cuh"
#include "vp_internal.h"

namespace {

constexpr int kPutThreads = 256;
constexpr int kPutStages = 6;

struct PutArgs {
    const int32_t* n_steps;
    const int16_t* lane_dst;
    const int64_t *send_off, *recv_off;
    int N, rank, k_max;
    const unsigned char* staged;
    unsigned char* const* recv_bufs;
    const int64_t* recv_capacity;
    unsigned long long* const* arrived;
    int32_t* status;
};

// The step that holds byte `at` of the send buffer: the last k < K with send_off[k] <= at (offsets do not decrease).  Whole
// warp: one trip to L2 for plans of up to 256 activations, else 32 places are read at a time.
__device__ __forceinline__ int put_step_of(const PutArgs& a, int K, long long at) {
    const int lane = threadIdx.x & 31;
    if (K <= 256) {
        int before = 0;
#pragma unroll
        for (int i = 0; i < 8; i++) {
            const int k = i * 32 + lane;
            before += k < K && a.send_off[(size_t)k * a.N + a.rank] <= at;
        }
        return max((int)__reduce_add_sync(0xffffffffu, (unsigned)before) - 1, 0);
    }
    int lo = 0, n = K;                               // the answer is in [lo, lo + n)
    while (n > 1) {
        const int stride = (n + 31) / 32, k = lo + lane * stride;
        const bool before = lane * stride < n && a.send_off[(size_t)k * a.N + a.rank] <= at;
        const int last = 31 - __clz((int)(__ballot_sync(0xffffffffu, before) | 1u));
        n = min(stride, n - last * stride);
        lo += last * stride;
    }
    return lo;
}

// Calls f(from, bytes, destination, j) for every part of a chunk inside the bytes [lo, hi), from the step k0 on; whole warp.
// The figures of 32 steps are fetched together, a step per lane.  A part that would overrun its receiver is left out.
template <typename F>
__device__ __forceinline__ bool put_parts(const PutArgs& a, int K, int k0, long long lo, long long hi, F f) {
    const int lane = threadIdx.x & 31;
    bool over = false;
    for (; k0 < K; k0 += 32) {
        long long s0 = 0, s1 = 0, room = 0;
        unsigned long long dst = 0;
        int j = -1;
        if (k0 + lane < K) {
            const size_t at = (size_t)(k0 + lane) * a.N;
            s0 = a.send_off[at + a.rank];
            s1 = a.send_off[at + a.N + a.rank];
            j = a.lane_dst[at + a.rank];
            if (j >= 0) {
                const long long r = a.recv_off[at + j];
                room = a.recv_capacity[j] - r;
                dst = (unsigned long long)(uintptr_t)a.recv_bufs[j] + (unsigned long long)r;
            }
        }
        const int n = min(32, K - k0);
        for (int i = 0; i < n; i++) {
            const long long c0 = __shfl_sync(0xffffffffu, s0, i), c1 = __shfl_sync(0xffffffffu, s1, i);
            if (c0 >= hi) return over;
            const int to_j = __shfl_sync(0xffffffffu, j, i);
            const long long left = __shfl_sync(0xffffffffu, room, i);
            unsigned char* const base = (unsigned char*)(uintptr_t)__shfl_sync(0xffffffffu, dst, i);
            const long long from = max(c0, lo), to = min(c1, hi);
            if (to_j < 0 || from >= to) continue;
            if (to - c0 > left) { over = true; continue; }          // not copied, reported
            f(from, to - from, base + (from - c0), to_j);
        }
    }
    return over;
}

// Copies n bytes between addresses of any alignment, warp w of n_warps.  The destination's 16-byte vectors are put together
// from pairs of aligned source vectors by funnel shifts; only the first and last bytes go one by one.  (Byte loads and
// stores throughout moved 4,100-byte rows at a tenth of the bandwidth.)
template <int WORDS>
__device__ __forceinline__ uint4 put_shift(const uint4& x, const uint4& y, int bits) {
    const uint32_t w[8] = {x.x, x.y, x.z, x.w, y.x, y.y, y.z, y.w};
    return make_uint4(__funnelshift_r(w[WORDS], w[WORDS + 1], bits), __funnelshift_r(w[WORDS + 1], w[WORDS + 2], bits),
                      __funnelshift_r(w[WORDS + 2], w[WORDS + 3], bits), __funnelshift_r(w[WORDS + 3], w[WORDS + 4], bits));
}
template <int WORDS>
__device__ __forceinline__ void put_vectors(unsigned char* dst, const unsigned char* src, long long vecs, int bits, int w, int n_warps) {
    const int lane = threadIdx.x & 31;
    const uint4* const s = (const uint4*)src;         // (aligned down: vector v + 1 holds the rest)
    for (long long v0 = (long long)w * 128 + lane; v0 - lane < vecs; v0 += (long long)n_warps * 128) {
        uint4 x[4], y[4];
#pragma unroll
        for (int u = 0; u < 4; u++)
            if (v0 + 32 * u < vecs) { x[u] = __ldg(s + v0 + 32 * u); y[u] = __ldg(s + v0 + 32 * u + 1); }
#pragma unroll
        for (int u = 0; u < 4; u++)
            if (v0 + 32 * u < vecs) ((uint4*)dst)[v0 + 32 * u] = put_shift<WORDS>(x[u], y[u], bits);
    }
}
__device__ __forceinline__ void put_any(unsigned char* dst, const unsigned char* src, long long n, int w, int n_warps) {
    const int lane = threadIdx.x & 31;
    // the vectors start at the first aligned destination byte whose aligned source vector lies inside [src, src + n) ...
    long long head = min(n, (long long)((16 - ((uintptr_t)dst & 15)) & 15));
    if (((uintptr_t)(src + head) & 15) > (unsigned long long)head) head = min(n, head + 16);
    const int off = (int)((uintptr_t)(src + head) & 15);
    // ... and end where the second source vector would leave it
    long long vecs = (n - head - 16 + off) / 16;
    if (vecs < 0 || n - head - 16 + off < 0) vecs = 0;
    for (long long e = lane + 32 * w; e < head; e += 32 * n_warps) dst[e] = src[e];
    const unsigned char* const s = src + head - off;
    switch (off >> 2) {
        case 0: put_vectors<0>(dst + head, s, vecs, 8 * (off & 3), w, n_warps); break;
        case 1: put_vectors<1>(dst + head, s, vecs, 8 * (off & 3), w, n_warps); break;
        case 2: put_vectors<2>(dst + head, s, vecs, 8 * (off & 3), w, n_warps); break;
        default: put_vectors<3>(dst + head, s, vecs, 8 * (off & 3), w, n_warps); break;
    }
    for (long long e = head + vecs * 16 + lane + 32 * w; e < n; e += 32 * n_warps) dst[e] = src[e];
}

// CTA c moves the bytes [c, c + 1) x total / CTAs of the send buffer (rounded to 16 bytes), chunk part by chunk part.  (Pieces
// dealt round robin copy 2 % faster, but every CTA then walks the whole plan: 10 us on the 290 activations of 64 ranks.)
// Parts whose addresses and size are multiples of 16 go through shared memory as bulk asynchronous copies that one thread of
// warp 0 issues (pieces of up to 16 KB, six stages); others are moved by all warps.  One system fence by one warp per CTA
// announces all its parts: fences by every thread, and a second walk over the plan behind them, took 12 us of any call.
// Bound by HBM.  On one GPU 2,048 tokens x top-8 of 14,336 B (440 MB read and written) took 92 us with plain 16-byte loads
// and stores, now 81; 32 tokens take 12 us less.
__global__ void __launch_bounds__(kPutThreads) exchange_put_kernel(PutArgs a) {
    extern __shared__ __align__(128) unsigned char ring[];
    __shared__ __align__(8) unsigned long long bars[kPutStages];
    __shared__ unsigned char* s_dst[kPutStages];
    __shared__ unsigned s_bytes[kPutStages];
    __shared__ unsigned long long* s_counter[VP_MAX_N];       // every rank's counter, and the bytes this CTA adds to it
    __shared__ unsigned long long s_count[VP_MAX_N];
    const int tid = threadIdx.x, warp = tid >> 5;
    if (tid == 0) {
        for (int s = 0; s < kPutStages; s++) mbar_init(smem_u32(&bars[s]), 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    grid_wait();
    const int K = min(max(*a.n_steps, 0), a.k_max);
    const long long total = a.send_off[(size_t)K * a.N + a.rank];
    // (small sends: 16 KB per CTA and fewer CTAs, each of which costs a system fence)
    const long long ctas = min((long long)gridDim.x, (total + kPiece - 1) / kPiece), c = blockIdx.x;
    if (c >= ctas) return;
    const long long lo = (total * c / ctas) & ~15ll, hi = c == ctas - 1 ? total : (total * (c + 1) / ctas) & ~15ll;
    if (lo >= hi) return;
    for (int j = tid; j < a.N; j += kPutThreads) { s_counter[j] = a.arrived ? a.arrived[j] : nullptr; s_count[j] = 0; }
    const int k0 = put_step_of(a, K, lo);
    __syncthreads();
    constexpr int S = kPutStages, kLook = S / 2;
    int issued = 0, done = 0;                        // pieces (thread 0)
    bool failed = false;
    auto retire = [&]() {                            // oldest piece: wait for its load, store it
        const int s = done % S;
        if (!mbar_wait_bounded(smem_u32(&bars[s]), (unsigned)(done / S) & 1u, kSpinLimit)) failed = true;
        if (!failed) {
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            bulk_store(s_dst[s], smem_u32(ring + (size_t)s * kPiece), s_bytes[s]);
        }
        bulk_commit();
        done++;
    };
    const bool over = put_parts(a, K, k0, lo, hi, [&](long long from, long long n, unsigned char* dst, int j) {
        const unsigned char* const src = a.staged + from;
        if (tid == 0) s_count[j] += (unsigned long long)n;
        if ((((uintptr_t)src | (uintptr_t)dst | (uintptr_t)n) & 15) == 0) {
            if (tid == 0)
                for (long long at = 0; at < n && !failed; at += kPiece) {
                    if (issued - done == kLook) retire();
                    if (failed) break;
                    bulk_wait_read<S - kLook - 1>();
                    const int s = issued % S;
                    const unsigned bytes = (unsigned)min((long long)kPiece, n - at);
                    mbar_expect_tx(smem_u32(&bars[s]), bytes);
                    bulk_load(smem_u32(ring + (size_t)s * kPiece), src + at, bytes, smem_u32(&bars[s]));
                    s_dst[s] = dst + at; s_bytes[s] = bytes;
                    issued++;
                }
            __syncwarp();
        } else {
            put_any(dst, src, n, warp, kPutThreads / 32);
        }
    });
    if (tid == 0) {
        while (done < issued) retire();              // (once a wait has given up: only waits, bounded, for the loads in flight)
        bulk_wait_all();
        asm volatile("fence.proxy.async;" ::: "memory");     // the bulk stores before the counters below
        if (over) atomicOr(a.status, VP_ST_PACK_CAPACITY);
        if (failed) atomicOr(a.status, VP_ST_INTERNAL_TIMEOUT);
    }
    if (a.arrived) {
        // every thread's stores become visible system-wide before the counts that announce them
        if (__syncthreads_or(failed)) return;
        if (warp == 0)
            announce_counts(tid, a.N, s_count, [] { __threadfence_system(); },
                            [&](int j, unsigned long long bytes) { if (s_counter[j]) atomicAdd_system(s_counter[j], bytes); });
    }
}

// One thread polls this rank's counter with acquire loads until it holds the expected bytes, at most max_polls times.
__global__ void exchange_wait_kernel(const int32_t* __restrict__ n_steps, const int64_t* __restrict__ recv_off, int N, int rank,
                                     int k_max, const unsigned long long* counter, unsigned long long base,
                                     unsigned int max_polls, int32_t* __restrict__ status) {
    const int K = min(max(*n_steps, 0), k_max);
    const unsigned long long want = base + (unsigned long long)recv_off[(size_t)K * N + rank];
    for (unsigned int p = 0; p <= max_polls; p++) {
        unsigned long long seen;
        asm volatile("ld.acquire.sys.global.u64 %0, [%1];" : "=l"(seen) : "l"(counter) : "memory");
        if (seen >= want) return;
        __nanosleep(200);
    }
    atomicOr(status, VP_ST_EXCHANGE_TIMEOUT);                   // gave up: the caller reads the bit; nothing hangs
}

}  // namespace

extern "C" int vp_exchange_put(const int32_t* n_steps_b, const int16_t* lane_dst_b, const int64_t* send_off_b,
                               const int64_t* recv_off_b, int N, int rank, int k_max, const void* staged,
                               void* const* recv_bufs, const int64_t* recv_capacity_bytes, uint64_t* const* arrived,
                               int32_t* status, void* cuda_stream) {
    if (!n_steps_b || !lane_dst_b || !send_off_b || !recv_off_b || !staged || !recv_bufs || !recv_capacity_bytes || !status)
        return VP_E_BAD_ARG;
    if (N <= 0 || N > VP_MAX_N || rank < 0 || rank >= N || k_max <= 0) return VP_E_BAD_ARG;
    const int sms = sm_count_of_device();
    if (!sms) return VP_E_CUDA;
    static bool s_attr_set[64] = {false};            // per device, once
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return VP_E_CUDA;
    const size_t smem = (size_t)kPutStages * kPiece;
    if (dev < 0 || dev >= 64 || !s_attr_set[dev]) {
        if (cudaFuncSetAttribute(exchange_put_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) return VP_E_CUDA;
        if (dev >= 0 && dev < 64) s_attr_set[dev] = true;
    }
    const PutArgs a{n_steps_b, lane_dst_b, send_off_b, recv_off_b, N, rank, k_max, (const unsigned char*)staged,
                    (unsigned char* const*)recv_bufs, recv_capacity_bytes, (unsigned long long* const*)arrived, status};
    return launch_after(exchange_put_kernel, sms * 2, kPutThreads, smem, (cudaStream_t)cuda_stream, a) == cudaSuccess ? VP_OK : VP_E_CUDA;
}

extern "C" int vp_exchange_wait(const int32_t* n_steps_b, const int64_t* recv_off_b, int N, int rank, int k_max,
                                const uint64_t* arrived_counter, uint64_t counter_base, uint32_t max_polls, int32_t* status,
                                void* cuda_stream) {
    if (!n_steps_b || !recv_off_b || !arrived_counter || !status) return VP_E_BAD_ARG;
    if (N <= 0 || N > VP_MAX_N || rank < 0 || rank >= N || k_max <= 0) return VP_E_BAD_ARG;
    exchange_wait_kernel<<<1, 1, 0, (cudaStream_t)cuda_stream>>>(n_steps_b, recv_off_b, N, rank, k_max,
                                                                 (const unsigned long long*)arrived_counter,
                                                                 (unsigned long long)counter_base, max_polls, status);
    g_vp_launches++;
    return cudaGetLastError() == cudaSuccess ? VP_OK : VP_E_CUDA;
}
