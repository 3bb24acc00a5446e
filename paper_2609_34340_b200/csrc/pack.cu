// vp_pack: stage one rank's routed token rows in activation x destination order
// (Section 5, "Device-resident buffer layout").
//
// Up to kSmallItems routed copies: one kernel (pack_small_kernel).  More: three kernels on the caller's stream:
//   count : per chunk of copies a histogram of destination ranks; one more CTA builds, meanwhile, the rank's run table
//           (for every destination the activations that send to it, with the stream position they start at and their
//           first staged row) from the plan's send offsets
//   map   : stable position of every copy inside its destination's stream -> staged row; writes src_map and the status
//   copy  : token-major: every source row is read ONCE and written to each of its staged rows (row_copy.cuh)
#include <cuda_runtime.h>

#include "row_copy.cuh"
#include "vp_internal.h"

namespace {

struct PackArgs {
    const int32_t* n_steps;
    const int16_t* lane_dst;
    const int64_t *lane_bytes, *send_off;
    int N, rank, k_max, T, topk;
    SmallDiv epr;
    const int32_t* idx;
    RowDiv row;
    int64_t capacity;
    int32_t *src_map, *status;
};

struct PackWs {
    int32_t* flags;      // [0] abort, [1] status bits of the run table
    int32_t* hist;       // [n_chunks][N] copies of each chunk per destination
    int32_t* bad;        // [n_chunks] status bits of each chunk
    int32_t* total;      // [N] rows the plan sends to each destination
    int32_t* ptr;        // [N+1] \ run table (see Runs)
    int32_t* start;      // [k_max] |
    int32_t* row;        // [k_max] /
    int32_t* dst_row;    // [T*topk] staged row of each copy, -1 = not staged
    size_t bytes;
};

PackWs carve(void* base, int N, int T, int topk, int k_max) {
    PackWs w;
    size_t o = 0;
    auto take = [&](size_t n) { size_t at = o; o += vp_align256(n); return (int32_t*)((char*)base + at); };
    const long long E = (long long)T * topk, chunk = chunk_items(E, N);
    const size_t n_chunks = (size_t)((E + chunk - 1) / chunk);
    w.flags = take(256);
    w.hist = take(n_chunks * N * 4);
    w.bad = take(n_chunks * 4);
    w.total = take((size_t)N * 4);
    w.ptr = take((size_t)(N + 1) * 4);
    w.start = take((size_t)k_max * 4);
    w.row = take((size_t)k_max * 4);
    w.dst_row = take((size_t)E * 4);
    w.bytes = o;
    return w;
}

// Destination rank of a routed copy, or -1 if it is not staged (dropped, local, out of range: that one sets `bad`).
__device__ __forceinline__ int dest_of(int x, const PackArgs& a, int& bad) {
    if (x < 0) return -1;
    const int j = a.epr.div(x);
    if (j >= a.N) { bad = VP_ST_PACK_MISMATCH; return -1; }
    return j == a.rank ? -1 : j;
}

__device__ __forceinline__ int steps_in_use(const PackArgs& a) { return min(max(*a.n_steps, 0), a.k_max); }

// A step's figures as the plan has them; pack_step makes rows of them.
struct RawStep { int j; int64_t bytes, off; };
__device__ __forceinline__ RawStep raw_step(const PackArgs& a, int k) {
    const size_t at = (size_t)k * a.N + a.rank;
    return RawStep{a.lane_dst[at], a.lane_bytes[at], a.send_off[at]};
}
__device__ __forceinline__ Step pack_step(const PackArgs& a, const RawStep& raw, int& bad) {
    int64_t odd, ignore;
    const int j = raw.j;
    const int64_t rows = a.row.div(raw.bytes, odd), row0 = a.row.div(raw.off, ignore);
    if (j < 0 || j >= a.N) return Step{-1, 0, 0};
    if (odd) bad = VP_ST_PACK_MISMATCH;
    return Step{j, (int)rows, (int)row0};
}

// Status bits of the run table, the same in every thread (left out unless `report`).
__device__ __forceinline__ int pack_runs(const PackArgs& a, int K, Step first, int bad, Runs out, int* cnt, int* scratch, bool cleared = false, bool report = true) {
    if ((int)threadIdx.x >= K) bad = 0;
    build_runs(K, a.N, first, [&](int k) { return pack_step(a, raw_step(a, k), bad); }, out, cnt, scratch, cleared);
    if (!report) return 0;
    if (threadIdx.x == 0 && out.total[a.rank] != 0) bad = VP_ST_PACK_MISMATCH;
    return __syncthreads_or(bad) ? VP_ST_PACK_MISMATCH : 0;
}

// ---- one launch -------------------------------------------------------------------------------------------------

struct PackSmall { int key, cnt, hist, total, ptr, start, row, src, dst, scratch, ints; };   // offsets in ints
__host__ __device__ inline PackSmall pack_small_layout(int N, int k_max, int own) {
    PackSmall L;
    int o = 0;
    L.key = o;     o += (own + 3) & ~3;              // (read four at a time)
    L.cnt = o;     o += N;
    L.hist = o;    o += N;
    L.total = o;   o += N;
    L.ptr = o;     o += N + 1;
    L.start = o;   o += k_max;
    L.row = o;     o += k_max;
    L.src = o;     o += own;
    L.dst = o;     o += own;
    L.scratch = o; o += runs_scratch_ints(N);
    L.ints = o;
    return L;
}

// Decode steps and prefill chunks of a few thousand tokens.  Bound by latency (launch, one trip to L2 for plan and routing, the
// run table: 3 us), then by HBM writes.  CTA c owns the tokens [c T / grid, (c + 1) T / grid) -- or one of `pieces` column
// ranges of one token while there are fewer tokens than SMs -- and finds their places by itself: the run table from the
// plan, and how many copies to each destination come before its own.  The last CTA thereby sees every copy and writes the
// status.  Replaces two memsets and four kernels: 128 tokens x top-8 of 14,336 B 30 -> 6.8 us a call.
template <typename V, bool BULK>
__global__ void __launch_bounds__(kIdxThreads, BULK ? 1 : 2)
pack_small_kernel(PackArgs a, const char* __restrict__ rows, char* __restrict__ staged, SmallLaunch z) {
    extern __shared__ __align__(128) int sm[];
    __shared__ __align__(8) unsigned long long bars[kOwnWarps * kOwnStages];
    const PackSmall L = pack_small_layout(a.N, a.k_max, z.own);
    const int pieces = z.pieces;
    int* const hist = sm + L.hist;
    const int tid = threadIdx.x, n_cta = gridDim.x / pieces, c = blockIdx.x / pieces, piece = blockIdx.x - c * pieces;
    const int t0 = (int)((long long)a.T * c / n_cta), t1 = (int)((long long)a.T * (c + 1) / n_cta);
    const int vecs = (int)(a.row.d / (int64_t)sizeof(V)), v_lo = (int)((long long)vecs * piece / pieces),
              v_hi = (int)((long long)vecs * (piece + 1) / pieces);
    for (int j = tid; j < a.N; j += kIdxThreads) hist[j] = 0;
    OwnRing ring;
    if (BULK && tid < kOwnWarps * 32) ring.init(z, rows, staged, a.row.d, v_lo, v_hi, sm, bars);
    int *const src = sm + L.src, *const dst = sm + L.dst, *const own_key = sm + L.key;
    clear_runs_scratch(a.N, sm + L.scratch);
    __syncthreads();
    grid_wait();
    // All that the index needs is asked for at once; rows are loaded behind it (ahead of it they keep it waiting).
    const RawStep raw = tid < a.k_max ? raw_step(a, tid) : RawStep{-1, 0, 0};
    const int K = steps_in_use(a), own = (t1 - t0) * a.topk;
    int bad = 0, bad_step = 0;
    for (int i = tid; i < own; i += kIdxThreads) own_key[i] = dest_of(a.idx[t0 * a.topk + i], a, bad);
    for_each_item(a.idx, 0, t0 * a.topk, [&](int, int x) {
        const int j = dest_of(x, a, bad);
        if (j >= 0) atomicAdd(&hist[j], 1);
    });
    const int64_t end = a.send_off[(size_t)K * a.N + a.rank];
    if (BULK && tid < kOwnWarps * 32) ring.start(t1 - t0, [&](int i) { return t0 + i; });
    const Step first = pack_step(a, raw, bad_step);
    const Runs runs{sm + L.start, sm + L.row, sm + L.ptr, sm + L.total};
    const bool last = c == n_cta - 1 && piece == 0;
    const int st = pack_runs(a, K, first, bad_step, runs, sm + L.cnt, sm + L.scratch, true, last);   // (has barriers: the histogram and the own copies are complete, too)
    const bool over = end > a.capacity;
    own_positions(own_key, own, hist, [&](int i, int j, int p) {
        const int row = p >= 0 && !over ? run_lookup(runs, j, p) : -1;
        dst[i] = row;
        if (row >= 0 && a.src_map && piece == 0) a.src_map[row] = t0 * a.topk + i;
    });
    if (!BULK)
        for (int i = tid; i < t1 - t0; i += kIdxThreads) src[i] = t0 + i;
    __syncthreads();
    if (last) {                                      // every copy has been counted here, but for its own
        for (int i = tid; i < own; i += kIdxThreads)
            if (own_key[i] >= 0) atomicAdd(&hist[own_key[i]], 1);
        __syncthreads();
        if (tid < a.N && tid != a.rank && hist[tid] != runs.total[tid]) bad = VP_ST_PACK_MISMATCH;
        const int any = __syncthreads_or(bad);
        if (tid == 0) *a.status = st | (any ? VP_ST_PACK_MISMATCH : 0) | (over ? VP_ST_PACK_CAPACITY : 0);
    }
    if (BULK) {
        if (tid < kOwnWarps * 32 && !(over ? ring.drain() : ring.finish(a.topk, dst, [&](int i) { return t0 + i; })) && (tid & 31) == 0)
            atomicOr(a.status, VP_ST_INTERNAL_TIMEOUT);
        return;
    }
    if (over) return;
    move_rows<V>(rows, staged, a.row.d, t1 - t0, a.topk, src, dst, v_lo, v_hi);
}

// ---- chunked form -----------------------------------------------------------------------------------------------

// CTA b < n_chunks counts chunk b; the last CTA builds the run table: the two need nothing from each other.
__global__ void __launch_bounds__(kIdxThreads) pack_count_kernel(PackArgs a, PackWs w, int chunk, int n_chunks) {
    extern __shared__ int sm[];
    const int tid = threadIdx.x, N = a.N;
    grid_wait();
    if ((int)blockIdx.x == n_chunks) {
        int bad = 0;
        const Step first = pack_step(a, tid < a.k_max ? raw_step(a, tid) : RawStep{-1, 0, 0}, bad);
        const int K = steps_in_use(a);
        const int st = pack_runs(a, K, first, bad, Runs{w.start, w.row, w.ptr, w.total}, sm, sm + N);
        if (tid == 0) {
            const bool over = a.send_off[(size_t)K * N + a.rank] > a.capacity;
            w.flags[0] = over;
            w.flags[1] = st | (over ? VP_ST_PACK_CAPACITY : 0);
        }
        return;
    }
    const ChunkRange mine = chunk_range(blockIdx.x, chunk, (long long)a.T * a.topk);
    for (int j = tid; j < N; j += kIdxThreads) sm[j] = 0;
    __syncthreads();
    int bad = 0;
#pragma unroll 4
    for (long long e = mine.lo + tid; e < mine.hi; e += kIdxThreads) {
        const int j = dest_of(a.idx[e], a, bad);
        if (j >= 0) atomicAdd(&sm[j], 1);
    }
    bad = __syncthreads_or(bad);
    for (int j = tid; j < N; j += kIdxThreads) w.hist[(size_t)blockIdx.x * N + j] = sm[j];
    if (tid == 0) w.bad[blockIdx.x] = bad ? VP_ST_PACK_MISMATCH : 0;
}

// CTA b maps chunk b, every warp a contiguous slice of it; the last CTA, whose base and own counts are all counts, checks
// them against the plan and writes the status.  The routing is read before the wait for the count kernel: that kernel has
// started, so whatever wrote the routing has finished.
constexpr int kMapRuns = 2048;                       // runs whose table is copied to shared memory
__host__ __device__ inline int pack_map_ints(int N, int k_max) { return N * (kIdxWarps + 1) + 2 * N + 1 + 2 * (k_max < kMapRuns ? k_max : kMapRuns); }

__global__ void __launch_bounds__(kIdxThreads) pack_map_kernel(PackArgs a, PackWs w, int chunk) {
    extern __shared__ int sm[];                      // [N] base, [kIdxWarps][N] next position of every warp's slice, run table
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, N = a.N;
    int* const base = sm;
    int* const next = sm + N + warp * N;
    for (int j = tid; j < N * (kIdxWarps + 1); j += kIdxThreads) sm[j] = 0;
    __syncthreads();
    const ChunkRange mine = chunk_range(blockIdx.x, chunk, (long long)a.T * a.topk);
    const long long s0 = min(mine.lo + (long long)warp * (chunk / kIdxWarps), mine.hi), s1 = min(s0 + chunk / kIdxWarps, mine.hi);
    int ignore = 0;
    const long long own0 = s0 + lane;
    const int dest0 = own0 < s1 ? dest_of(a.idx[own0], a, ignore) : -1;
    for (long long e = own0; e < s1; e += 32) {
        const int j = e == own0 ? dest0 : dest_of(a.idx[e], a, ignore);
        if (j >= 0) atomicAdd(&next[j], 1);
    }
    grid_wait();
#pragma unroll 8
    for (int i = tid; i < (int)blockIdx.x * N; i += kIdxThreads) {
        const int v = w.hist[i];
        if (v) atomicAdd(&base[i % N], v);
    }
    const bool over = w.flags[0] != 0;
    const Runs runs = runs_to_shared(Runs{w.start, w.row, w.ptr, w.total}, N, kMapRuns, sm + N * (kIdxWarps + 1));
    __syncthreads();
    for (int j = tid; j < N; j += kIdxThreads) {     // exclusive prefix over the warps
        base[j] = slices_prefix(sm + N + j, N, base[j]);     // copies up to the end of this chunk
    }
    __syncthreads();
    if (blockIdx.x == gridDim.x - 1) {
        int bad = w.flags[1];
        for (int j = tid; j < N; j += kIdxThreads)
            if (j != a.rank && base[j] != runs.total[j]) bad |= VP_ST_PACK_MISMATCH;
        for (int b = tid; b < (int)gridDim.x; b += kIdxThreads) bad |= w.bad[b];
        const int mismatch = __syncthreads_or(bad & VP_ST_PACK_MISMATCH);
        if (tid == 0) *a.status = (bad & VP_ST_PACK_CAPACITY) | (mismatch ? VP_ST_PACK_MISMATCH : 0);
    }
    warp_positions(s0, s1, next, [&](long long e) { return e == own0 ? dest0 : dest_of(a.idx[e], a, ignore); },
                   [&](long long e, int j, int p) {
                       const int row = p >= 0 && !over ? run_lookup(runs, j, p) : -1;
                       w.dst_row[e] = row;
                       if (row >= 0 && a.src_map) a.src_map[row] = (int)e;
                   });
}

}  // namespace

extern "C" size_t vp_pack_workspace_bytes(int N, int T, int topk, int k_max) {
    if (N <= 0 || N > VP_MAX_N || T <= 0 || topk <= 0 || k_max <= 0) return 0;
    return carve(nullptr, N, T, topk, k_max).bytes;
}

extern "C" int vp_pack(const int32_t* n_steps_b, const int16_t* lane_dst_b, const int64_t* lane_bytes_b,
                       const int64_t* send_off_b, int N, int rank, int k_max, const int32_t* expert_idx, int T,
                       int topk, int experts_per_rank, const void* rows, int64_t row_bytes, void* staged,
                       int64_t staged_capacity_bytes, int32_t* src_map, int32_t* status, void* workspace,
                       size_t workspace_bytes, void* cuda_stream) {
    if (!n_steps_b || !lane_dst_b || !lane_bytes_b || !send_off_b || !expert_idx || !rows || !staged || !status)
        return VP_E_BAD_ARG;
    if (N <= 0 || N > VP_MAX_N || rank < 0 || rank >= N || k_max <= 0 || T <= 0 || topk <= 0 || experts_per_rank <= 0 ||
        row_bytes <= 0 || staged_capacity_bytes < 0)
        return VP_E_BAD_ARG;
    if (staged_capacity_bytes / row_bytes >= ((int64_t)1 << 31) || (long long)T * topk >= ((long long)1 << 31))
        return VP_E_UNSUPPORTED;
    if (!workspace || ((uintptr_t)workspace & 255) || workspace_bytes < vp_pack_workspace_bytes(N, T, topk, k_max))
        return VP_E_WORKSPACE;
    cudaStream_t stream = (cudaStream_t)cuda_stream;
    const long long E = (long long)T * topk;
    const PackArgs a{n_steps_b, lane_dst_b, lane_bytes_b, send_off_b, N, rank, k_max, T, topk, small_div(experts_per_rank),
                     expert_idx, row_div(row_bytes), staged_capacity_bytes, src_map, status};
    const int sms = sm_count_of_device();
    if (!sms) return VP_E_CUDA;
    if (E <= kSmallItems && k_max <= kSmallSteps && row_bytes <= kSmallRow) {
        const int width = copy_width(rows, staged, row_bytes);
        const SmallLaunch z = small_launch(T, sms, topk, row_bytes, width, kMinOwnBulk, [&](int own) { return pack_small_layout(N, k_max, own * topk).ints; });
        if (z.own <= kSmallOwn) {
            const char* from = (const char*)rows;
            vp_prof_mark(2, 0, stream);
            const auto go = [&](auto fn) { return launch_wide(fn, z.grid, z.smem, stream, a, from, (char*)staged, z); };
            const cudaError_t e = z.bulk ? go(pack_small_kernel<uint4, true>) : width == 16 ? go(pack_small_kernel<uint4, false>)
                                : width == 4 ? go(pack_small_kernel<uint32_t, false>) : go(pack_small_kernel<uint8_t, false>);
            vp_prof_mark(2, 1, stream);
            return e == cudaSuccess ? VP_OK : VP_E_CUDA;
        }
    }
    const PackWs w = carve(workspace, N, T, topk, k_max);
    const int chunk = chunk_items(E, N), n_chunks = chunks_of((unsigned)E, chunk);
    vp_prof_mark(1, 0, stream);
    cudaError_t e = launch_after(pack_count_kernel, n_chunks + 1, kIdxThreads, (size_t)(N + runs_scratch_ints(N)) * 4, stream, a, w, chunk, n_chunks);
    if (e == cudaSuccess) e = launch_after(pack_map_kernel, n_chunks, kIdxThreads, (size_t)pack_map_ints(N, k_max) * 4, stream, a, w, chunk);
    vp_prof_mark(1, 1, stream);
    if (e != cudaSuccess) return VP_E_CUDA;
    vp_prof_mark(2, 0, stream);
    const int rc = launch_row_copy(rows, staged, w.dst_row, w.flags, T, topk, false, false, row_bytes, status, stream);
    vp_prof_mark(2, 1, stream);
    return rc;
}

// ---- vp_pack_static: the pack with its scratch built into the library ---------------------------------
//
// Some callers of the pack have no way to obtain device scratch at the moment they call it: they sit inside
// a serving engine's steady-state step, are handed only the input and output buffers, hold no allocator of
// their own, and must not call cudaMalloc there (it synchronises the whole device, it can fail under the
// engine's memory cap, and the engine accounts for every byte itself).  For them the library keeps one
// fixed block of device memory, reserved when the library is loaded on a GPU and held until the process
// exits, and uses it in place of the caller's workspace.
//
// In host code `g_pack_static_scratch` is only a handle for the device array; its device address has to be
// asked for with cudaGetSymbolAddress, once per device, with that device current.
static __device__ __align__(256) unsigned char g_pack_static_scratch[VP_PACK_STATIC_SCRATCH_BYTES];

namespace {
constexpr int kMaxDevices = 64;
void* g_static_scratch_addr[kMaxDevices] = {nullptr};

// Device address of the built-in scratch on the current device (looked up on first use).
int static_scratch_address(void** out) {
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return VP_E_CUDA;
    void* p = __atomic_load_n(&g_static_scratch_addr[dev], __ATOMIC_ACQUIRE);
    if (!p) {
        if (cudaGetSymbolAddress(&p, g_pack_static_scratch) != cudaSuccess || !p) return VP_E_CUDA;
        __atomic_store_n(&g_static_scratch_addr[dev], p, __ATOMIC_RELEASE);
    }
    *out = p;
    return VP_OK;
}
}  // namespace

extern "C" int vp_pack_static(const int32_t* n_steps_b, const int16_t* lane_dst_b, const int64_t* lane_bytes_b,
                              const int64_t* send_off_b, int N, int rank, int k_max, const int32_t* expert_idx, int T,
                              int topk, int experts_per_rank, const void* rows, int64_t row_bytes, void* staged,
                              int64_t staged_capacity_bytes, int32_t* src_map, int32_t* status, void* cuda_stream) {
    if (N <= 0 || N > VP_MAX_N || T <= 0 || topk <= 0 || k_max <= 0) return VP_E_BAD_ARG;
    // the problem must fit the built-in block; nothing is launched otherwise
    const size_t need = vp_pack_workspace_bytes(N, T, topk, k_max);
    if (need == 0 || need > (size_t)VP_PACK_STATIC_SCRATCH_BYTES) return VP_E_WORKSPACE;
    void* scratch = nullptr;
    const int rc = static_scratch_address(&scratch);
    if (rc != VP_OK) return rc;
    // vp_pack writes every scratch word before it reads it, so whatever the previous call left in the block does not matter
    return vp_pack(n_steps_b, lane_dst_b, lane_bytes_b, send_off_b, N, rank, k_max, expert_idx, T, topk,
                   experts_per_rank, rows, row_bytes, staged, staged_capacity_bytes, src_map, status, scratch,
                   (size_t)VP_PACK_STATIC_SCRATCH_BYTES, cuda_stream);
}
