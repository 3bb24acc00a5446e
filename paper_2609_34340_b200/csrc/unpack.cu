// vp_unpack: the receive side of the buffer layout (Section 5: "the receive kernel unpacks them directly
// into the output layout").
//
// The receive buffer of a rank holds, step after step, the rows its one sender of that step delivered
// (at recv_off[k][rank]).  The output is expert-major: all rows of local expert 0, then 1, ...; inside an
// expert by source rank; inside a source in arrival order.  That is a stable sort of the received rows by
// the key (expert, source), done as a counting sort:
//   steps : receive row and sender of every step (only for plans too large for every count CTA to read)
//   count : key of every row (binary search of its step), per chunk of rows a histogram of keys
//   map   : stable position of every row among the rows of its key -> output row
//   copy  : the row copy shared with the pack (each received row read once, written once)
// vp_unpack_tokens, the return direction, sorts the routed copies by expert id the same way; a copy's position among the
// copies to its expert's rank is its position in that sender's stream, whose runs give the receive row.
// Up to kSmallItems rows (kSmallReturn copies) each call is one kernel (see route_index.cuh).
#include <cuda_runtime.h>

#include "row_copy.cuh"
#include "vp_internal.h"

namespace {

struct UnpackArgs {
    const int32_t* n_steps;
    const int16_t* lane_dst;
    const int64_t *lane_bytes, *recv_off;    // (lane_bytes: return direction only)
    int N, rank, k_max, epr, keys, items;    // items: capacity in rows, or routed copies
    SmallDiv by_epr;
    const int32_t* item_expert;              // local expert of each received row, or global expert of each routed copy
    RowDiv row;
    int64_t capacity_rows;
    int32_t *expert_off, *out_src, *out_map, *status;
};

struct UnpackWs {
    int32_t* flags;      // [0] abort, [1] status bits, [2] rows received
    int32_t* bad;        // [n_chunks] status bits of each chunk
    int32_t* step_row;   // [k_max + 1] first receive row of a step
    int32_t* step_peer;  // [k_max] its sender, -1 = none
    int32_t* hist;       // [n_chunks][keys]
    int32_t* item_key;   // [items] key of a received row or routed copy, -1 = none
    int32_t* map;        // [items] output row of a received row, or receive row of a routed copy; -1 = none
    int32_t *total, *ptr, *start, *row;      // (return direction) run table of the senders, see Runs
    size_t bytes;
};

UnpackWs carve(void* base, int N, int keys, long long items, int k_max) {
    UnpackWs w;
    size_t o = 0;
    auto take = [&](size_t n) { size_t at = o; o += vp_align256(n); return (int32_t*)((char*)base + at); };
    const size_t n_chunks = (size_t)chunks_of((unsigned)items, chunk_items(items, keys));
    w.flags = take(256);
    w.bad = take(n_chunks * 4);
    w.step_row = take((size_t)(k_max + 1) * 4);
    w.step_peer = take((size_t)k_max * 4);
    w.hist = take(n_chunks * keys * 4);
    w.item_key = take((size_t)items * 4);
    w.map = take((size_t)items * 4);
    w.total = take((size_t)N * 4);
    w.ptr = take((size_t)(N + 1) * 4);
    w.start = take((size_t)k_max * 4);
    w.row = take((size_t)k_max * 4);
    w.bytes = o;
    return w;
}

__device__ __forceinline__ int steps_in_use(const UnpackArgs& a) { return min(max(*a.n_steps, 0), a.k_max); }

// Rows this rank receives in K steps (0 when they exceed the buffer), with status bits.
__device__ __forceinline__ int rows_received(const UnpackArgs& a, int K, int& st) {
    int64_t odd;
    const int64_t rows = a.row.div(a.recv_off[(size_t)K * a.N + a.rank], odd);
    const bool over = rows > a.capacity_rows;
    st = (odd ? VP_ST_PACK_MISMATCH : 0) | (over ? VP_ST_PACK_CAPACITY : 0);
    return over ? 0 : (int)rows;
}

// Step k of the dispatch plan, apart from its sender: first receive row, or -1 - row if its bytes are not whole rows;
// `any` if it delivers something.
__device__ __forceinline__ int step_rows(const UnpackArgs& a, int k, bool& any) {
    const int64_t lo = a.recv_off[(size_t)k * a.N + a.rank], hi = a.recv_off[(size_t)(k + 1) * a.N + a.rank];
    int64_t odd_lo, odd_hi;
    const int row = (int)a.row.div(lo, odd_lo);
    a.row.div(hi, odd_hi);
    any = hi > lo;
    return any && (odd_lo || odd_hi) ? -1 - row : row;
}
// With its sender: a step whose bytes are not whole rows, or that has bytes and no sender, is left out (peer -1) and reported.
__device__ __forceinline__ int check_step(int row, bool any, int& peer, int& bad) {
    if (any && (peer < 0 || row < 0)) { peer = -1; bad = VP_ST_PACK_MISMATCH; }
    return row < 0 ? -1 - row : row;
}

// Keys of the received rows r .. r + n - 1 < R with the experts e[]: (local expert, sender of its step), -1 if either is missing.  The
// searches for the last step that starts at or before a row run side by side, without branches (one by one 700 cycles each).
template <int n>
__device__ __forceinline__ void row_keys_of(const UnpackArgs& a, int r, const int (&e)[n], int K, const int* step_row, const int* step_peer, int (&key)[n]) {
    int lo[n];
#pragma unroll
    for (int q = 0; q < n; q++) lo[q] = 0;
    for (int w = K > 1 ? 1 << (31 - __clz(K - 1)) : 0; w; w >>= 1) {
#pragma unroll
        for (int q = 0; q < n; q++) {
            const int mid = min(lo[q] + w, K - 1);
            lo[q] = step_row[mid] <= r + q ? mid : lo[q];
        }
    }
#pragma unroll
    for (int q = 0; q < n; q++) {
        const int src = K > 0 ? step_peer[lo[q]] : -1;
        key[q] = e[q] < 0 || e[q] >= a.epr || src < 0 ? -1 : e[q] * a.N + src;
    }
}

// Key of a routed copy: its expert id, -1 if it does not travel.
__device__ __forceinline__ int copy_key_of(const UnpackArgs& a, int e) {
    return e >= 0 && e < a.keys && a.by_epr.div(e) != a.rank ? e : -1;
}

// Run table of the return plan: bucket = sender, runs = its segments in the receive buffer.  peer(k) is the sender of step k;
// row0 is the first row of step threadIdx.x as return_row gives it.
__device__ __forceinline__ int return_row(const UnpackArgs& a, int64_t off) {
    int64_t odd;
    const int row = (int)a.row.div(off, odd);
    return odd ? -1 : row;
}
__device__ __forceinline__ int return_row(const UnpackArgs& a, int k) { return return_row(a, a.recv_off[(size_t)k * a.N + a.rank]); }
template <typename Peer>
__device__ __forceinline__ int return_runs(const UnpackArgs& a, int K, int row0, Peer peer, Runs out, int* cnt, int* scratch, bool cleared = false,
                                           bool report = true) {
    int bad = 0;
    const auto step = [&](int k, int at) {
        const int j = peer(k);
        if (j < 0) return Step{-1, 0, 0};
        int64_t odd;
        const int64_t rows = a.row.div(a.lane_bytes[(size_t)k * a.N + j], odd);
        if (odd || at < 0) { bad = VP_ST_PACK_MISMATCH; return Step{-1, 0, 0}; }   // left out
        return Step{rows > 0 ? j : -1, (int)rows, at};
    };
    const Step first = (int)threadIdx.x < K ? step(threadIdx.x, row0) : Step{-1, 0, 0};
    build_runs(K, a.N, first, [&](int k) { return step(k, return_row(a, k)); }, out, cnt, scratch, cleared);
    if (!report) return 0;
    return __syncthreads_or(bad) ? VP_ST_PACK_MISMATCH : 0;
}

// total[key] -> exclusive prefix over the keys in first[0 .. keys]; all threads.
__device__ __forceinline__ void scan_keys(const int* total, int* first, int keys, int* wsum) {
    int run = 0;
    for (int k0 = 0; k0 < keys; k0 += kIdxThreads) {
        const int k = k0 + threadIdx.x;
        int all;
        const int at = cta_exclusive_scan(k < keys ? total[k] : 0, wsum, all);
        if (k < keys) first[k] = run + at;
        run += all;
    }
    if (threadIdx.x == 0) first[keys] = run;
    __syncthreads();
}

// The same by one warp, of all[key] + next[key]; no barrier.
__device__ __forceinline__ void warp_scan_keys(const int* all, const int* next, int* first, int keys) {
    const int lane = threadIdx.x & 31;
    int run = 0;
#pragma unroll 4
    for (int k = lane; k - lane < keys; k += 32) {
        const int mine = k < keys ? all[k] + next[k] : 0;
        int incl = mine;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += t;
        }
        if (k < keys) first[k] = run + incl - mine;
        run += __shfl_sync(0xffffffffu, incl, 31);
    }
    if (lane == 0) first[keys] = run;
}

// ---- one launch -------------------------------------------------------------------------------------------------

struct UnpackSmall { int key, peer, step_row, all, next, first, wsum, cnt, total, ptr, start, row, src, dst, scratch, ints; };
__host__ __device__ inline UnpackSmall unpack_small_layout(int N, int keys, int k_max, int own, bool tokens) {
    UnpackSmall L;
    int o = 0;
    L.key = o;      o += (own + 3) & ~3;             // (read four at a time)
    L.peer = o;     o += k_max;
    L.step_row = o; o += tokens ? 0 : k_max + 1;
    L.all = o;      o += keys;
    L.next = o;     o += keys;
    L.first = o;    o += keys + 1;
    L.wsum = o;     o += tokens ? 0 : kIdxWarps + 1;
    L.cnt = o;      o += tokens ? N : 0;
    L.total = o;    o += tokens ? N : 0;
    L.ptr = o;      o += tokens ? N + 1 : 0;
    L.start = o;    o += tokens ? k_max : 0;
    L.row = o;      o += tokens ? k_max : 0;
    L.src = o;      o += own;
    L.dst = o;      o += own;
    L.scratch = o;  o += tokens ? runs_scratch_ints(N) : 0;
    L.ints = o;
    return L;
}

// Receive side of small calls.  Every CTA reads the plan and the keys of all received rows, counts them (all of them, and
// those before its own), and moves its own contiguous range of rows.  Bound by latency, then by HBM.  Replaces two memsets
// and six kernels.
template <typename V, bool BULK>
__global__ void __launch_bounds__(kIdxThreads, BULK ? 1 : 2)
unpack_small_kernel(UnpackArgs a, const char* __restrict__ recv, char* __restrict__ out, SmallLaunch z) {
    extern __shared__ __align__(128) int sm[];
    __shared__ __align__(8) unsigned long long bars[kOwnWarps * kOwnStages];
    const UnpackSmall L = unpack_small_layout(a.N, a.keys, a.k_max, z.own, false);
    const int pieces = z.pieces;
    int *const peer = sm + L.peer, *const step_row = sm + L.step_row, *const all = sm + L.all, *const next = sm + L.next;
    const int tid = threadIdx.x, n_cta = gridDim.x / pieces, c = blockIdx.x / pieces, piece = blockIdx.x - c * pieces;
    const int vecs = (int)(a.row.d / (int64_t)sizeof(V)), v_lo = (int)((long long)vecs * piece / pieces),
              v_hi = (int)((long long)vecs * (piece + 1) / pieces);
    for (int j = tid; j < a.keys; j += kIdxThreads) { all[j] = 0; next[j] = 0; }
    OwnRing ring;
    if (BULK && tid < kOwnWarps * 32) ring.init(z, recv, out, a.row.d, v_lo, v_hi, sm, bars);
    for (int k = tid; k < a.k_max; k += kIdxThreads) peer[k] = -1;
    __syncthreads();
    grid_wait();
    // what the index needs first is asked for at once, before K is known
    const uint4 cells = sender_cells(a.lane_dst, a.N, a.k_max);
    constexpr int kAhead = 4;                        // loads of rows' experts per thread: of one up to 2,048 rows, else of four
    const bool by4 = ((uintptr_t)a.item_expert & 15) == 0 && a.items > kAhead * kIdxThreads;
    const int ahead = by4 ? min(a.items / 4, kAhead * kIdxThreads) : min(a.items, kAhead * kIdxThreads);
    int4 expert[kAhead];
#pragma unroll
    for (int u = 0; u < kAhead; u++) {
        const int v = tid + u * kIdxThreads;
        expert[u] = make_int4(0, 0, 0, 0);
        if (v < ahead) {
            if (by4) expert[u] = __ldg((const int4*)a.item_expert + v);
            else expert[u].x = __ldg(a.item_expert + v);
        }
    }
    bool any0 = false;
    const int row0 = tid < a.k_max ? step_rows(a, tid, any0) : 0;
    const int K = steps_in_use(a);
    int st, bad = 0;
    const int R = rows_received(a, K, st);
    const int r0 = (int)((long long)R * c / n_cta), r1 = (int)((long long)R * (c + 1) / n_cta);
    find_senders(a.lane_dst, a.N, a.rank, 0, K, cells, peer);
    for (int k = tid; k < K; k += kIdxThreads) {
        bool any = any0;
        const int row = k == tid ? row0 : step_rows(a, k, any);
        int p = peer[k];
        step_row[k] = check_step(row, any, p, bad);
        peer[k] = p;
    }
    __syncthreads();
    int* const own_key = sm + L.key;
    const auto add = [&](int r, int key) {
        if (r >= r0 && r < r1) own_key[r - r0] = key;
        if (key < 0) bad = VP_ST_PACK_MISMATCH;
        else atomicAdd(&sm[(r < r0 ? L.next : L.all) + key], 1);
    };
    const auto count = [&](int r, int x) {
        const int e[1] = {x};
        int key[1];
        row_keys_of(a, r, e, K, step_row, peer, key);
        add(r, key[0]);
    };
#pragma unroll
    for (int u = 0; u < kAhead; u++) {
        const int v = tid + u * kIdxThreads;
        if (v >= ahead) break;
        if (!by4) {
            if (v < R) count(v, expert[u].x);
        } else if (4 * v < R) {
            const int e[4] = {expert[u].x, expert[u].y, expert[u].z, expert[u].w};
            int key[4];
            row_keys_of(a, 4 * v, e, K, step_row, peer, key);
#pragma unroll
            for (int q = 0; q < 4; q++)
                if (4 * v + q < R) add(4 * v + q, key[q]);
        }
    }
    for_each_item(a.item_expert, min(by4 ? 4 * ahead : ahead, R), R, count);
    if (BULK && tid < kOwnWarps * 32) ring.start(r1 - r0, [&](int i) { return r0 + i; });
    bad = __syncthreads_or(bad) ? VP_ST_PACK_MISMATCH : 0;
    for (int j = tid; j < a.keys; j += kIdxThreads) all[j] += next[j];     // (scan_keys reads what the thread wrote)
    int* const first = sm + L.first;
    scan_keys(all, first, a.keys, sm + L.wsum);
    if (blockIdx.x == 0) {
        for (int e = tid; e <= a.epr; e += kIdxThreads) a.expert_off[e] = first[e * a.N];
        if (tid == 0) *a.status = st | bad | (!(st & VP_ST_PACK_CAPACITY) && first[a.keys] != R ? VP_ST_PACK_MISMATCH : 0);
    }
    int *const src = sm + L.src, *const dst = sm + L.dst;
    own_positions(own_key, r1 - r0, next, [&](int i, int key, int p) {
        const int o = p >= 0 ? first[key] + p : -1;
        src[i] = o >= 0 ? r0 + i : -1;
        dst[i] = o;
        if (o >= 0 && piece == 0) {
            if (a.out_src) a.out_src[o] = key % a.N;
            if (a.out_map) a.out_map[o] = r0 + i;
        }
    });
    __syncthreads();
    if (BULK) {
        if (tid < kOwnWarps * 32 && !ring.finish(1, dst, [&](int i) { return r0 + i; }) && (tid & 31) == 0) atomicOr(a.status, VP_ST_INTERNAL_TIMEOUT);
        return;
    }
    move_rows<V>(recv, out, a.row.d, r1 - r0, 1, src, dst, v_lo, v_hi);
}

// Return direction of small calls, the same way: own range = output rows (routed copies).
template <typename V, bool BULK>
__global__ void __launch_bounds__(kIdxThreads, BULK ? 1 : 2)
tokens_small_kernel(UnpackArgs a, const char* __restrict__ recv, char* __restrict__ out, SmallLaunch z) {
    extern __shared__ __align__(128) int sm[];
    __shared__ __align__(8) unsigned long long bars[kOwnWarps * kOwnStages];
    const UnpackSmall L = unpack_small_layout(a.N, a.keys, a.k_max, z.own, true);
    const int pieces = z.pieces;
    int *const peer = sm + L.peer, *const all = sm + L.all, *const next = sm + L.next, *const first = sm + L.first;
    const int tid = threadIdx.x, n_cta = gridDim.x / pieces, c = blockIdx.x / pieces, piece = blockIdx.x - c * pieces;
    const int vecs = (int)(a.row.d / (int64_t)sizeof(V)), v_lo = (int)((long long)vecs * piece / pieces),
              v_hi = (int)((long long)vecs * (piece + 1) / pieces);
    for (int j = tid; j < a.keys; j += kIdxThreads) { all[j] = 0; next[j] = 0; }
    OwnRing ring;
    if (BULK && tid < kOwnWarps * 32) ring.init(z, recv, out, a.row.d, v_lo, v_hi, sm, bars);
    for (int k = tid; k < a.k_max; k += kIdxThreads) peer[k] = -1;
    clear_runs_scratch(a.N, sm + L.scratch);
    __syncthreads();
    grid_wait();
    // all that the index needs first is asked for at once, before K is known
    const uint4 cells = sender_cells(a.lane_dst, a.N, a.k_max);
    const int64_t off0 = tid < a.k_max ? a.recv_off[(size_t)tid * a.N + a.rank] : 0;
    const int K = steps_in_use(a);
    const int c0 = (int)((long long)a.items * c / n_cta), c1 = (int)((long long)a.items * (c + 1) / n_cta);
    int* const own_key = sm + L.key;
    for (int i = tid; i < c1 - c0; i += kIdxThreads) own_key[i] = copy_key_of(a, a.item_expert[c0 + i]);
    for_each_item(a.item_expert, 0, a.items, [&](int i, int e) {
        const int key = copy_key_of(a, e);
        if (key >= 0) atomicAdd(&sm[(i < c0 ? L.next : L.all) + key], 1);
    });
    const int64_t end = a.recv_off[(size_t)K * a.N + a.rank];
    find_senders(a.lane_dst, a.N, a.rank, 0, K, cells, peer);         // (ends with a barrier: the counts are complete, too)
    if (tid >= kIdxThreads - 32) warp_scan_keys(all, next, first, a.keys);   // (while the others fetch the steps' bytes)
    const int row0 = return_row(a, off0);
    const Runs runs{sm + L.start, sm + L.row, sm + L.ptr, sm + L.total};
    const int st = return_runs(a, K, row0, [&](int k) { return peer[k]; }, runs, sm + L.cnt, sm + L.scratch, true, blockIdx.x == 0);
    const bool over = end > a.capacity_rows * a.row.d;                // nothing is unpacked then
    if (blockIdx.x == 0) {                           // every sender's stream is used up exactly
        int bad = st;
        if (tid < a.N && tid != a.rank && first[(tid + 1) * a.epr] - first[tid * a.epr] != runs.total[tid]) bad = VP_ST_PACK_MISMATCH;
        bad = __syncthreads_or(bad) ? VP_ST_PACK_MISMATCH : 0;
        if (tid == 0) *a.status = over ? VP_ST_PACK_CAPACITY : bad;
    }
    int *const src = sm + L.src, *const dst = sm + L.dst;
    own_positions(own_key, c1 - c0, next, [&](int i, int key, int p) {
        int row = -1;
        if (p >= 0 && !over) {
            const int j = a.by_epr.div(key);
            row = run_lookup(runs, j, first[key] + p - first[j * a.epr]);      // position in sender j's stream
        }
        src[i] = row;
        dst[i] = c0 + i;
        if (a.out_map && piece == 0) a.out_map[c0 + i] = row;
    });
    __syncthreads();
    if (BULK) {
        if (tid < kOwnWarps * 32) {
            const auto from = [&](int i) { return src[i]; };
            ring.start(c1 - c0, from);
            if (!ring.finish(1, dst, from) && (tid & 31) == 0) atomicOr(a.status, VP_ST_INTERNAL_TIMEOUT);
        }
        return;
    }
    move_rows<V>(recv, out, a.row.d, c1 - c0, 1, src, dst, v_lo, v_hi);
}

// ---- chunked form -----------------------------------------------------------------------------------------------

// A count CTA reads the plan's lane_dst itself up to this many cells (64 KB, five 16-byte loads per thread for the 300 of
// 512 activations a 64-rank plan uses); larger plans have their steps resolved by steps_kernel first.  Unpack of 2,000 tokens x
// top-8, 4,096 B, in place | by steps_kernel, us: 16 ranks, 2,048 plan rows 50.1 | 50.2, 4,096 48.1 | 50.2; 64 ranks, 512 rows
// 56.3 | 54.3, 1,024 56.3 | 53.3; 256 ranks, 128 rows 21.5 | 19.5, 1,024 72.7 | 35.9.
constexpr int kInlineCells = 32768;
constexpr int kStepTile = 32;                        // steps per CTA of steps_kernel

__global__ void __launch_bounds__(kIdxThreads) unpack_steps_kernel(UnpackArgs a, UnpackWs w) {
    __shared__ int peer[kStepTile];
    grid_wait();
    const int K = steps_in_use(a);
    const int k0 = blockIdx.x * kStepTile, k1 = min(k0 + kStepTile, K);
    if (k0 >= k1) return;
    find_senders(a.lane_dst, a.N, a.rank, k0, k1, peer);
    if (k0 + (int)threadIdx.x < k1) w.step_peer[k0 + threadIdx.x] = peer[threadIdx.x];
}

// (Chunks in use are those that hold one of the R rows received; return direction: all of them.)
// steps: 0 the plan is read here, 1 its senders come from unpack_steps_kernel, 2 the same, and the tables stay in the
// workspace because they exceed shared memory (every CTA then writes the same values there).
__global__ void __launch_bounds__(kIdxThreads) unpack_count_kernel(UnpackArgs a, UnpackWs w, int chunk, int steps) {
    extern __shared__ int sm[];                      // [keys] histogram, [k_max] sender, [k_max] first row of every step
    int* const hist = sm;
    int* const peer = steps == 2 ? w.step_peer : sm + a.keys;
    int* const step_row = steps == 2 ? w.step_row : sm + a.keys + a.k_max;
    const int tid = threadIdx.x;
    for (int j = tid; j < a.keys; j += kIdxThreads) hist[j] = 0;
    if (steps == 0)
        for (int k = tid; k < a.k_max; k += kIdxThreads) peer[k] = -1;
    __syncthreads();
    grid_wait();
    // plan cells and the first row's expert, before it is known how many there are
    const uint4 cells = steps == 0 ? sender_cells(a.lane_dst, a.N, a.k_max) : make_uint4(0, 0, 0, 0);
    const long long own0 = (long long)blockIdx.x * chunk + tid;
    const int expert0 = own0 < a.items ? __ldg(a.item_expert + own0) : 0;
    bool any0 = false;
    const int row0 = tid < a.k_max ? step_rows(a, tid, any0) : 0;
    const int K = steps_in_use(a);
    int st, bad = 0;
    const int R = rows_received(a, K, st);
    if (blockIdx.x == 0 && tid == 0) { w.flags[0] = (st & VP_ST_PACK_CAPACITY) != 0; w.flags[1] = st; w.flags[2] = R; }
    if ((int)blockIdx.x > 0 && (int)blockIdx.x >= chunks_of(R, chunk)) return;     // (CTA 0 always reports on the plan)
    if (steps == 0) find_senders(a.lane_dst, a.N, a.rank, 0, K, cells, peer);
    for (int k = tid; k < K; k += kIdxThreads) {
        bool any = any0;
        const int row = k == tid ? row0 : step_rows(a, k, any);
        int p = steps == 0 ? peer[k] : w.step_peer[k];
        step_row[k] = check_step(row, any, p, bad);
        peer[k] = p;
    }
    __syncthreads();
    const ChunkRange mine = chunk_range(blockIdx.x, chunk, R);
    for (long long r = mine.lo + tid; r < mine.hi; r += kIdxThreads) {
        const int e[1] = {r == own0 ? expert0 : a.item_expert[r]};
        int keys[1];
        row_keys_of(a, (int)r, e, K, step_row, peer, keys);
        const int key = keys[0];
        w.item_key[r] = key;
        if (key >= 0) atomicAdd(&hist[key], 1);
        else bad = VP_ST_PACK_MISMATCH;
    }
    bad = __syncthreads_or(bad);
    for (int j = tid; j < a.keys; j += kIdxThreads) w.hist[(size_t)blockIdx.x * a.keys + j] = hist[j];
    if (tid == 0) w.bad[blockIdx.x] = bad ? VP_ST_PACK_MISMATCH : 0;
}

__global__ void __launch_bounds__(kIdxThreads) tokens_count_kernel(UnpackArgs a, UnpackWs w, int chunk, int n_chunks, int inline_steps) {
    extern __shared__ int sm[];
    const int tid = threadIdx.x;
    grid_wait();
    if ((int)blockIdx.x == n_chunks) {               // the senders' run table
        int *const cnt = sm, *const scratch = sm + a.N, *const peer = scratch + runs_scratch_ints(a.N);
        const int row0 = tid < a.k_max ? return_row(a, (int)tid) : 0;
        const int K = steps_in_use(a);
        if (inline_steps) find_senders(a.lane_dst, a.N, a.rank, 0, K, peer);
        const int st = return_runs(a, K, row0, [&](int k) { return inline_steps ? peer[k] : w.step_peer[k]; },
                                   Runs{w.start, w.row, w.ptr, w.total}, cnt, scratch);
        if (tid == 0) {
            const bool over = a.recv_off[(size_t)K * a.N + a.rank] > a.capacity_rows * a.row.d;
            w.flags[0] = over;
            w.flags[1] = over ? VP_ST_PACK_CAPACITY : st;
        }
        return;
    }
    for (int j = tid; j < a.keys; j += kIdxThreads) sm[j] = 0;
    __syncthreads();
    const ChunkRange mine = chunk_range(blockIdx.x, chunk, a.items);
#pragma unroll 4
    for (long long i = mine.lo + tid; i < mine.hi; i += kIdxThreads) {
        const int key = copy_key_of(a, a.item_expert[i]);
        if (key >= 0) atomicAdd(&sm[key], 1);
    }
    __syncthreads();
    for (int j = tid; j < a.keys; j += kIdxThreads) w.hist[(size_t)blockIdx.x * a.keys + j] = sm[j];
}

// Map of one chunk: all counts, the counts before this chunk, their prefix over the keys, then stable positions, every warp
// a contiguous slice.  Shared memory: [keys] all, [keys] before, [keys + 1] first, wsum, [kIdxWarps][keys] slices, run table.
// The return direction counts its slices before the wait for the count kernel: that kernel has started, so whatever wrote the
// routing has finished.
constexpr int kMapRuns = 2048;                       // runs whose table is copied to shared memory
__host__ __device__ inline int map_ints(int keys) { return 3 * keys + 1 + kIdxWarps + 1 + kIdxWarps * keys; }
inline int map_smem_ints(int N, int keys, int k_max, bool tokens) {
    return map_ints(keys) + (tokens ? 2 * N + 1 + 2 * (k_max < kMapRuns ? k_max : kMapRuns) : 0);
}

template <bool TOKENS>
__global__ void __launch_bounds__(kIdxThreads) unpack_map_kernel(UnpackArgs a, UnpackWs w, int chunk) {
    extern __shared__ int sm[];
    const int keys = a.keys, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    int *const all = sm, *const before = all + keys, *const first = before + keys, *const wsum = first + keys + 1;
    int *const slices = wsum + kIdxWarps + 1, *const next = slices + warp * keys;
    for (int j = tid; j < 2 * keys; j += kIdxThreads) all[j] = 0;
    for (int j = tid; j < kIdxWarps * keys; j += kIdxThreads) slices[j] = 0;
    __syncthreads();
    auto key_of = [&](long long i) { return TOKENS ? copy_key_of(a, a.item_expert[i]) : w.item_key[i]; };
    long long s0, s1;
    const long long own0 = (long long)blockIdx.x * chunk + (long long)warp * (chunk / kIdxWarps) + lane;
    int key0 = -1;                                   // the slice's first 32 keys: asked for with the flags, and read twice
    auto count_slice = [&](int items) {
        const ChunkRange own = chunk_range(blockIdx.x, chunk, items);
        s0 = min(own.lo + (long long)warp * (chunk / kIdxWarps), own.hi);
        s1 = min(s0 + chunk / kIdxWarps, own.hi);
        for (long long i = s0 + lane; i < s1; i += 32) {
            const int key = i == own0 ? key0 : key_of(i);
            if (key >= 0) atomicAdd(&next[key], 1);
        }
    };
    if (TOKENS) {
        if (own0 < a.items) key0 = key_of(own0);
        count_slice(a.items);
    }
    grid_wait();
    if (!TOKENS && own0 < a.items) key0 = key_of(own0);      // (beyond the rows received: not used)
    const bool over = w.flags[0] != 0;
    const int items = TOKENS ? a.items : w.flags[2];
    const int n_chunks = chunks_of(items, chunk);
    if (!TOKENS && (int)blockIdx.x > 0 && (int)blockIdx.x >= n_chunks) return;
    if (!TOKENS) count_slice(items);
    // thread t adds up column t mod keys of every (kIdxThreads / keys)-th chunk (keys <= kIdxThreads), or columns t, t + kIdxThreads
    const int lanes = keys <= kIdxThreads ? kIdxThreads / keys : 1, mine = tid / min(keys, kIdxThreads);
    for (int key = tid - mine * keys; mine < lanes && key < keys; key += kIdxThreads) {
        int sum = 0, early = 0;
#pragma unroll 8
        for (int b = mine; b < n_chunks; b += lanes) {
            const int v = w.hist[(size_t)b * keys + key];
            sum += v;
            early += b < (int)blockIdx.x ? v : 0;
        }
        if (sum) atomicAdd(&all[key], sum);
        if (early) atomicAdd(&before[key], early);
    }
    Runs runs{w.start, w.row, w.ptr, w.total};
    if (TOKENS) runs = runs_to_shared(runs, a.N, kMapRuns, sm + map_ints(keys));
    __syncthreads();
    scan_keys(all, first, keys, wsum);
    if (blockIdx.x == 0) {
        int bad = 0;
        if (TOKENS) {                                // every sender's stream is used up exactly
            for (int j = tid; j < a.N; j += kIdxThreads)
                if (j != a.rank && first[(j + 1) * a.epr] - first[j * a.epr] != runs.total[j]) bad = VP_ST_PACK_MISMATCH;
        } else {
            for (int e = tid; e <= a.epr; e += kIdxThreads) a.expert_off[e] = first[e * a.N];
            for (int b = tid; b < (n_chunks > 1 ? n_chunks : 1); b += kIdxThreads) bad |= w.bad[b];
            if (!over && first[keys] != items) bad = VP_ST_PACK_MISMATCH;
        }
        bad = __syncthreads_or(bad) ? VP_ST_PACK_MISMATCH : 0;
        if (tid == 0) *a.status = w.flags[1] | (TOKENS && over ? 0 : bad);
    }
    for (int j = tid; j < keys; j += kIdxThreads) {  // start of every warp's slice: key, chunks before, warps before
        slices_prefix(slices + j, keys, first[j] + before[j]);
    }
    __syncthreads();
    warp_positions(s0, s1, next, [&](long long i) { return i == own0 ? key0 : key_of(i); }, [&](long long i, int key, int p) {
        if (TOKENS) {
            int row = -1;
            if (p >= 0 && !over) {
                const int j = a.by_epr.div(key);
                row = run_lookup(runs, j, p - first[j * a.epr]);
            }
            w.map[i] = row;
            if (a.out_map) a.out_map[i] = row;
        } else {
            w.map[i] = p;
            if (p >= 0) {
                if (a.out_src) a.out_src[p] = key % a.N;
                if (a.out_map) a.out_map[p] = (int)i;
            }
        }
    });
}

// Both calls once their arguments are checked.
template <bool TOKENS>
int unpack_launch(const UnpackArgs& a, const void* recv, void* out, void* workspace, cudaStream_t stream) {
    const int sms = sm_count_of_device();
    if (!sms) return VP_E_CUDA;
    const long long items = a.items;
    // (shared memory of unpack_count_kernel: histogram and both step tables)
    const bool steps_fit = ((long long)a.keys + 2ll * a.k_max) * 4 <= (long long)kSmemLimit;
    const bool inline_steps = (long long)a.k_max * a.N <= kInlineCells && steps_fit;
    cudaError_t e = cudaSuccess;
    if (items <= (TOKENS ? kSmallReturn : kSmallItems) && a.k_max <= kSmallSteps && inline_steps && a.row.d <= kSmallRow) {
        const int width = copy_width(recv, out, a.row.d);
        const SmallLaunch z = small_launch(a.items, sms, 1, a.row.d, width, TOKENS ? kMinReturnBulk : kMinOwnBulk, [&](int own) { return unpack_small_layout(a.N, a.keys, a.k_max, own, TOKENS).ints; });
        if (z.own <= kSmallOwn) {
            const char* from = (const char*)recv;
            vp_prof_mark(3, 0, stream);
            const auto go = [&](auto fn) { return launch_wide(fn, z.grid, z.smem, stream, a, from, (char*)out, z); };
            if constexpr (TOKENS)
                e = z.bulk ? go(tokens_small_kernel<uint4, true>) : width == 16 ? go(tokens_small_kernel<uint4, false>)
                  : width == 4 ? go(tokens_small_kernel<uint32_t, false>) : go(tokens_small_kernel<uint8_t, false>);
            else
                e = z.bulk ? go(unpack_small_kernel<uint4, true>) : width == 16 ? go(unpack_small_kernel<uint4, false>)
                  : width == 4 ? go(unpack_small_kernel<uint32_t, false>) : go(unpack_small_kernel<uint8_t, false>);
            vp_prof_mark(3, 1, stream);
            return e == cudaSuccess ? VP_OK : VP_E_CUDA;
        }
    }
    const UnpackWs w = carve(workspace, a.N, a.keys, items, a.k_max);
    const int chunk = chunk_items(items, a.keys), n_chunks = chunks_of((unsigned)items, chunk);
    if (!inline_steps) e = launch_after(unpack_steps_kernel, (a.k_max + kStepTile - 1) / kStepTile, kIdxThreads, 0, stream, a, w);
    if (e == cudaSuccess) {
        if constexpr (TOKENS) {
            const size_t ints_runs = (size_t)a.N + runs_scratch_ints(a.N) + (inline_steps ? a.k_max : 0);
            const size_t ints = ints_runs > (size_t)a.keys ? ints_runs : (size_t)a.keys;
            e = launch_wide(tokens_count_kernel, n_chunks + 1, ints * 4, stream, a, w, chunk, n_chunks, (int)inline_steps);
        } else {
            const size_t ints = (size_t)a.keys + (steps_fit ? 2 * (size_t)a.k_max : 0);
            e = launch_wide(unpack_count_kernel, n_chunks, ints * 4, stream, a, w, chunk, inline_steps ? 0 : (steps_fit ? 1 : 2));
        }
    }
    if (e == cudaSuccess) e = launch_wide(unpack_map_kernel<TOKENS>, n_chunks, (size_t)map_smem_ints(a.N, a.keys, a.k_max, TOKENS) * 4, stream, a, w, chunk);
    if (e != cudaSuccess) return VP_E_CUDA;
    vp_prof_mark(3, 0, stream);
    const int rc = launch_row_copy(recv, out, w.map, w.flags, a.items, 1, TOKENS, !TOKENS, a.row.d, a.status, stream);
    vp_prof_mark(3, 1, stream);
    return rc;
}

}  // namespace

extern "C" size_t vp_unpack_workspace_bytes(int N, int64_t capacity_rows, int experts_per_rank, int k_max) {
    if (N <= 0 || N > VP_MAX_N || capacity_rows <= 0 || experts_per_rank <= 0 || k_max <= 0) return 0;
    if ((long long)N * experts_per_rank > kMaxKeys || capacity_rows >= ((int64_t)1 << 31)) return 0;
    return carve(nullptr, N, N * experts_per_rank, capacity_rows, k_max).bytes;
}

extern "C" int vp_unpack(const int32_t* n_steps_b, const int16_t* lane_dst_b, const int64_t* recv_off_b, int N, int rank,
                         int k_max, const void* recv, int64_t row_bytes, int64_t capacity_rows, const int32_t* recv_expert,
                         int experts_per_rank, void* out, int32_t* expert_off, int32_t* out_src, int32_t* out_map,
                         int32_t* status, void* workspace, size_t workspace_bytes, void* cuda_stream) {
    if (!n_steps_b || !lane_dst_b || !recv_off_b || !recv || !recv_expert || !out || !expert_off || !status) return VP_E_BAD_ARG;
    if (N <= 0 || N > VP_MAX_N || rank < 0 || rank >= N || k_max <= 0 || row_bytes <= 0 || capacity_rows <= 0 ||
        experts_per_rank <= 0)
        return VP_E_BAD_ARG;
    if ((long long)N * experts_per_rank > kMaxKeys || capacity_rows >= ((int64_t)1 << 31)) return VP_E_UNSUPPORTED;
    if (!workspace || ((uintptr_t)workspace & 255) || workspace_bytes < vp_unpack_workspace_bytes(N, capacity_rows, experts_per_rank, k_max))
        return VP_E_WORKSPACE;
    const UnpackArgs a{n_steps_b, lane_dst_b, nullptr, recv_off_b, N, rank, k_max, experts_per_rank, N * experts_per_rank,
                       (int)capacity_rows, small_div(experts_per_rank), recv_expert, row_div(row_bytes), capacity_rows, expert_off, out_src, out_map, status};
    return unpack_launch<false>(a, recv, out, workspace, (cudaStream_t)cuda_stream);
}

// ---- return direction: receive buffer -> token layout ---------------------------------------------------

extern "C" size_t vp_unpack_tokens_workspace_bytes(int N, int T, int topk, int experts_per_rank, int64_t capacity_rows, int k_max) {
    if (N <= 0 || N > VP_MAX_N || T <= 0 || topk <= 0 || capacity_rows <= 0 || experts_per_rank <= 0 || k_max <= 0) return 0;
    if ((long long)N * experts_per_rank > kMaxKeys || capacity_rows >= ((int64_t)1 << 31) || (long long)T * topk >= ((long long)1 << 31)) return 0;
    return carve(nullptr, N, N * experts_per_rank, (long long)T * topk, k_max).bytes;
}

extern "C" int vp_unpack_tokens(const int32_t* n_steps_b, const int16_t* lane_dst_b, const int64_t* lane_bytes_b,
                                const int64_t* recv_off_b, int N, int rank, int k_max, const int32_t* expert_idx, int T, int topk,
                                int experts_per_rank, const void* recv, int64_t row_bytes, int64_t capacity_rows, void* out,
                                int32_t* out_map, int32_t* status, void* workspace, size_t workspace_bytes, void* cuda_stream) {
    if (!n_steps_b || !lane_dst_b || !lane_bytes_b || !recv_off_b || !expert_idx || !recv || !out || !status) return VP_E_BAD_ARG;
    if (N <= 0 || N > VP_MAX_N || rank < 0 || rank >= N || k_max <= 0 || T <= 0 || topk <= 0 || row_bytes <= 0 ||
        capacity_rows <= 0 || experts_per_rank <= 0)
        return VP_E_BAD_ARG;
    const size_t need = vp_unpack_tokens_workspace_bytes(N, T, topk, experts_per_rank, capacity_rows, k_max);
    if (!need) return VP_E_UNSUPPORTED;
    if (!workspace || ((uintptr_t)workspace & 255) || workspace_bytes < need) return VP_E_WORKSPACE;
    const UnpackArgs a{n_steps_b, lane_dst_b, lane_bytes_b, recv_off_b, N, rank, k_max, experts_per_rank, N * experts_per_rank,
                       T * topk, small_div(experts_per_rank), expert_idx, row_div(row_bytes), capacity_rows, nullptr, nullptr, out_map, status};
    return unpack_launch<true>(a, recv, out, workspace, (cudaStream_t)cuda_stream);
}
