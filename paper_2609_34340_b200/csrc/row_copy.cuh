// Row copy shared by the pack and the unpack directions: every source row is read once and written to each of its
// destination rows.  The map is either map[row * fanout + slot] = destination row, or (gather, fan-out 1) map[i] = source
// row of destination row i; -1 = none.  Rows of at least 2 KB that are 16-byte aligned travel global -> shared -> global as
// bulk asynchronous copies (TMA): one warp per CTA drives a ring of shared-memory stages, an mbarrier per stage signals the
// load, the stores of a source row form one bulk group whose read completion frees the stage, and the mbarrier wait is
// bounded.  Other rows take a plain vector-load kernel.  Included by the translation units that launch it.
#pragma once
#include <cuda_runtime.h>

#include "bulk_copy.cuh"
#include "route_index.cuh"
#include "vp_internal.h"

namespace {

constexpr int kPiece = 16384;              // bytes per bulk transfer (rows longer than this are split)
constexpr int kStages = 6;
constexpr int kMinBulkRow = 2048;          // shorter rows use the plain-load kernel
constexpr unsigned kSpinLimit = 1u << 22;  // bounded mbarrier wait

struct RowCopy {
    const char* rows;
    char* out;
    const int32_t* map;
    const int32_t* flags;      // device: [0] != 0 turns the copy into a no-op; [2] = rows in use when `bounded`
    int n, fanout, gather, bounded;
    long long row_bytes;
    int pieces, stage_bytes;   // bulk form: pieces per row, ring stage
    int32_t* status;
};

// One warp per CTA.  A "unit" is one piece (<= kPiece bytes) of one source row.  Rows are dealt to the CTAs round robin (with
// a contiguous range each the copy is 10 % slower).  Unit m is loaded into stage m % S, S / 2 units ahead of its stores.
//
// The map entries of the CTA's next 32 / fan-out rows are fetched by one load while the rows before are in flight.  (With one fetch per
// unit each unit waited for a trip to L2: 0.85 us a unit and CTA whatever its size, so rows of 4 to 8 KB reached half of
// the bandwidth with two CTAs per SM.)  Stores carry no L2 policy: marking them evict-first cost 10 % at fan-out 1
// (32,768 rows of 14,336 B: 157 -> 142 us) and at 4 KB rows (214 -> 195 us), and changed nothing elsewhere.
__global__ void __launch_bounds__(32) row_copy_bulk_kernel(RowCopy c) {
    constexpr int S = kStages, kLook = S / 2;
    extern __shared__ __align__(128) unsigned char ring[];
    __shared__ __align__(8) unsigned long long bars[S];
    __shared__ int32_t sdst[S][32];                  // destination row of this lane's slot, per unit in flight
    const int lane = threadIdx.x;
    if (lane == 0) {
        for (int s = 0; s < S; s++) mbar_init(smem_u32(&bars[s]), 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncwarp();
    grid_wait();
    if (c.flags[0]) return;
    const int n = c.bounded ? min(c.n, c.flags[2]) : c.n;
    const int F = c.fanout, pieces = c.pieces;
    const bool wide = F > 32;                        // destinations of a row are then handled 32 slots at a time
    const int batch = wide ? 1 : 32 / F;             // rows whose map entries are fetched together
    const int mine = n > (int)blockIdx.x ? (n - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;   // this CTA's rows
    unsigned phase = 0;                              // parity per stage (bit s)
    unsigned loaded = 0;                             // stage holds a load that was issued (bit s)
    bool failed = false;
    const int f_row = wide ? 0 : lane / F, f_slot = wide ? 0 : lane - f_row * F;
    auto fetch = [&](int q) {                        // map entries of rows q .. q + batch - 1: lane = row x fan-out + slot
        const long long r = (long long)blockIdx.x + (long long)(q + f_row) * gridDim.x;
        return !wide && f_row < batch && r < n ? c.map[r * F + f_slot] : -1;
    };
    int cur = -1, nxt = fetch(0);
    // next load (row, place in its batch, piece) and next store (row, piece); ls, ss: ring stages
    int lr = 0, lb = 0, lp = 0, ls = 0, sr = 0, sp = 0, ss = 0;
    const long long units = (long long)mine * pieces;
    for (long long it = 0; it < units + kLook && !failed; it++) {
        if (it < units) {                            // ---- issue the load of unit `it`
            if (lb == 0 && lp == 0) { cur = nxt; nxt = fetch(lr + batch); }
            const long long r = (long long)blockIdx.x + (long long)lr * gridDim.x;
            int d = wide ? -1 : __shfl_sync(0xffffffffu, cur, min(lb * F + lane, 31));
            if (lane >= F) d = -1;
            bool any;
            long long src = r;
            if (wide) {
                any = false;
                for (int f = lane; f < F; f += 32) any |= c.map[r * F + f] >= 0;
                any = __any_sync(0xffffffffu, any);
            } else {
                any = __any_sync(0xffffffffu, d >= 0);
                if (c.gather) {
                    src = __shfl_sync(0xffffffffu, d, 0);
                    d = any && lane == 0 ? (int)r : -1;
                }
            }
            bulk_wait_read<S - kLook - 1>();         // every lane: its stores that last read this stage are done
            __syncwarp();
            sdst[ls][lane] = d;
            if (any && lane == 0) {
                const unsigned bytes = (unsigned)min((long long)kPiece, c.row_bytes - (long long)lp * kPiece);
                const unsigned bar = smem_u32(&bars[ls]);
                mbar_expect_tx(bar, bytes);
                bulk_load(smem_u32(ring + (size_t)ls * c.stage_bytes), c.rows + src * c.row_bytes + (long long)lp * kPiece, bytes, bar);
            }
            loaded = any ? (loaded | (1u << ls)) : (loaded & ~(1u << ls));
            ls = ls + 1 == S ? 0 : ls + 1;
            if (++lp == pieces) { lp = 0; lr++; if (++lb == batch) lb = 0; }
        }
        if (it >= kLook) {                           // ---- unit it - kLook: wait for its load, issue its stores
            if (loaded & (1u << ss)) {
                const unsigned bar = smem_u32(&bars[ss]);
                unsigned spins = 0;
                while (!mbar_try_wait(bar, (phase >> ss) & 1u)) {
                    if (++spins > kSpinLimit) { failed = true; break; }
                }
                failed = __any_sync(0xffffffffu, failed);
                phase ^= 1u << ss;
                if (!failed) {
                    loaded &= ~(1u << ss);           // this stage's load has landed
                    const unsigned bytes = (unsigned)min((long long)kPiece, c.row_bytes - (long long)sp * kPiece);
                    const unsigned from = smem_u32(ring + (size_t)ss * c.stage_bytes);
                    char* const to = c.out + (long long)sp * kPiece;
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                    if (!wide) {
                        const int d = sdst[ss][lane];
                        if (d >= 0) bulk_store(to + (long long)d * c.row_bytes, from, bytes);
                    } else {
                        const long long r = (long long)blockIdx.x + (long long)sr * gridDim.x;
                        for (int f = lane; f < F; f += 32) {
                            const int d = c.map[r * F + f];
                            if (d >= 0) bulk_store(to + (long long)d * c.row_bytes, from, bytes);
                        }
                    }
                }
            }
            bulk_commit();                           // one group per unit from every lane, empty or not
            ss = ss + 1 == S ? 0 : ss + 1;
            if (++sp == pieces) { sp = 0; sr++; }
        }
    }
    bulk_wait_read<0>();                             // stores must have read shared memory before it is released
    if (failed) {
        // Give-up path: no further loads were issued.  Loads already in flight must not land in shared memory that
        // the next CTA owns, so each is given one more bounded wait (the stage whose wait gave up had its parity
        // flipped: put it back first).  Then the status bit tells the caller that the output is incomplete.
        for (int s = 0; s < S; s++) {
            if (!(loaded & (1u << s))) continue;
            unsigned spins = 0;
            while (!mbar_try_wait(smem_u32(&bars[s]), ((phase >> s) & 1u) ^ 1u) && !mbar_try_wait(smem_u32(&bars[s]), (phase >> s) & 1u) &&
                   ++spins < (1u << 18)) {
            }
        }
        if (lane == 0) atomicOr(c.status, VP_ST_INTERNAL_TIMEOUT);
    }
}

// Plain-load path (short or unaligned rows): a warp takes 32 U vectors of one row at a time, all loads in flight before the
// first store (one load per lane at a time left a few KB in flight per SM: 4,100-byte rows ran at a third of the bandwidth).
// I numbers the vectors of a row: int up to kSmallRow bytes (8,192 x 8 rows of 4,100 B, fan-out 1, by 64-bit numbers: 105 -> 112 us).
template <typename V, typename I>
__global__ void __launch_bounds__(256) row_copy_plain_kernel(RowCopy c) {
    constexpr int U = PieceOf<V>::U;
    grid_wait();
    if (c.flags[0]) return;
    const int n = c.bounded ? min(c.n, c.flags[2]) : c.n, F = c.fanout;
    const int lane = threadIdx.x & 31;
    const long long warp = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const long long n_warps = ((long long)gridDim.x * blockDim.x) >> 5;
    const I vecs = (I)(c.row_bytes / (long long)sizeof(V)), pieces = (vecs + 32 * U - 1) / (32 * U);
    for (long long it = warp; it < (long long)n * pieces; it += n_warps) {
        const long long r = it / pieces;
        const I v0 = (I)(it - r * pieces) * 32 * U + lane;
        long long src = r;
        if (c.gather) {
            src = c.map[r];
            if (src < 0) continue;
        } else {
            bool any = false;
            for (int f = lane; f < F; f += 32) any |= c.map[r * F + f] >= 0;
            if (!__any_sync(0xffffffffu, any)) continue;
        }
        const V* from = (const V*)(c.rows + src * c.row_bytes);
        V x[U];
#pragma unroll
        for (int u = 0; u < U; u++)
            if (v0 + 32 * u < vecs) x[u] = __ldg(from + v0 + 32 * u);
        for (int f = 0; f < F; f++) {
            const long long d = c.gather ? r : (long long)c.map[r * F + f];
            if (d < 0) continue;
            V* to = (V*)(c.out + d * c.row_bytes);
#pragma unroll
            for (int u = 0; u < U; u++)
                if (v0 + 32 * u < vecs) to[v0 + 32 * u] = x[u];
        }
    }
}

// Widest vector (bytes) that source, destination and row size allow.
inline int copy_width(const void* rows, const void* out, long long row_bytes) {
    const uintptr_t mix = (uintptr_t)rows | (uintptr_t)out | (uintptr_t)row_bytes;
    return mix % 16 == 0 ? 16 : (mix % 4 == 0 ? 4 : 1);
}

// Enqueues the copy behind the kernel that wrote map and flags.  With `bounded`, only the first flags[2] rows (device) are
// in use.  Returns VP_OK or VP_E_CUDA.
inline int launch_row_copy(const void* rows, void* out, const int32_t* map, const int32_t* flags, int n, int fanout, bool gather,
                           bool bounded, long long row_bytes, int32_t* status, cudaStream_t stream) {
    static bool s_attr_set[64] = {false};       // per device, once: the bulk kernel's shared-memory limit
    int dev = 0;
    const int sms = sm_count_of_device();
    if (!sms || cudaGetDevice(&dev) != cudaSuccess) return VP_E_CUDA;
    RowCopy c;
    c.rows = (const char*)rows; c.out = (char*)out; c.map = map; c.flags = flags;
    c.n = n; c.fanout = fanout; c.gather = gather; c.bounded = bounded; c.row_bytes = row_bytes; c.status = status;
    c.pieces = 1; c.stage_bytes = 0;
    const int width = copy_width(rows, out, row_bytes);
    // Many short CTAs rather than one wave of long ones: 64 KB of stores per CTA in the plain form, 80 KB or two rows, whichever is
    // more, in the bulk form (14,336 B at fan-out 8: two rows, 229 KB).  The hardware hands out CTAs in order, so the rows in flight stay neighbours, and so do their destinations in every stream;
    // in one wave the CTAs drift apart and DRAM takes the stores at 5.0 TB/s instead of 5.7.  16,384 rows of 14,336 B,
    // fan-out 8: 371 us in one wave, 328 so; 8,192 rows of 4,096 B: 98 and 44 us; rows claimed in order from a counter by one
    // wave: 325 and 53 us.  (Where the rows in use are known on the device only, half of the buffer is expected.)
    const double row_stores = (double)row_bytes * fanout;
    const auto ctas = [&](double most_per_cta) {
        const double want = (double)n * row_stores / most_per_cta * (bounded ? 0.5 : 1.0);
        return want < sms ? (n < sms ? n : sms) : (want > 1e6 ? 1000000 : (int)want);
    };
    cudaError_t e;
    if (width == 16 && row_bytes >= kMinBulkRow) {
        if (dev < 0 || dev >= 64 || !s_attr_set[dev]) {
            if (cudaFuncSetAttribute(row_copy_bulk_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kStages * kPiece) != cudaSuccess)
                return VP_E_CUDA;
            if (dev >= 0 && dev < 64) s_attr_set[dev] = true;
        }
        c.pieces = (int)((row_bytes + kPiece - 1) / kPiece);
        c.stage_bytes = row_bytes < kPiece ? (int)((row_bytes + 127) & ~127ll) : kPiece;
        e = launch_after(row_copy_bulk_kernel, ctas(row_stores > 40960 ? 2 * row_stores : 81920), 32, (size_t)kStages * c.stage_bytes, stream, c);
    } else {
        const auto go = [&](auto fn) { return launch_after(fn, ctas(65536), 256, 0, stream, c); };
        if (width == 16) e = go(row_copy_plain_kernel<uint4, int>);                    // (short rows)
        else if (width == 4) e = row_bytes <= kSmallRow ? go(row_copy_plain_kernel<uint32_t, int>) : go(row_copy_plain_kernel<uint32_t, long long>);
        else e = row_bytes <= kSmallRow ? go(row_copy_plain_kernel<uint8_t, int>) : go(row_copy_plain_kernel<uint8_t, long long>);
    }
    return e == cudaSuccess ? VP_OK : VP_E_CUDA;
}

}  // namespace
