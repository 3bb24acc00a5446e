// Host-buffer variants of the two entry points: copy in, run the device path, copy out.
#include <cuda_runtime.h>

#include "vp_internal.h"

namespace {

struct Carver {
    char* base;
    size_t off = 0;
    void* take(size_t bytes) {
        size_t at = off;
        off += vp_align256(bytes);
        return base ? base + at : nullptr;
    }
};

struct SchedBufs {
    int64_t *demand, *tau_in, *lane_bytes, *send_off, *recv_off, *tau_out;
    int32_t *n_steps, *chan_id, *status;
    int16_t* lane_dst;
    uint16_t* lane_inst;
    void* ws;
    size_t ws_bytes, total;
};

SchedBufs carve_sched(void* base, const vp_catalog* c, int B, const vp_sched_params* p) {
    vp_info I;
    vp_catalog_info(c, &I);
    const size_t N = (size_t)I.N, K = (size_t)p->k_max, b = (size_t)B;
    Carver cv{(char*)base};
    SchedBufs s;
    s.demand = (int64_t*)cv.take(b * N * N * 8);
    s.tau_in = (int64_t*)cv.take(b * 8);
    s.n_steps = (int32_t*)cv.take(b * 4);
    s.chan_id = (int32_t*)cv.take(b * K * 4);
    s.lane_dst = (int16_t*)cv.take(b * K * N * 2);
    s.lane_inst = (uint16_t*)cv.take(b * K * N * 2);
    s.lane_bytes = (int64_t*)cv.take(b * K * N * 8);
    s.send_off = (int64_t*)cv.take(b * (K + 1) * N * 8);
    s.recv_off = (int64_t*)cv.take(b * (K + 1) * N * 8);
    s.tau_out = (int64_t*)cv.take(b * 8);
    s.status = (int32_t*)cv.take(b * 4);
    s.ws_bytes = vp_schedule_workspace_bytes(c, B, p);
    s.ws = cv.take(s.ws_bytes);
    s.total = cv.off;
    return s;
}

#define VP_COPY(dst, src, bytes, kind)                                                        \
    do {                                                                                      \
        if ((bytes) && cudaMemcpyAsync((dst), (src), (bytes), (kind), stream) != cudaSuccess) \
            return VP_E_CUDA;                                                                 \
    } while (0)

// Makes a device current for the lifetime of a call and puts the caller's device back on every way out.
struct DeviceScope {
    int prev = -1;
    bool ok = true;
    explicit DeviceScope(int device) {
        cudaGetDevice(&prev);
        if (prev != device) ok = cudaSetDevice(device) == cudaSuccess;
    }
    ~DeviceScope() { if (prev >= 0) cudaSetDevice(prev); }
};

}  // namespace

extern "C" size_t vp_schedule_host_scratch_bytes(const vp_catalog* c, int B, const vp_sched_params* p) {
    if (!c || !p || B <= 0 || p->k_max <= 0) return 0;
    SchedBufs s = carve_sched(nullptr, c, B, p);
    return s.ws_bytes ? s.total : 0;
}

namespace {

// Copies of one chunk's results to host memory on `stream`.  With used_only the plan arrays come back only up to each
// matrix's n_steps, which must already be in host memory.
int copy_plan_out(const SchedBufs& s, size_t N, size_t K, size_t lo, size_t n, int32_t* n_steps, int32_t* chan_id,
                  int16_t* lane_dst, uint16_t* lane_inst, int64_t* lane_bytes, int64_t* send_off, int64_t* recv_off,
                  bool used_only, cudaStream_t stream) {
    if (!used_only) {
        VP_COPY(chan_id + lo * K, s.chan_id, n * K * 4, cudaMemcpyDeviceToHost);
        VP_COPY(lane_dst + lo * K * N, s.lane_dst, n * K * N * 2, cudaMemcpyDeviceToHost);
        VP_COPY(lane_inst + lo * K * N, s.lane_inst, n * K * N * 2, cudaMemcpyDeviceToHost);
        VP_COPY(lane_bytes + lo * K * N, s.lane_bytes, n * K * N * 8, cudaMemcpyDeviceToHost);
        VP_COPY(send_off + lo * (K + 1) * N, s.send_off, n * (K + 1) * N * 8, cudaMemcpyDeviceToHost);
        if (recv_off) VP_COPY(recv_off + lo * (K + 1) * N, s.recv_off, n * (K + 1) * N * 8, cudaMemcpyDeviceToHost);
        return VP_OK;
    }
    for (size_t m = 0; m < n; m++) {
        const size_t g = lo + m;
        const size_t k = n_steps[g] < 0 ? 0 : ((size_t)n_steps[g] > K ? K : (size_t)n_steps[g]);
        VP_COPY(chan_id + g * K, s.chan_id + m * K, k * 4, cudaMemcpyDeviceToHost);
        VP_COPY(lane_dst + g * K * N, s.lane_dst + m * K * N, k * N * 2, cudaMemcpyDeviceToHost);
        VP_COPY(lane_inst + g * K * N, s.lane_inst + m * K * N, k * N * 2, cudaMemcpyDeviceToHost);
        VP_COPY(lane_bytes + g * K * N, s.lane_bytes + m * K * N, k * N * 8, cudaMemcpyDeviceToHost);
        VP_COPY(send_off + g * (K + 1) * N, s.send_off + m * (K + 1) * N, (k + 1) * N * 8, cudaMemcpyDeviceToHost);
        if (recv_off) VP_COPY(recv_off + g * (K + 1) * N, s.recv_off + m * (K + 1) * N, (k + 1) * N * 8, cudaMemcpyDeviceToHost);
    }
    return VP_OK;
}

// Used plan rows straight into pinned host memory.  Per matrix six copies of a few KB to a few 100 KB each are needed, of lengths
// that only the device knows: as cudaMemcpyAsync calls they cost a wait for n_steps and 3 us of host time each (128 matrices of
// 64 ranks: 768 calls).  One kernel of posted 16-byte writes keeps PCIe as busy as the copy engine does.
struct UsedRows {
    const int32_t *n_steps, *status, *chan_id;
    const int16_t* lane_dst;
    const uint16_t* lane_inst;
    const int64_t *lane_bytes, *send_off, *recv_off, *tau;
    int32_t *h_n_steps, *h_status, *h_chan_id;               // device addresses of the host buffers, from the chunk's first matrix on
    int16_t* h_lane_dst;
    uint16_t* h_lane_inst;
    int64_t *h_lane_bytes, *h_send_off, *h_recv_off, *h_tau;
    int B, N, K;
};
constexpr int kUsedPieces = 4;                               // CTAs' units per matrix

template <typename V>
__device__ __forceinline__ void copy_units(void* dst, const void* src, size_t lo, size_t hi) {
    constexpr int T = 256;
    size_t e = lo + threadIdx.x;
    for (; e + 3 * T < hi; e += 4 * T) {                     // four loads in flight per thread
        const V a = ((const V*)src)[e], b = ((const V*)src)[e + T], c = ((const V*)src)[e + 2 * T], d = ((const V*)src)[e + 3 * T];
        ((V*)dst)[e] = a; ((V*)dst)[e + T] = b; ((V*)dst)[e + 2 * T] = c; ((V*)dst)[e + 3 * T] = d;
    }
    for (; e < hi; e += T) ((V*)dst)[e] = ((const V*)src)[e];
}
__device__ __forceinline__ void copy_part(void* dst, const void* src, size_t bytes, int piece) {
    const uintptr_t mix = (uintptr_t)dst | (uintptr_t)src | bytes;
    const size_t n = mix % 16 == 0 ? bytes / 16 : (mix % 4 == 0 ? bytes / 4 : bytes / 2);      // (every array's rows are whole 16-bit words)
    const size_t lo = n * piece / kUsedPieces, hi = n * (piece + 1) / kUsedPieces;
    if (mix % 16 == 0) copy_units<uint4>(dst, src, lo, hi);
    else if (mix % 4 == 0) copy_units<uint32_t>(dst, src, lo, hi);
    else copy_units<uint16_t>(dst, src, lo, hi);
}
__global__ void __launch_bounds__(256) copy_used_rows_kernel(UsedRows u) {
    const size_t N = (size_t)u.N, K = (size_t)u.K;
    for (int unit = blockIdx.x; unit < u.B * kUsedPieces; unit += gridDim.x) {
        const size_t m = (size_t)(unit / kUsedPieces);
        const int piece = unit % kUsedPieces, n = u.n_steps[m];
        const size_t k = n < 0 ? 0 : ((size_t)n > K ? K : (size_t)n);
        copy_part(u.h_lane_bytes + m * K * N, u.lane_bytes + m * K * N, k * N * 8, piece);
        copy_part(u.h_send_off + m * (K + 1) * N, u.send_off + m * (K + 1) * N, (k + 1) * N * 8, piece);
        if (u.h_recv_off) copy_part(u.h_recv_off + m * (K + 1) * N, u.recv_off + m * (K + 1) * N, (k + 1) * N * 8, piece);
        copy_part(u.h_lane_dst + m * K * N, u.lane_dst + m * K * N, k * N * 2, piece);
        copy_part(u.h_lane_inst + m * K * N, u.lane_inst + m * K * N, k * N * 2, piece);
        copy_part(u.h_chan_id + m * K, u.chan_id + m * K, k * 4, piece);
        if (piece == 0 && threadIdx.x == 0) {
            u.h_n_steps[m] = n;
            u.h_status[m] = u.status[m];
            if (u.h_tau) u.h_tau[m] = u.tau[m];
        }
    }
}

// Device address of `bytes` of page-locked host memory, or null if the device cannot write there.
template <typename T>
T* pinned_address(T* host, size_t bytes) {
    cudaPointerAttributes a, z;
    if (!host || !bytes) return nullptr;
    if (cudaPointerGetAttributes(&a, host) != cudaSuccess || cudaPointerGetAttributes(&z, (const char*)host + bytes - 1) != cudaSuccess) {
        cudaGetLastError();
        return nullptr;
    }
    if (a.type != cudaMemoryTypeHost || z.type != cudaMemoryTypeHost || !a.devicePointer || !z.devicePointer) return nullptr;
    return (const char*)z.devicePointer - (const char*)a.devicePointer == (ptrdiff_t)(bytes - 1) ? (T*)a.devicePointer : nullptr;
}

// Both host-buffer scheduler calls: copy in, run vp_schedule_batch, copy out.
int schedule_host(const vp_catalog* cc, const vp_sched_params* p, const int64_t* demand, const int64_t* tau_ns_in, int B,
                  int32_t* n_steps, int32_t* chan_id, int16_t* lane_dst, uint16_t* lane_inst, int64_t* lane_bytes,
                  int64_t* send_off, int64_t* recv_off, int64_t* tau_ns_out, int32_t* status, void* device_scratch,
                  size_t device_scratch_bytes, void* cuda_stream, bool used_only) {
    vp_catalog* c = const_cast<vp_catalog*>(cc);
    if (!c || !p || B <= 0 || p->k_max <= 0 || !demand || !n_steps || !chan_id || !lane_dst || !lane_inst || !lane_bytes ||
        !send_off || !status)
        return VP_E_BAD_ARG;
    if (!device_scratch || ((uintptr_t)device_scratch & 255)) return VP_E_WORKSPACE;
    SchedBufs whole = carve_sched(nullptr, c, B, p);
    if (!whole.ws_bytes) return VP_E_BAD_ARG;
    if (device_scratch_bytes < whole.total) return VP_E_WORKSPACE;
    cudaStream_t stream = (cudaStream_t)cuda_stream;
    const size_t N = (size_t)c->info.N, K = (size_t)p->k_max;
    DeviceScope scope(c->device);
    if (!scope.ok) return VP_E_CUDA;

    // Large batches are worked through in chunks, two of them in flight: while one chunk is decomposed on the caller's stream,
    // the results of the chunk before it travel to the host on a second stream.  About one matrix per SM each: a chunk lasts as
    // long as its longest matrix's chain however few it holds, so smaller batches are one chunk.  Two chunks' buffers must fit
    // the scratch of the whole batch.
    int n_chunks = 1, chunk = B;
    if (c->sm_count > 0 && B >= 2 * c->sm_count) {
        n_chunks = B / c->sm_count;
        chunk = (B + n_chunks - 1) / n_chunks;
        n_chunks = (B + chunk - 1) / chunk;
        const SchedBufs one = carve_sched(nullptr, c, chunk, p);
        if (!one.ws_bytes || 2 * one.total > device_scratch_bytes) { n_chunks = 1; chunk = B; }
    }
    // Used rows by a kernel where every host buffer is page-locked.  From 128 ranks on a matrix's rows are MBs: the copy engine
    // then needs few enough calls, and no SM has to have room beside the scheduler's CTAs.
    UsedRows host;
    bool by_kernel = false;
    if (used_only && N < 128) {
        const size_t b = (size_t)B;
        host.h_n_steps = pinned_address(n_steps, b * 4);
        host.h_status = pinned_address(status, b * 4);
        host.h_chan_id = pinned_address(chan_id, b * K * 4);
        host.h_lane_dst = pinned_address(lane_dst, b * K * N * 2);
        host.h_lane_inst = pinned_address(lane_inst, b * K * N * 2);
        host.h_lane_bytes = pinned_address(lane_bytes, b * K * N * 8);
        host.h_send_off = pinned_address(send_off, b * (K + 1) * N * 8);
        host.h_recv_off = pinned_address(recv_off, b * (K + 1) * N * 8);
        host.h_tau = pinned_address(tau_ns_out, b * 8);
        by_kernel = host.h_n_steps && host.h_status && host.h_chan_id && host.h_lane_dst && host.h_lane_inst && host.h_lane_bytes &&
                    host.h_send_off && (host.h_recv_off || !recv_off) && (host.h_tau || !tau_ns_out);
    }
    if (n_chunks > 1 && !c->host_pipe_ready) {
        // (highest priority: the copy kernel's CTAs go ahead of the next chunk's)
        int least = 0, greatest = 0;
        if (cudaDeviceGetStreamPriorityRange(&least, &greatest) != cudaSuccess ||
            cudaStreamCreateWithPriority(&c->copy_stream, cudaStreamNonBlocking, greatest) != cudaSuccess)
            return VP_E_CUDA;
        for (cudaEvent_t& e : c->host_ev)
            if (cudaEventCreateWithFlags(&e, cudaEventDisableTiming) != cudaSuccess) return VP_E_CUDA;
        c->host_pipe_ready = 1;
    }
    const size_t slot_bytes = n_chunks > 1 ? carve_sched(nullptr, c, chunk, p).total : 0;
    SchedBufs slot[2];
    slot[0] = carve_sched(device_scratch, c, chunk, p);
    slot[1] = n_chunks > 1 ? carve_sched((char*)device_scratch + slot_bytes, c, chunk, p) : slot[0];
    cudaStream_t copy = n_chunks > 1 ? c->copy_stream : stream;
    cudaEvent_t* done = c->host_ev;          // [0], [1]: chunk decomposed;  [2], [3]: its results copied out
    cudaEvent_t* copied = c->host_ev + 2;

    for (int i = 0; i <= n_chunks; i++) {
        if (i < n_chunks) {                  // ---- chunk i: copy in and decompose, on the caller's stream
            const SchedBufs& s = slot[i & 1];
            const size_t lo = (size_t)i * chunk, n = (size_t)(B - (int)lo < chunk ? B - (int)lo : chunk);
            if (n_chunks > 1 && i >= 2 && cudaStreamWaitEvent(stream, copied[i & 1], 0) != cudaSuccess) return VP_E_CUDA;
            VP_COPY(s.demand, demand + lo * N * N, n * N * N * 8, cudaMemcpyHostToDevice);
            if (tau_ns_in) VP_COPY(s.tau_in, tau_ns_in + lo, n * 8, cudaMemcpyHostToDevice);
            const int rc = vp_schedule_batch(c, p, s.demand, tau_ns_in ? s.tau_in : nullptr, (int)n, s.n_steps, s.chan_id,
                                             s.lane_dst, s.lane_inst, s.lane_bytes, s.send_off, recv_off ? s.recv_off : nullptr,
                                             tau_ns_out ? s.tau_out : nullptr, s.status, s.ws, s.ws_bytes, cuda_stream);
            if (rc) return rc;
            if (n_chunks > 1 && cudaEventRecord(done[i & 1], stream) != cudaSuccess) return VP_E_CUDA;
        }
        if (i >= 1 || n_chunks == 1) {       // ---- chunk i - 1 (the only chunk when there is one): results to the host
            const int j = n_chunks == 1 ? 0 : i - 1;
            if (n_chunks == 1 && i == 1) break;
            const SchedBufs& s = slot[j & 1];
            const size_t lo = (size_t)j * chunk, n = (size_t)(B - (int)lo < chunk ? B - (int)lo : chunk);
            if (n_chunks > 1 && cudaStreamWaitEvent(copy, done[j & 1], 0) != cudaSuccess) return VP_E_CUDA;
            if (by_kernel) {
                UsedRows u = host;
                u.n_steps = s.n_steps; u.status = s.status; u.chan_id = s.chan_id; u.lane_dst = s.lane_dst; u.lane_inst = s.lane_inst;
                u.lane_bytes = s.lane_bytes; u.send_off = s.send_off; u.recv_off = s.recv_off; u.tau = s.tau_out;
                u.h_n_steps += lo; u.h_status += lo; u.h_chan_id += lo * K; u.h_lane_dst += lo * K * N; u.h_lane_inst += lo * K * N;
                u.h_lane_bytes += lo * K * N; u.h_send_off += lo * (K + 1) * N;
                if (u.h_recv_off) u.h_recv_off += lo * (K + 1) * N;
                if (u.h_tau) u.h_tau += lo;
                u.B = (int)n; u.N = (int)N; u.K = (int)K;
                copy_used_rows_kernel<<<(int)(n * kUsedPieces < 256 ? n * kUsedPieces : 256), 256, 0, copy>>>(u);
                g_vp_launches++;
                if (cudaGetLastError() != cudaSuccess) return VP_E_CUDA;
            } else {
                cudaStream_t stream = copy;  // (VP_COPY issues on `stream`)
                VP_COPY(n_steps + lo, s.n_steps, n * 4, cudaMemcpyDeviceToHost);
                if (tau_ns_out) VP_COPY(tau_ns_out + lo, s.tau_out, n * 8, cudaMemcpyDeviceToHost);
                VP_COPY(status + lo, s.status, n * 4, cudaMemcpyDeviceToHost);
                if (used_only && cudaStreamSynchronize(copy) != cudaSuccess) return VP_E_CUDA;   // n_steps is needed on the host now
                const int rc = copy_plan_out(s, N, K, lo, n, n_steps, chan_id, lane_dst, lane_inst, lane_bytes, send_off, recv_off,
                                             used_only, copy);
                if (rc) return rc;
            }
            if (n_chunks > 1 && cudaEventRecord(copied[j & 1], copy) != cudaSuccess) return VP_E_CUDA;
        }
    }
    if (n_chunks > 1 && cudaStreamSynchronize(copy) != cudaSuccess) return VP_E_CUDA;
    if (cudaStreamSynchronize(stream) != cudaSuccess) return VP_E_CUDA;
    return VP_OK;
}

}  // namespace

extern "C" int vp_schedule_batch_host(const vp_catalog* c, const vp_sched_params* p, const int64_t* demand,
                                      const int64_t* tau_ns_in, int B, int32_t* n_steps, int32_t* chan_id,
                                      int16_t* lane_dst, uint16_t* lane_inst, int64_t* lane_bytes, int64_t* send_off,
                                      int64_t* recv_off, int64_t* tau_ns_out, int32_t* status, void* device_scratch,
                                      size_t device_scratch_bytes, void* cuda_stream) {
    return schedule_host(c, p, demand, tau_ns_in, B, n_steps, chan_id, lane_dst, lane_inst, lane_bytes, send_off, recv_off,
                         tau_ns_out, status, device_scratch, device_scratch_bytes, cuda_stream, false);
}

extern "C" int vp_schedule_batch_host_used(const vp_catalog* c, const vp_sched_params* p, const int64_t* demand,
                                           const int64_t* tau_ns_in, int B, int32_t* n_steps, int32_t* chan_id,
                                           int16_t* lane_dst, uint16_t* lane_inst, int64_t* lane_bytes, int64_t* send_off,
                                           int64_t* recv_off, int64_t* tau_ns_out, int32_t* status, void* device_scratch,
                                           size_t device_scratch_bytes, void* cuda_stream) {
    return schedule_host(c, p, demand, tau_ns_in, B, n_steps, chan_id, lane_dst, lane_inst, lane_bytes, send_off, recv_off,
                         tau_ns_out, status, device_scratch, device_scratch_bytes, cuda_stream, true);
}

namespace {

struct PackBufs {
    int32_t *n_steps, *idx, *src_map, *status;
    int16_t* lane_dst;
    int64_t *lane_bytes, *send_off;
    char *rows, *staged;
    void* ws;
    size_t ws_bytes, total;
};

PackBufs carve_pack(void* base, int N, int T, int topk, int k_max, int64_t row_bytes, int64_t cap) {
    Carver cv{(char*)base};
    PackBufs s;
    const size_t K = (size_t)k_max, n = (size_t)N;
    s.n_steps = (int32_t*)cv.take(4);
    s.lane_dst = (int16_t*)cv.take(K * n * 2);
    s.lane_bytes = (int64_t*)cv.take(K * n * 8);
    s.send_off = (int64_t*)cv.take((K + 1) * n * 8);
    s.idx = (int32_t*)cv.take((size_t)T * topk * 4);
    s.rows = (char*)cv.take((size_t)T * row_bytes);
    s.staged = (char*)cv.take((size_t)cap);
    s.src_map = (int32_t*)cv.take((size_t)(cap / row_bytes + 1) * 4);
    s.status = (int32_t*)cv.take(4);
    s.ws_bytes = vp_pack_workspace_bytes(N, T, topk, k_max);
    s.ws = cv.take(s.ws_bytes);
    s.total = cv.off;
    return s;
}

}  // namespace

extern "C" size_t vp_pack_host_scratch_bytes(int N, int T, int topk, int k_max, int64_t row_bytes, int64_t cap) {
    if (N <= 0 || T <= 0 || topk <= 0 || k_max <= 0 || row_bytes <= 0 || cap < 0) return 0;
    PackBufs s = carve_pack(nullptr, N, T, topk, k_max, row_bytes, cap);
    return s.ws_bytes ? s.total : 0;
}

extern "C" int vp_pack_host(const int32_t* n_steps_b, const int16_t* lane_dst_b, const int64_t* lane_bytes_b,
                            const int64_t* send_off_b, int N, int rank, int k_max, const int32_t* expert_idx, int T,
                            int topk, int experts_per_rank, const void* rows, int64_t row_bytes, void* staged,
                            int64_t cap, int32_t* src_map, int32_t* status, void* device_scratch,
                            size_t device_scratch_bytes, void* cuda_stream) {
    if (!n_steps_b || !lane_dst_b || !lane_bytes_b || !send_off_b || !expert_idx || !rows || !staged || !status)
        return VP_E_BAD_ARG;
    if (N <= 0 || T <= 0 || topk <= 0 || k_max <= 0 || row_bytes <= 0 || cap < 0) return VP_E_BAD_ARG;
    if (!device_scratch || ((uintptr_t)device_scratch & 255)) return VP_E_WORKSPACE;
    PackBufs s = carve_pack(device_scratch, N, T, topk, k_max, row_bytes, cap);
    if (!s.ws_bytes) return VP_E_BAD_ARG;
    if (device_scratch_bytes < s.total) return VP_E_WORKSPACE;
    cudaStream_t stream = (cudaStream_t)cuda_stream;
    const size_t K = (size_t)k_max, n = (size_t)N;
    VP_COPY(s.n_steps, n_steps_b, 4, cudaMemcpyHostToDevice);
    VP_COPY(s.lane_dst, lane_dst_b, K * n * 2, cudaMemcpyHostToDevice);
    VP_COPY(s.lane_bytes, lane_bytes_b, K * n * 8, cudaMemcpyHostToDevice);
    VP_COPY(s.send_off, send_off_b, (K + 1) * n * 8, cudaMemcpyHostToDevice);
    VP_COPY(s.idx, expert_idx, (size_t)T * topk * 4, cudaMemcpyHostToDevice);
    VP_COPY(s.rows, rows, (size_t)T * row_bytes, cudaMemcpyHostToDevice);
    int rc = vp_pack(s.n_steps, s.lane_dst, s.lane_bytes, s.send_off, N, rank, k_max, s.idx, T, topk, experts_per_rank,
                     s.rows, row_bytes, s.staged, cap, src_map ? s.src_map : nullptr, s.status, s.ws, s.ws_bytes,
                     cuda_stream);
    if (rc) return rc;
    VP_COPY(status, s.status, 4, cudaMemcpyDeviceToHost);
    if (cudaStreamSynchronize(stream) != cudaSuccess) return VP_E_CUDA;
    // only the bytes the plan covers come back: the send volume is send_off[n_steps][rank]
    const int K_used = *n_steps_b < 0 ? 0 : (*n_steps_b > k_max ? k_max : *n_steps_b);
    int64_t used = send_off_b[(size_t)K_used * n + rank];
    if (used < 0) used = 0;
    if (used > cap) used = cap;
    if (!(*status & VP_ST_PACK_CAPACITY)) {
        VP_COPY(staged, s.staged, (size_t)used, cudaMemcpyDeviceToHost);
        if (src_map) VP_COPY(src_map, s.src_map, (size_t)(used / row_bytes) * 4, cudaMemcpyDeviceToHost);
    }
    if (cudaStreamSynchronize(stream) != cudaSuccess) return VP_E_CUDA;
    return VP_OK;
}
