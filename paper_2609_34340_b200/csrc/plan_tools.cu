// Around the scheduler: the demand matrix from routing indices (its input side) and the modeled
// completion time of a plan, Eq. (2) (its quality measure).
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include "route_index.cuh"
#include "vp_internal.h"

namespace {

// One warp per group of four activations: slowest lane (bytes x rate_lcm / bw of its path), then lambda * rate_lcm + that,
// summed over the activations of the matrix.  Integer throughout, so the order of the sums does not matter.
__global__ void __launch_bounds__(256)
plan_time_kernel(const uint32_t* __restrict__ inst_wdiv, int n_inst, int64_t W, int N, int k_max, int B,
                 const int32_t* __restrict__ n_steps, const uint16_t* __restrict__ lane_inst,
                 const int64_t* __restrict__ lane_bytes, int64_t lambda_ns, int64_t* __restrict__ time_xw) {
    __shared__ unsigned long long s_sum;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, n_warps = blockDim.x >> 5;
    for (int b = blockIdx.x; b < B; b += gridDim.x) {
        if (threadIdx.x == 0) s_sum = 0;
        __syncthreads();
        int K = n_steps[b];
        K = K < 0 ? 0 : (K > k_max ? k_max : K);
        unsigned long long acc = 0;
        // four activations per warp step: their loads are independent, so they overlap
        for (int k0 = warp * 4; k0 < K; k0 += n_warps * 4) {
            int64_t tmax[4] = {0, 0, 0, 0};
#pragma unroll
            for (int u = 0; u < 4; u++) {
                if (k0 + u >= K) continue;
                const size_t row = ((size_t)b * k_max + k0 + u) * N;
                for (int i = lane; i < N; i += 32) {
                    const int64_t x = lane_bytes[row + i];
                    const unsigned id = lane_inst[row + i];
                    if (x > 0 && id < (unsigned)n_inst) {
                        const int64_t t = x * (int64_t)inst_wdiv[id];
                        tmax[u] = t > tmax[u] ? t : tmax[u];
                    }
                }
            }
#pragma unroll
            for (int o = 16; o; o >>= 1)
#pragma unroll
                for (int u = 0; u < 4; u++) {
                    const int64_t other = __shfl_xor_sync(0xffffffffu, tmax[u], o);
                    tmax[u] = other > tmax[u] ? other : tmax[u];
                }
#pragma unroll
            for (int u = 0; u < 4; u++)
                if (k0 + u < K) acc += (unsigned long long)(lambda_ns * W + tmax[u]);
        }
        if (lane == 0 && acc) atomicAdd(&s_sum, acc);
        __syncthreads();
        if (threadIdx.x == 0) time_xw[b] = (int64_t)s_sum;
        __syncthreads();
    }
}

// Histogram of (source rank, destination rank) pairs of routed copies.  One cluster of one to eight CTAs takes the `group`
// sources from blockIdx / cluster size on, every CTA a slice of their copies; the counts meet in distributed shared memory,
// so a demand row is written once, by plain stores, and nothing has to be zeroed before the launch.  Bound by latency: with two
// memsets ahead of it and global atomics behind, the row of one rank with 128 tokens took 6.4 us of GPU time, now 2.0.
// Many copies: bound by the additions in shared memory; a loop of its own for a single source (no division), 16-byte loads and one wave
// of CTAs.  16,384 tokens x top-8 from 1, 64 and 256 sources: 16.4, 24.6 and 69.5 us by slices of 16,384 copies and global atomics,
// now 5.5, 18.6 and 47.1 (GPU time in a graph).
constexpr int kDemandCells = 4096;                 // group x N at most
// WIDE: a CTA has more than 2^kDemandCarry copies of one source; it moves the high bits of its counts on after every so many, and the
// row is a 64-bit sum.  (As a case at run time it cost one source of a few thousand copies 4.5 -> 4.8 us.)
constexpr int kDemandCarry = 28;
template <bool WIDE>
__global__ void __launch_bounds__(kIdxThreads)
demand_kernel(const int32_t* __restrict__ idx, int n_src, int group, long long per_src, SmallDiv by_epr, int N, int src0,
              long long row_bytes, int64_t* __restrict__ demand_rows, int32_t* __restrict__ status) {
    namespace cg = cooperative_groups;
    __shared__ unsigned int cnt[kDemandCells];
    __shared__ unsigned int carried[WIDE ? VP_MAX_N : 1];     // counts in units of 2^kDemandCarry
    __shared__ int s_bad;
    const cg::cluster_group cluster = cg::this_cluster();
    const int tid = threadIdx.x, rank = (int)cluster.block_rank(), n_cta = (int)cluster.num_blocks();
    const int s0 = (int)(blockIdx.x / n_cta) * group, ns = min(group, n_src - s0), cells = ns * N;
    for (int j = tid; j < cells; j += kIdxThreads) cnt[j] = 0;
    grid_wait();
    __syncthreads();
    const long long items = ns * per_src, lo = items * rank / n_cta, hi = items * (rank + 1) / n_cta;
    const int32_t* const x0 = idx + s0 * per_src;
    int bad = 0;
    auto count = [&](int x, int first) {
        if (x < 0) return;                         // dropped copy
        const int j = by_epr.div(x);
        if (j >= N) { bad = 1; return; }
        atomicAdd(&cnt[first + j], 1u);
    };
    auto count_run = [&](const int32_t* from, long long n) {   // 16 bytes at a time between the first and the last aligned address
        const long long head = min(n, (long long)((16 - ((uintptr_t)from & 15)) & 15) / 4), quads = (n - head) / 4;
        const int4* const v = (const int4*)(from + head);
        if (tid < head) count(from[tid], 0);
#pragma unroll 4
        for (long long q = tid; q < quads; q += kIdxThreads) {
            const int4 x = v[q];
            count(x.x, 0); count(x.y, 0); count(x.z, 0); count(x.w, 0);
        }
        const long long e = head + quads * 4 + tid;
        if (e < n) count(from[e], 0);
    };
    if (WIDE) {
        for (int j = tid; j < N; j += kIdxThreads) carried[j] = 0;
        for (long long at = lo; at < hi; at += 1ll << kDemandCarry) {
            count_run(x0 + at, min(1ll << kDemandCarry, hi - at));
            __syncthreads();
            for (int j = tid; j < N; j += kIdxThreads) { carried[j] += cnt[j] >> kDemandCarry; cnt[j] &= (1u << kDemandCarry) - 1; }
            __syncthreads();
        }
    } else if (ns == 1) {
        count_run(x0 + lo, hi - lo);
    } else {                                       // (a 64-bit division per copy)
#pragma unroll 8
        for (long long e = lo + tid; e < hi; e += kIdxThreads) count(x0[e], (int)(e / per_src) * N);
    }
    bad = __syncthreads_or(bad);
    if (tid == 0) s_bad = bad;
    if (n_cta > 1) cluster.sync();
    for (int j = rank * kIdxThreads + tid; j < cells; j += n_cta * kIdxThreads) {
        unsigned int n = 0;
        for (int c = 0; c < n_cta; c++) n += cluster.map_shared_rank(cnt, c)[j];
        long long copies = n;
        if (WIDE)
            for (int c = 0; c < n_cta; c++) copies += (long long)cluster.map_shared_rank(carried, c)[j] << kDemandCarry;
        const int s = s0 + j / N, d = j % N;       // D_ii = 0: self traffic is handled locally (Section 3)
        demand_rows[(size_t)s * N + d] = d == src0 + s ? 0 : copies * row_bytes;
    }
    if (rank == 0 && tid == 0) {
        for (int c = 1; c < n_cta; c++) bad |= *cluster.map_shared_rank(&s_bad, c);
        if (group >= n_src) *status = bad ? 1 : 0;            // this cluster saw every source
        else if (bad) atomicOr(status, 1);                    // (zeroed before the launch)
    }
    if (n_cta > 1) cluster.sync();                 // no CTA leaves while another reads its counts
}

}  // namespace

extern "C" int vp_plan_time(const vp_catalog* c, int B, int k_max, const int32_t* n_steps, const uint16_t* lane_inst,
                            const int64_t* lane_bytes, int64_t lambda_ns, int64_t* time_xw, void* cuda_stream) {
    if (!c || c->device < 0 || B <= 0 || k_max <= 0 || !n_steps || !lane_inst || !lane_bytes || !time_xw) return VP_E_BAD_ARG;
    if (lambda_ns < 0 || lambda_ns >= VP_ENTRY_LIMIT) return VP_E_BAD_ARG;
    int prev = -1;
    cudaGetDevice(&prev);
    if (cudaSetDevice(c->device) != cudaSuccess) return VP_E_CUDA;
    const int grid = B < c->sm_count * 8 ? B : c->sm_count * 8;
    plan_time_kernel<<<grid, 256, 0, (cudaStream_t)cuda_stream>>>(c->dc.inst_wdiv, c->dc.n_inst, c->dc.W, c->dc.N, k_max, B,
                                                                  n_steps, lane_inst, lane_bytes, lambda_ns, time_xw);
    g_vp_launches++;
    const int rc = cudaGetLastError() == cudaSuccess ? VP_OK : VP_E_CUDA;
    if (prev >= 0) cudaSetDevice(prev);
    return rc;
}

extern "C" int vp_demand_from_routing(const int32_t* expert_idx, int n_src, int T, int topk, int experts_per_rank, int N,
                                      int src0, int64_t row_bytes, int64_t* demand_rows, int32_t* status,
                                      void* cuda_stream) {
    if (!expert_idx || !demand_rows || !status) return VP_E_BAD_ARG;
    if (n_src <= 0 || T <= 0 || topk <= 0 || experts_per_rank <= 0 || N <= 0 || N > VP_MAX_N || src0 < 0 ||
        src0 + n_src > N || row_bytes <= 0 || row_bytes >= VP_ENTRY_LIMIT)
        return VP_E_BAD_ARG;
    cudaStream_t stream = (cudaStream_t)cuda_stream;
    const long long per_src = (long long)T * topk, total = per_src * n_src;
    // Few copies from few sources: one cluster counts them all and writes the status itself.  Otherwise a cluster per source,
    // which share the status word.
    const bool one = (long long)n_src * N <= kDemandCells && total <= 65536;
    const int group = one ? n_src : 1;
    if (group < n_src && cudaMemsetAsync(status, 0, sizeof(int32_t), stream) != cudaSuccess) return VP_E_CUDA;
    const long long items = group * per_src;
    int ctas = 1;
    // four copies per thread, then more CTAs, up to one wave of them (four per SM): every further wave is another launch latency and trip to memory
    const int groups = (n_src + group - 1) / group;
    while (ctas < 8 && (long long)ctas * 4 * kIdxThreads < items && (ctas == 1 || groups * ctas * 2 <= 4 * sm_count_of_device())) ctas *= 2;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(groups * ctas));
    cfg.blockDim = dim3(kIdxThreads);
    cfg.stream = stream;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    at[1].id = cudaLaunchAttributeClusterDimension;
    at[1].val.clusterDim.x = (unsigned)ctas; at[1].val.clusterDim.y = 1; at[1].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = ctas > 1 ? 2 : 1;
    g_vp_launches++;
    const auto kernel = items > (long long)ctas << kDemandCarry ? demand_kernel<true> : demand_kernel<false>;
    return cudaLaunchKernelEx(&cfg, kernel, expert_idx, n_src, group, per_src, small_div(experts_per_rank), N, src0,
                              (long long)row_bytes, demand_rows, status) == cudaSuccess ? VP_OK : VP_E_CUDA;
}

// ---- plan-quality sweep: Eq. (2) over a grid of (lambda, K_target) ---------------------------------------------------

namespace {

struct SweepBufs {
    int32_t *n_steps, *chan_id, *status;
    int16_t* lane_dst;
    uint16_t* lane_inst;
    int64_t *lane_bytes, *send_off, *tau;
    void* ws;
    size_t ws_bytes, total;
};

SweepBufs carve_sweep(char* base, const vp_catalog* c, int B, const vp_sched_params* p) {
    const size_t N = (size_t)c->info.N, K = (size_t)p->k_max, b = (size_t)B;
    size_t off = 0;
    auto take = [&](size_t bytes) { char* at = base ? base + off : nullptr; off += vp_align256(bytes); return (void*)at; };
    SweepBufs s;
    s.n_steps = (int32_t*)take(b * 4);
    s.chan_id = (int32_t*)take(b * K * 4);
    s.status = (int32_t*)take(b * 4);
    s.lane_dst = (int16_t*)take(b * K * N * 2);
    s.lane_inst = (uint16_t*)take(b * K * N * 2);
    s.lane_bytes = (int64_t*)take(b * K * N * 8);
    s.send_off = (int64_t*)take(b * (K + 1) * N * 8);
    s.tau = (int64_t*)take(b * 8);
    s.ws_bytes = vp_schedule_workspace_bytes(c, B, p);
    s.ws = take(s.ws_bytes);
    s.total = off;
    return s;
}

}  // namespace

extern "C" size_t vp_sweep_workspace_bytes(const vp_catalog* c, int B, const vp_sched_params* p) {
    if (!c || !p || B <= 0 || p->k_max <= 0) return 0;
    SweepBufs s = carve_sweep(nullptr, c, B, p);
    return s.ws_bytes ? s.total : 0;
}

extern "C" int vp_sweep_plan_time(const vp_catalog* c, const vp_sched_params* p, const int64_t* demand, int B,
                                  const int64_t* lambda_ns, int n_lambda, const int32_t* k_target, int n_k, int64_t* time_xw,
                                  int32_t* n_steps_out, int32_t* status_out, void* workspace, size_t workspace_bytes,
                                  void* cuda_stream) {
    if (!c || !p || !demand || !lambda_ns || !k_target || !time_xw || B <= 0 || n_lambda <= 0 || n_k <= 0 || p->k_max <= 0)
        return VP_E_BAD_ARG;
    if (!workspace || ((uintptr_t)workspace & 255)) return VP_E_WORKSPACE;
    SweepBufs s = carve_sweep((char*)workspace, c, B, p);
    if (!s.ws_bytes) return VP_E_BAD_ARG;
    if (workspace_bytes < s.total) return VP_E_WORKSPACE;
    cudaStream_t stream = (cudaStream_t)cuda_stream;
    for (int i = 0; i < n_lambda; i++)
        for (int j = 0; j < n_k; j++) {
            vp_sched_params q = *p;
            q.lambda_ns = lambda_ns[i];
            q.k_target = k_target[j];
            int rc = vp_schedule_batch(c, &q, demand, nullptr, B, s.n_steps, s.chan_id, s.lane_dst, s.lane_inst, s.lane_bytes, s.send_off,
                                       nullptr, s.tau, s.status, s.ws, s.ws_bytes, cuda_stream);
            if (rc) return rc;
            const size_t at = ((size_t)i * n_k + j) * B;
            rc = vp_plan_time(c, B, p->k_max, s.n_steps, s.lane_inst, s.lane_bytes, q.lambda_ns, time_xw + at, cuda_stream);
            if (rc) return rc;
            if (n_steps_out && cudaMemcpyAsync(n_steps_out + at, s.n_steps, (size_t)B * 4, cudaMemcpyDeviceToDevice, stream) != cudaSuccess)
                return VP_E_CUDA;
            if (status_out && cudaMemcpyAsync(status_out + at, s.status, (size_t)B * 4, cudaMemcpyDeviceToDevice, stream) != cudaSuccess)
                return VP_E_CUDA;
        }
    return VP_OK;
}
