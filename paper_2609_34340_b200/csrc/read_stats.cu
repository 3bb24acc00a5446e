// vp_schedule_read_stats: host code only (it compiles as plain C++, too).
#include <cuda_runtime.h>

#include "vp_internal.h"

extern "C" int vp_schedule_read_stats(const void* workspace, void* cuda_stream, uint64_t* out3) {
    if (!workspace || !out3) return VP_E_BAD_ARG;
    cudaStream_t stream = (cudaStream_t)cuda_stream;
    const auto fetch = [&](void* to, size_t at, size_t bytes) {
        return cudaMemcpyAsync(to, (const char*)workspace + at, bytes, cudaMemcpyDeviceToHost, stream) == cudaSuccess &&
               cudaStreamSynchronize(stream) == cudaSuccess;
    };
    uint64_t head[32];
    if (!fetch(head, 0, sizeof(head))) return VP_E_CUDA;
    const uint32_t warps = (uint32_t)(head[1] >> 32);
    for (int i = 0; i < 3; i++) out3[i] = head[kStatsTagWord] ? 0 : head[2 + i];
    if (!warps || warps > kStatsMaxWarps || head[kStatsTagWord] != vp_stats_tag((uint64_t)(uintptr_t)workspace, warps)) return VP_OK;
    uint64_t part[3 * 256];                       // the warps' counters, 256 warps at a time
    for (uint32_t w = 0; w < warps; w += 256) {
        const size_t n = 3 * (size_t)(warps - w < 256 ? warps - w : 256);
        if (!fetch(part, sizeof(head) + (size_t)w * 24, n * 8)) return VP_E_CUDA;
        for (size_t i = 0; i < n; i++) out3[i % 3] += part[i];
    }
    return VP_OK;
}
