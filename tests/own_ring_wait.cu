// The rings of the one-launch forms when a bounded wait gives up (tests/test_gpu_index_forms.py).  All loads of the first units have landed
// before the limit is made to run out: from stage `at` on the wait is for the phase after them, which nothing completes.
#include "route_index.cuh"

namespace {

__global__ void __launch_bounds__(kOwnWarps * 32) ring_kernel(const char* rows, char* out, long long row_bytes, int own, int fanout, const int* src, const int* dst, int at, SmallLaunch z, int* gave_up) {
    extern __shared__ __align__(128) int sm[];
    __shared__ __align__(8) unsigned long long bars[kOwnWarps * kOwnStages];
    OwnRingOf<256> ring;
    ring.init(z, rows, out, row_bytes, 0, (int)(row_bytes / 16), sm, bars);
    const auto from = [&](int i) { return src[i]; };
    ring.start(own, from);
    bool landed = true;
    for (int s = 0; s < kOwnStages; s++)
        if (ring.loaded >> s & 1) landed &= mbar_wait_bounded(ring.bars + 8 * s, 0, kOwnSpins);
    if (!__all_sync(0xffffffffu, landed)) return;
    ring.phase |= ring.loaded >> at << at;
    if (!ring.finish(fanout, dst, from) && (threadIdx.x & 31) == 0) atomicAdd(gave_up, 1);
}

}  // namespace

// own rows of row_bytes (a multiple of 16, at least 2 KB); src [own], dst [own * fanout]; gave_up: warps whose wait ran out.
extern "C" int run_ring(const void* rows, void* out, long long row_bytes, int own, int fanout, const int* src, const int* dst, int at, int* gave_up) {
    SmallLaunch z = small_launch(own, 1, fanout, row_bytes, 16, kMinOwnBulk, [](int) { return 0; });
    if (!z.bulk || z.grid != 1) return -1;
    if (cudaFuncSetAttribute(ring_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)z.smem) != cudaSuccess) return -2;
    ring_kernel<<<1, kOwnWarps * 32, z.smem>>>((const char*)rows, (char*)out, row_bytes, own, fanout, src, dst, at, z, gave_up);
    if (cudaGetLastError() != cudaSuccess) return -3;
    return cudaDeviceSynchronize() == cudaSuccess ? 0 : -4;
}
