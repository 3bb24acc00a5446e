// What the sender of an exchange does once its chunk parts are stored: every receiver's arrival counter grows by the bytes that
// arrived there.  Device code; it compiles as plain C++ too, with the fence and the addition given by the caller.
#pragma once

#ifdef __CUDACC__
#define VP_ANNOUNCE __device__ __forceinline__
#else
#define VP_ANNOUNCE inline
#endif

// Lane `lane` of one warp, after a barrier behind all stores of the CTA: adds count[j] for the ranks j = lane, lane + 32, ...  The
// fence is each lane's own.  A receiver's acquire load synchronises with a relaxed addition only if the thread that adds has a
// release fence before it in its program order; a fence of lane 0 and a warp barrier announce nothing for the other lanes.
// (The barrier orders the CTA's stores before the fence, which is cumulative.)
template <typename Fence, typename Add>
VP_ANNOUNCE void announce_counts(int lane, int n, const unsigned long long* count, Fence fence, Add add) {
    fence();
    for (int j = lane; j < n; j += 32)
        if (count[j]) add(j, count[j]);
}
