// How the items of a call (routed copies, received rows) are dealt to chunks, a CTA each: arithmetic that host and device share.
// It compiles as plain C++, too.
#pragma once

#ifdef __CUDACC__
#define VP_CHUNKS __host__ __device__ __forceinline__
#else
#define VP_CHUNKS inline
#endif

constexpr int kIdxThreads = 512;                    // threads of every index CTA
constexpr int kMinChunk = kIdxThreads;              // items per histogram of the chunked form, at least: one per thread

// Items per chunk and chunks of the chunked form: a map CTA adds up the histograms of all chunks, so their number times the
// keys is kept within 16 K words (16 chunks at least, however many keys there are).
inline int chunk_items(long long items, int keys) {
    long long most = 16384 / keys;
    if (most > 512) most = 512;
    if (most < 16) most = 16;
    long long c = (items + most - 1) / most;
    if (c < kMinChunk) c = kMinChunk;
    return (int)((c + kIdxThreads - 1) / kIdxThreads * kIdxThreads);
}

// Chunks that hold one of `items` < 2^31 items.  (Unsigned: chunks have up to 2^27 items, and a 64-bit division is long.)
VP_CHUNKS int chunks_of(unsigned items, unsigned chunk) { return (int)((items + chunk - 1) / chunk); }

// Items lo <= i < hi of chunk b.
struct ChunkRange { long long lo, hi; };
VP_CHUNKS ChunkRange chunk_range(unsigned b, int chunk, long long items) {
    const long long lo = (long long)b * chunk;
    return ChunkRange{lo, lo + chunk < items ? lo + chunk : items};
}
