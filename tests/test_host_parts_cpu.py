"""Parts of the CUDA library that decide something without a GPU, compiled as plain C++ and run here: what each lane of a warp does,
index arithmetic near the accepted limits, and host code against a runtime that the test supplies."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2609_34340_b200", "csrc")


def _run(tmp_path, code, *sources):
    """Compiles the C++ program ``code`` (with ``sources`` of csrc/ as C++) and runs it: its checks are assertions."""
    main = tmp_path / "main.cpp"
    main.write_text("#undef NDEBUG\n#include <cassert>\n#include <initializer_list>\n" + code)
    exe = str(tmp_path / "main")
    subprocess.check_call(["g++", "-O1", "-g", "-std=c++17", "-Wall", "-fsanitize=undefined", "-fno-sanitize-recover=all", "-I", CSRC,
                           "-I", os.path.join(ROOT, "include"), "-I", "/usr/local/cuda/include", "-x", "c++", str(main)]
                          + [os.path.join(CSRC, s) for s in sources] + ["-o", exe])
    subprocess.check_call([exe], timeout=120)


def test_every_lane_fences_before_it_announces(tmp_path):
    """The arrival counters of an exchange: whichever lane adds to a counter has a system fence of its own before it, every rank's
    bytes are added once, and ranks that got nothing are left alone."""
    _run(tmp_path, r'''
#include "announce.h"
int main() {
    for (int n : {1, 8, 31, 32, 33, 64, 256}) {
        unsigned long long count[256], got[256] = {};
        for (int j = 0; j < n; j++) count[j] = j % 3 ? 100 + j : 0;
        for (int lane = 0; lane < 32; lane++) {
            bool fenced = false;
            announce_counts(lane, n, count, [&] { fenced = true; }, [&](int j, unsigned long long bytes) { assert(fenced && bytes); got[j] += bytes; });
        }
        for (int j = 0; j < n; j++) assert(got[j] == count[j]);
    }
}
''')


def test_no_plan_lowers_a_kernels_shared_memory_limit(tmp_path):
    """Launches are planned once and replayed: with many kernels on several devices, planned in any order and with any sizes, each
    launch planned so far stays within its kernel's limit."""
    _run(tmp_path, r'''
#include "smem_limit.h"
#include <map>
#include <utility>
#include <vector>
constexpr int kOptin = 232448;
static int device = 0;
static std::map<std::pair<int, const void*>, int> limit;
extern "C" cudaError_t cudaGetDevice(int* d) { *d = device; return cudaSuccess; }
extern "C" cudaError_t cudaFuncSetAttribute(const void* fn, cudaFuncAttribute a, int value) {
    assert(a == cudaFuncAttributeMaxDynamicSharedMemorySize && value <= kOptin);
    limit[{device, fn}] = value;
    return cudaSuccess;
}
int main() {
    static char kernel[30];
    struct Planned { int device; const void* fn; int bytes; };
    std::vector<Planned> planned;
    unsigned x = 1;
    for (int i = 0; i < 4000; i++) {
        x = x * 1664525u + 1013904223u;
        device = (x >> 8) % 4;
        const void* fn = &kernel[(x >> 16) % 30];
        const int bytes = (int)((x >> 4) % (unsigned)(dynamic_smem_limit(kOptin) + 1));
        assert(set_dynamic_smem_limit(fn, kOptin) == VP_OK);
        planned.push_back({device, fn, bytes});
        for (const Planned& p : planned) assert(p.bytes <= (limit[{p.device, p.fn}]));
    }
}
''')


def test_work_counters_of_any_workspace(tmp_path):
    """vp_schedule_read_stats gets no workspace size: whatever a workspace holds that no launch has used, nothing beyond its first
    256 bytes is read and nothing is allocated.  Sums, and counters of every warp, are read as they were written."""
    _run(tmp_path, r'''
#include <string.h>
#include <vector>
#include "vp_internal.h"
static const char *lo, *hi;                      // the workspace
static cudaError_t copy_result = cudaSuccess;
extern "C" cudaError_t cudaMemcpyAsync(void* dst, const void* src, size_t n, cudaMemcpyKind, cudaStream_t) {
    if (copy_result != cudaSuccess) return copy_result;
    assert((const char*)src >= lo && n <= (size_t)(hi - (const char*)src));
    memcpy(dst, src, n);
    return cudaSuccess;
}
extern "C" cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
static void read(const std::vector<uint64_t>& ws, uint64_t* out, int want = VP_OK) {
    lo = (const char*)ws.data(); hi = lo + ws.size() * 8;
    out[0] = out[1] = out[2] = 99;
    assert(vp_schedule_read_stats(ws.data(), nullptr, out) == want);
}
int main() {
    uint64_t out[3], x = 1;
    std::vector<uint64_t> ws(32);
    auto zeros = [&] { return out[0] == 0 && out[1] == 0 && out[2] == 0; };
    for (uint64_t fill : {~0ull, 0x0000040000000400ull, 0x5a5a5a5a5a5a5a5aull, 0x0000000100000001ull, 0ull}) {
        ws.assign(32, fill);
        read(ws, out);
        assert(zeros());
    }
    for (int i = 0; i < 1000; i++) {             // random bytes, and a small number of warps beside them
        for (uint64_t& w : ws) { x = x * 6364136223846793005ull + 1442695040888963407ull; w = x; }
        if (i & 1) ws[1] = (uint64_t)(1 + i) << 32;
        read(ws, out);
        assert(zeros());
    }
    ws.assign(32, 0);                            // sums
    ws[0] = 7; ws[2] = 11; ws[3] = 12; ws[4] = 13;
    read(ws, out);
    assert(out[0] == 11 && out[1] == 12 && out[2] == 13);
    for (uint32_t warps : {1u, 255u, 256u, 257u, 9472u, kStatsMaxWarps}) {       // counters of every warp
        ws.assign(32 + 3 * (size_t)warps, 0x5a5a5a5a5a5a5a5aull);
        ws[1] = (uint64_t)warps << 32 | 0x5a5a5a5a;
        ws[kStatsTagWord] = vp_stats_tag((uint64_t)(uintptr_t)ws.data(), warps);
        for (uint32_t w = 0; w < warps; w++) { ws[32 + 3 * w] = 1; ws[33 + 3 * w] = w; ws[34 + 3 * w] = 3ull << 40; }
        read(ws, out);
        assert(out[0] == warps && out[1] == (uint64_t)warps * (warps - 1) / 2 && out[2] == (3ull << 40) * warps);
        std::vector<uint64_t> moved(ws.begin(), ws.begin() + 32);                // the same bytes in another, shorter workspace
        read(moved, out);
        assert(zeros());
    }
    copy_result = cudaErrorInvalidValue;
    read(ws, out, VP_E_CUDA);
}
''', "read_stats.cu")


def test_chunks_cover_every_item_up_to_the_accepted_limit(tmp_path):
    """The chunked index forms accept up to 2^31 - 1 items: the chunks cover all of them once, in order, however many of them a
    call turns out to use."""
    _run(tmp_path, r'''
#include "chunks.h"
int main() {
    const long long most = (1ll << 31) - 1;
    for (long long items : {1ll, 511ll, 512ll, 8193ll, 1ll << 20, (1ll << 20) + 1, 1ll << 27, most - (1 << 20), most - 512, most - 1, most})
        for (int keys : {1, 2, 16, 33, 256, 1000, 1024}) {
            const int chunk = chunk_items(items, keys);
            assert(chunk > 0 && chunk % kIdxThreads == 0);
            for (long long used : {items, items - 1, items / 2, 1ll}) {
                if (used < 1) continue;
                const int n = chunks_of((unsigned)used, chunk);
                assert(n >= 1 && n <= 512 && n <= chunks_of((unsigned)items, chunk));
                long long at = 0;
                for (int b = 0; b < n; b++) {
                    const ChunkRange c = chunk_range(b, chunk, used);
                    assert(c.lo == at && c.hi > c.lo && c.hi - c.lo <= chunk);
                    at = c.hi;
                }
                assert(at == used);
            }
        }
}
''')


def test_a_buffer_counts_as_page_locked_only_as_a_whole(tmp_path):
    """Plan rows are written straight into page-locked buffers: a buffer may be page-locked in pieces, but not have a gap."""
    _run(tmp_path, r'''
#include <string.h>
#include "pinned.h"
#include <cuda.h>
struct Range { char *host, *device; size_t bytes; };
static Range ranges[8];
static int n_ranges = 0;
static const Range* find(const void* p) {
    for (int i = 0; i < n_ranges; i++)
        if ((const char*)p >= ranges[i].host && (const char*)p < ranges[i].host + ranges[i].bytes) return &ranges[i];
    return nullptr;
}
extern "C" cudaError_t cudaGetLastError() { return cudaSuccess; }
extern "C" cudaError_t cudaPointerGetAttributes(cudaPointerAttributes* a, const void* p) {
    memset(a, 0, sizeof(*a));
    const Range* r = find(p);
    if (!r) { a->type = cudaMemoryTypeUnregistered; return cudaSuccess; }
    a->type = cudaMemoryTypeHost;
    a->hostPointer = (void*)p;
    a->devicePointer = r->device + ((const char*)p - r->host);
    return cudaSuccess;
}
static CUresult attribute(void* data, CUpointer_attribute what, CUdeviceptr p) {
    for (int i = 0; i < n_ranges; i++) {
        const Range& r = ranges[i];
        if ((char*)p < r.device || (char*)p >= r.device + r.bytes) continue;
        if (what == CU_POINTER_ATTRIBUTE_RANGE_START_ADDR) *(CUdeviceptr*)data = (CUdeviceptr)r.device;
        else if (what == CU_POINTER_ATTRIBUTE_RANGE_SIZE) *(size_t*)data = r.bytes;
        else return CUDA_ERROR_INVALID_VALUE;
        return CUDA_SUCCESS;
    }
    return CUDA_ERROR_INVALID_VALUE;
}
extern "C" cudaError_t cudaGetDriverEntryPoint(const char* name, void** fn, unsigned long long, cudaDriverEntryPointQueryResult* found) {
    assert(!strcmp(name, "cuPointerGetAttribute"));
    *fn = (void*)attribute;
    if (found) *found = cudaDriverEntryPointSuccess;
    return cudaSuccess;
}
int main() {
    static char mem[9 << 16];
    char* const p = mem;
    const size_t K = 1 << 16;
    auto set = [&](std::initializer_list<Range> rs) { n_ranges = 0; for (const Range& r : rs) ranges[n_ranges++] = r; };
    set({{p, p, 9 * K}});
    assert(pinned_address(p, 9 * K) == p && pinned_address(p + 5, 1) == p + 5 && pinned_address(p + K, 8 * K) == p + K);
    assert(!pinned_address(p, 9 * K + 1) && !pinned_address(p, 0) && !pinned_address((char*)nullptr, 4));
    set({{p, p, K}, {p + K, p + K, K}, {p + 2 * K, p + 2 * K, 7 * K}});           // in pieces
    assert(pinned_address(p, 9 * K) == p && pinned_address(p + K - 1, 2) == p + K - 1);
    set({{p, p, K}, {p + 8 * K, p + 8 * K, K}});                                  // both ends, nothing between
    assert(!pinned_address(p, 9 * K));
    assert(pinned_address(p, K) == p && !pinned_address(p, K + 1) && !pinned_address(p + 4 * K, K));
    set({{p, p, K}, {p + 2 * K, p + 2 * K, K}, {p + 8 * K, p + 8 * K, K}});
    assert(!pinned_address(p, 3 * K) && !pinned_address(p, 9 * K));
    set({{p, p, K}, {p + K, p + 4 * K, K}});                                      // device addresses that do not follow on
    assert(!pinned_address(p, 2 * K));
}
''')
