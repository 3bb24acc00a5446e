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
