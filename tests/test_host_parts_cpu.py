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
