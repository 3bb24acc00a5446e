"""Build the CUDA library in-tree for sm_100a: ``python -m paper_2609_34340_b200.build``."""
from __future__ import annotations

import importlib.metadata
import os
import subprocess
import sys
import sysconfig

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
LIB = os.path.join(PKG, "libvariopath.so")
CALLS = os.path.join(PKG, "_calls.so")
SOURCES = ["catalog.cu", "schedule.cu", "read_stats.cu", "pack.cu", "host_api.cu", "profile.cu", "plan_tools.cu", "analyzer.cu", "unpack.cu", "microbench.cu", "exchange.cu"]
FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
         "-Xcompiler", "-fPIC"]


def _stale(target: str, sources) -> bool:
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    deps = [os.path.join(CSRC, f) for f in sources] + [os.path.join(ROOT, "include", "variopath.h")]
    return any(os.path.getmtime(d) > t for d in deps)


def _built_for() -> str:
    """What the extension module depends on besides its sources: torch's C++ interface and Python's."""
    return f"torch {importlib.metadata.version('torch')}, python {sysconfig.get_config_var('SOABI')}"


def _calls_stale() -> bool:
    stamp = CALLS + ".built_for"
    return _stale(CALLS, ["calls.cpp"]) or not os.path.exists(stamp) or open(stamp).read() != _built_for()


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile ``csrc/*.cu`` into ``libvariopath.so`` (no GPU needed: nvcc cross-compiles) and ``csrc/calls.cpp``, the
    binding's frequent calls, into ``_calls.so``."""
    if force or _stale(LIB, [f for f in os.listdir(CSRC) if not f.endswith(".cpp")]):
        nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
        cmd = [nvcc] + FLAGS + ["-t", "0", "-I", os.path.join(ROOT, "include"), "-I", CSRC, "-shared", "-o", LIB]
        cmd += os.environ.get("VP_NVCC_EXTRA", "").split()
        cmd += [os.path.join(CSRC, s) for s in SOURCES]
        if verbose:
            cmd.insert(1, "-Xptxas=-v")
            print(" ".join(cmd))
        subprocess.check_call(cmd)
    if force or _calls_stale():
        import torch
        at = os.path.dirname(torch.__file__)
        cuda = os.path.dirname(os.path.dirname(os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")))
        cmd = ["g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-fvisibility=hidden",
               f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}", "-I", os.path.join(ROOT, "include")]
        for d in (os.path.join(at, "include"), os.path.join(at, "include", "torch", "csrc", "api", "include"),
                  os.path.join(cuda, "include"), sysconfig.get_paths()["include"]):
            cmd += ["-isystem", d]
        cmd += [os.path.join(CSRC, "calls.cpp"), "-o", CALLS, "-L" + os.path.join(at, "lib"), "-ltorch_python", "-ltorch_cpu", "-lc10",
                "-lc10_cuda", "-L" + PKG, "-l:libvariopath.so", "-Wl,-rpath,$ORIGIN"]
        subprocess.check_call(cmd)
        with open(CALLS + ".built_for", "w") as f:
            f.write(_built_for())
    return LIB


if __name__ == "__main__":
    build(force="--force" in sys.argv, verbose="-v" in sys.argv)
    print(LIB)
