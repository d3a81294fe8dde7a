"""Builds libfathom.so (nvcc, sm_100a) and the extension module that calls it (g++) in-tree (no JIT cache, no torch extension
machinery)."""
from __future__ import annotations

import concurrent.futures
import os
import subprocess
import sys
import sysconfig
import tempfile

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libfathom.so")
NATIVE = os.path.join(HERE, "_native" + sysconfig.get_config_var("EXT_SUFFIX"))
NATIVE_SOURCE = os.path.join(CSRC, "native_binding.cpp")
SOURCES = ["fathom_api.cu", "build_planes.cu", "alloc_depth.cu", "scan.cu", "scan_simt.cu", "topk.cu", "topk_resident.cu", "sparse_attend.cu", "gather_union.cu", "klt.cu", "klt_tc.cu", "klt_eig.cu", "layer_plan.cu"]


def nvcc_path() -> str:
    cand = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "bin", "nvcc")
    return cand if os.path.exists(cand) else "nvcc"


def needs_build() -> bool:
    if not (os.path.exists(LIB) and os.path.exists(NATIVE)):
        return True
    t = min(os.path.getmtime(LIB), os.path.getmtime(NATIVE))
    deps = [os.path.join(CSRC, f) for f in os.listdir(CSRC)] + [os.path.join(ROOT, "include", "fathom.h")]
    return any(os.path.getmtime(p) > t for p in deps)


def _run(cmd, verbose: bool = False) -> None:
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        sys.stderr.write(r.stdout + r.stderr)
        raise RuntimeError("%s failed: %s" % (os.path.basename(cmd[0]), " ".join(cmd)))
    if verbose:
        sys.stderr.write(r.stderr)


def build(force: bool = False, verbose: bool = False) -> str:
    if not force and not needs_build():
        return LIB
    nvcc = [nvcc_path(), "-gencode", "arch=compute_100a,code=sm_100a", "-O3", "-std=c++17", "-lineinfo", "-Xcompiler", "-fPIC",
            "-cudart", "static", "-I", os.path.join(ROOT, "include"), "-I", CSRC]
    nvcc += os.environ.get("FATHOM_NVCC_FLAGS", "").split()       # extra flags, e.g. "-DNDEBUG"
    with tempfile.TemporaryDirectory() as tmp:                    # one nvcc per source, side by side
        objs = [os.path.join(tmp, s + ".o") for s in SOURCES]
        compile_ = lambda s, o: _run(nvcc + (["-Xptxas", "-v"] if verbose else []) + ["-c", os.path.join(CSRC, s), "-o", o], verbose)
        with concurrent.futures.ThreadPoolExecutor(os.cpu_count() or 1) as pool:
            list(pool.map(compile_, SOURCES, objs))
        _run(nvcc + ["-shared"] + objs + ["-o", LIB], verbose)
    build_native()
    return LIB


def build_native() -> str:
    """The CPython extension behind binding.py, linked to the libfathom.so beside it."""
    cmd = [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-shared", "-fPIC", "-fvisibility=hidden",
           "-I", sysconfig.get_paths()["include"], "-I", os.path.join(ROOT, "include"), NATIVE_SOURCE,
           "-L", HERE, "-l:libfathom.so", "-Wl,-rpath,$ORIGIN", "-o", NATIVE]
    _run(cmd)
    return NATIVE


if __name__ == "__main__":
    print(build(force=True, verbose="-v" in sys.argv))
