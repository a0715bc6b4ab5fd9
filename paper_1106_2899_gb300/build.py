"""Build the sm_103a shared library behind include/slipspring.h, in-tree.

    python -m paper_1106_2899_gb300.build [--force] [--verbose]

produces paper_1106_2899_gb300/libslipspring.so: one nvcc call per translation
unit, in parallel (one -gencode: arch=compute_103a,code=sm_103a), then a link.
No CPU fallback exists: without the library the Python binding raises.
"""
import os
import subprocess
import sys
import tempfile
from concurrent.futures import ThreadPoolExecutor

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
LIB = os.path.join(PKG, "libslipspring.so")
# the longest to compile first
SOURCES = [os.path.join(CSRC, f) for f in ("ss_chunk_f64_flow.cu", "ss_chunk_f64.cu", "ss_chunk_f32_flow.cu",
                                           "ss_chunk_f32.cu", "ss_batched.cu", "ss_adjoint.cu", "ss_api.cu")]
DEPS = SOURCES + [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith((".cuh", ".h", ".inl"))] + [
    os.path.join(ROOT, "include", "slipspring.h")]

NVCC_FLAGS = ["-O3", "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", "-lineinfo",
              "-Xcompiler", "-fPIC", "--expt-relaxed-constexpr"]


def nvcc():
    for cand in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", "nvcc"):
        if cand and (os.path.sep not in cand or os.path.exists(cand)):
            return cand
    return "nvcc"


def build(force: bool = False, verbose: bool = False) -> str:
    newest = max(os.path.getmtime(p) for p in DEPS)
    if not force and os.path.exists(LIB) and os.path.getmtime(LIB) >= newest:
        return LIB
    flags = NVCC_FLAGS + ["-I", os.path.join(ROOT, "include"), "-I", CSRC] + (["-Xptxas=-v"] if verbose else [])
    with tempfile.TemporaryDirectory(dir=PKG, prefix="_build_") as tmp:
        objs = [os.path.join(tmp, os.path.basename(s) + ".o") for s in SOURCES]

        def compile_one(src, obj):
            cmd = [nvcc()] + flags + ["-c", "-o", obj, src]
            if verbose:
                print(" ".join(cmd))
            subprocess.check_call(cmd)

        with ThreadPoolExecutor(len(SOURCES)) as ex:
            for f in [ex.submit(compile_one, s, o) for s, o in zip(SOURCES, objs)]:
                f.result()
        lib = os.path.join(tmp, "lib.so")
        subprocess.check_call([nvcc(), "-shared", "-o", lib] + objs)
        os.replace(lib, LIB)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="--verbose" in sys.argv))
