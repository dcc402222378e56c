"""Builds libbitdelta.so in-tree with nvcc for sm_100a (cross-compiles without a GPU).

Every source is compiled to an object file on its own (in parallel), then linked; objects live in
csrc/build/ and are rebuilt only when their source or a header is newer.
"""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig
from concurrent.futures import ThreadPoolExecutor

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
OBJ = os.path.join(CSRC, "build")
LIB = os.path.join(HERE, "libbitdelta.so")
SOURCES = ["api.cu", "gemm_tc.cu", "gemm_fp4.cu", "gemm_row.cu", "compress.cu", "kernels_simple.cu"]
HEADERS = ["ptx.cuh", "plan.h", "gemm_tc.h", "gemm_common.cuh", "gemm_row.h", "row_plan.h", "early_start.h", os.path.join("..", "..", "include", "bitdelta.h")]
ARCH = ["-gencode", "arch=compute_100a,code=sm_100a"]


def _nvcc() -> str:
    cand = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "bin", "nvcc")
    return cand if os.path.exists(cand) else "nvcc"


def _newest_header() -> float:
    return max(os.path.getmtime(os.path.join(CSRC, h)) for h in HEADERS if os.path.exists(os.path.join(CSRC, h)))


def fastcall_path():
    """The extension module of csrc/fastcall.cpp (the product's CPython entry), named after what it is built against: it reads
    torch's tensors by their layout, so one of another torch or Python must not be loaded.  None without torch."""
    try:
        import torch
    except ImportError:
        return None
    commit = (getattr(torch.version, "git_version", None) or "")[:8]
    return os.path.join(HERE, f"_fastcall.torch-{torch.__version__}-{commit}{sysconfig.get_config_var('EXT_SUFFIX')}")


def fastcall_is_stale() -> bool:
    path = fastcall_path()
    return path is not None and not (os.path.exists(path) and os.path.getmtime(path) > os.path.getmtime(os.path.join(CSRC, "fastcall.cpp")))


def build_fastcall() -> None:
    """csrc/fastcall.cpp against the installed torch's headers (host code only)."""
    import torch
    from torch.utils import cpp_extension
    inc = [*cpp_extension.include_paths(), sysconfig.get_paths()["include"], os.path.join(os.path.dirname(os.path.dirname(_nvcc())), "include")]
    libs = os.path.join(os.path.dirname(torch.__file__), "lib")
    subprocess.run(["g++", "-std=c++17", "-O2", "-fPIC", "-shared", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
                    *(f"-I{d}" for d in inc), os.path.join(CSRC, "fastcall.cpp"), "-o", fastcall_path(), f"-L{libs}", "-ltorch_python",
                    "-ltorch_cpu", "-lc10", "-lc10_cuda"], check=True)


def is_stale() -> bool:
    if not os.path.exists(LIB):
        return True
    t = os.path.getmtime(LIB)
    deps = [os.path.join(CSRC, f) for f in SOURCES + HEADERS]
    return any(os.path.getmtime(d) > t for d in deps if os.path.exists(d))


def _compile(src: str, force: bool, verbose: bool, trace: bool = False, steps: bool = False) -> str:
    obj = os.path.join(OBJ, os.path.splitext(src)[0] + (".steps.o" if steps else ".trace.o" if trace else ".o"))
    path = os.path.join(CSRC, src)
    if (not force and os.path.exists(obj) and os.path.getmtime(obj) > os.path.getmtime(path)
            and os.path.getmtime(obj) > _newest_header()):
        return obj
    cmd = [_nvcc(), "-std=c++17", "-O3", "-lineinfo", *ARCH, "-Xcompiler", "-fPIC", "-c", path, "-o", obj]
    if verbose:
        cmd += ["-Xptxas", "-v"]
    if trace:
        cmd += ["-DBD_TRACE"]
    if steps:
        cmd += ["-DBD_TRACE_TIMELINE_ONLY", "-DBD_TRACE_STEPS"]
    subprocess.run(cmd, check=True)
    return obj


def build(force: bool = False, verbose: bool = False) -> str:
    if force or is_stale():
        os.makedirs(OBJ, exist_ok=True)
        with ThreadPoolExecutor(max_workers=len(SOURCES)) as pool:
            objs = list(pool.map(lambda s: _compile(s, force, verbose), SOURCES))
        subprocess.run([_nvcc(), *ARCH, "-shared", "-cudart", "shared", "-o", LIB, *objs], check=True)
    if force or fastcall_is_stale():
        # (the library does not depend on it: without torch, its headers or g++ the product's calls go through the binding's checks)
        try:
            build_fastcall()
        except (ImportError, OSError, subprocess.CalledProcessError) as e:
            print(f"the product's native entry was not built ({e}); calls go through Python", file=sys.stderr)
    return LIB


def build_trace(steps: bool = False) -> str:
    """The same library with -DBD_TRACE as libbitdelta_trace.so: the 4-bit decode kernel then adds up, per block and
    role, the cycles spent in each kind of wait into a buffer set with bitdelta_debug_set_trace_fp4 (see
    csrc/gemm_fp4.cu).  steps=True (libbitdelta_steps.so): no accumulators, but a time stamp per block, step and event
    behind the first 512 x 32 words of that buffer ([block][step mod 64][16 events]; the buffer must hold them).
    Load either by pointing BITDELTA_LIB at it.  Never the default build: the stamps cost time."""
    os.makedirs(OBJ, exist_ok=True)
    with ThreadPoolExecutor(max_workers=len(SOURCES)) as pool:
        objs = list(pool.map(lambda s: _compile(s, True, False, trace=True, steps=steps), SOURCES))
    lib = os.path.join(HERE, "libbitdelta_steps.so" if steps else "libbitdelta_trace.so")
    subprocess.run([_nvcc(), *ARCH, "-shared", "-cudart", "shared", "-o", lib, *objs], check=True)
    return lib


if __name__ == "__main__":
    if "--trace-steps" in sys.argv:
        print(build_trace(steps=True))
    elif "--trace" in sys.argv:
        print(build_trace())
    else:
        print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
