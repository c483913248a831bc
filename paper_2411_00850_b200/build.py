"""Builds the C-ABI shared library (libgwq.so) in-tree with nvcc for sm_100a, and the native half of its torch binding
(_gwq_torch.so) with the host compiler.

Every source is compiled to an object of its own (in parallel, rebuilt only when it or a header
is newer), then the objects are linked into the shared library."""
from __future__ import annotations

import os
import subprocess
import sys
from concurrent.futures import ThreadPoolExecutor

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
OBJ = os.path.join(HERE, "_build")
LIB = os.path.join(HERE, "libgwq.so")
AID_SRC = os.path.join(HERE, "bench_aid", "read_probe.cu")    # the benchmark's read-only launch, a library of its own
AID_LIB = os.path.join(HERE, "bench_aid", "libbench_read_probe.so")
EXT_SRC = os.path.join(CSRC, "torch_ext.cpp")
EXT_LIB = os.path.join(HERE, "_gwq_torch.so")
SOURCES = ("linear_skinny.cu", "stream_w4_f16.cu", "stream_w4_bf16.cu", "stream_w3_f16.cu", "stream_w3_bf16.cu", "stream_w8_f16.cu",
           "stream_w8_bf16.cu", "stream_w2_f16.cu", "stream_w2_bf16.cu",
           "decode_w4_f16.cu", "decode_w4_bf16.cu", "decode_w3_f16.cu", "decode_w3_bf16.cu", "decode_w8_f16.cu",
           "decode_w8_bf16.cu", "decode_w2_f16.cu", "decode_w2_bf16.cu", "alloc.cu", "select.cu",
           "select_fast.cu", "select_static.cu", "pack.cu", "linear_simt.cu", "linear_decode.cu", "linear_stream.cu", "linear_prefill.cu",
           "quality.cu", "gradmean.cu", "api.cu")
NVCC_FLAGS = (
    "-gencode", "arch=compute_100a,code=sm_100a", "-O3", "-lineinfo", "-std=c++17",
    "-Xcompiler", "-fPIC",
)


def _nvcc() -> str:
    for cand in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", "nvcc"):
        if cand and (os.path.isabs(cand) and os.path.exists(cand) or not os.path.isabs(cand)):
            return cand
    raise RuntimeError("nvcc not found")


def _headers():
    hs = [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith((".cuh", ".h"))]
    hs.append(os.path.join(os.path.dirname(HERE), "include", "gwq.h"))
    return hs


def _stale(target: str, deps) -> bool:
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    return any(os.path.getmtime(d) > t for d in deps)


def needs_build() -> bool:
    deps = [os.path.join(CSRC, f) for f in os.listdir(CSRC)] + _headers()
    return _stale(LIB, deps) or _stale(AID_LIB, [AID_SRC]) or _stale(EXT_LIB, _ext_deps())


def _build_aid(force: bool) -> None:
    if not force and not _stale(AID_LIB, [AID_SRC]):
        return
    res = subprocess.run([_nvcc(), *NVCC_FLAGS, "-shared", AID_SRC, "-o", AID_LIB, "-lcudart"],
                         capture_output=True, text=True)
    if res.returncode != 0:
        raise RuntimeError("nvcc failed on read_probe.cu:\n" + res.stdout + res.stderr)


def _ext_deps():
    return [EXT_SRC, os.path.join(os.path.dirname(HERE), "include", "gwq.h")]


def _build_ext(force: bool) -> None:
    """The CPython module of the torch binding; finds libgwq.so beside itself."""
    if not force and not _stale(EXT_LIB, _ext_deps()):
        return
    import sysconfig

    import torch
    from torch.utils import cpp_extension
    cuda = os.path.dirname(os.path.dirname(os.path.realpath(_nvcc())))
    includes = [sysconfig.get_paths()["include"], os.path.join(cuda, "include"), *cpp_extension.include_paths()]
    libs = cpp_extension.library_paths() + [os.path.join(cuda, "lib64")]
    res = subprocess.run(
        ["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-DNDEBUG",
         f"-D_GLIBCXX_USE_CXX11_ABI={int(torch.compiled_with_cxx11_abi())}",
         *(f"-I{d}" for d in includes), EXT_SRC, "-o", EXT_LIB, *(f"-L{d}" for d in libs),
         "-lc10", "-lc10_cuda", "-ltorch_cpu", "-ltorch_cuda", "-ltorch", "-ltorch_python", "-lcudart",
         f"-L{HERE}", "-l:libgwq.so", "-Wl,-rpath,$ORIGIN"], capture_output=True, text=True)
    if res.returncode != 0:
        raise RuntimeError("g++ failed on torch_ext.cpp:\n" + res.stdout + res.stderr)


def _compile(src: str, force: bool, verbose: bool) -> str:
    path = os.path.join(CSRC, src)
    obj = os.path.join(OBJ, src[:-3] + ".o")
    if not force and not _stale(obj, [path] + _headers()):
        return ""
    cmd = [_nvcc(), *NVCC_FLAGS, "-c", path, "-o", obj]
    if verbose:
        cmd += ["-Xptxas", "-v"]
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        raise RuntimeError(f"nvcc failed on {src}:\n" + res.stdout + res.stderr)
    return res.stderr


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile every CUDA source and link libgwq.so; returns the library path."""
    if not force and not needs_build():
        return LIB
    os.makedirs(OBJ, exist_ok=True)
    _build_aid(force)
    with ThreadPoolExecutor(max_workers=min(len(SOURCES), os.cpu_count() or 4)) as pool:
        logs = list(pool.map(lambda s: _compile(s, force, verbose), SOURCES))
    if verbose:
        sys.stderr.write("".join(logs))
    objs = [os.path.join(OBJ, s[:-3] + ".o") for s in SOURCES]
    res = subprocess.run([_nvcc(), "-shared", "-o", LIB, *objs, "-lcudart"], capture_output=True, text=True)
    if res.returncode != 0:
        raise RuntimeError("link failed:\n" + res.stdout + res.stderr)
    _build_ext(force)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
