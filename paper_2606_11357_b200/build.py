"""Build libtilefuse.so (sm_100a only) in-tree with nvcc.  `python -m paper_2606_11357_b200.build`."""
from __future__ import annotations

import os
import subprocess
import sys

PKG = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(PKG, "csrc")
LIB = os.path.join(PKG, "libtilefuse.so")
NATIVE = os.path.join(PKG, "_native.so")          # CPython module with the device calls of the binding
OBJ = os.path.join(PKG, "build")
SOURCES = ["pack.cpp", "api.cu", "gemv.cu", "gemv_raw.cu", "gemm.cu", "unpack.cu", "static_scratch.cu", "repack.cu"]
NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-std=c++17", "-O3", "-lineinfo",
    "-Xcompiler", "-fPIC", "-Xcompiler", "-fvisibility=hidden", "--use_fast_math=false",
]


def _nvcc() -> str:
    cand = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "bin", "nvcc")
    return cand if os.path.exists(cand) else "nvcc"


def _deps_mtime() -> float:
    paths = [os.path.join(CSRC, f) for f in os.listdir(CSRC)]
    paths.append(os.path.join(os.path.dirname(PKG), "include", "tilefuse.h"))
    paths.append(os.path.abspath(__file__))
    return max(os.path.getmtime(p) for p in paths)


def _compile(src: str, verbose: bool) -> str:
    obj = os.path.join(OBJ, src.rsplit(".", 1)[0] + ".o")
    flags = [f for f in NVCC_FLAGS if f != "--use_fast_math=false"]
    cmd = [_nvcc(), *flags, "-c", os.path.join(CSRC, src), "-o", obj]
    if verbose:
        cmd.insert(1, "-Xptxas=-v")
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        raise RuntimeError(f"nvcc failed on {src}:\n{res.stdout}\n{res.stderr}")
    if verbose:
        sys.stderr.write(res.stderr)
    return obj


def _torch_version() -> str:
    """Of the torch that is loaded, where one is (the binding asks on its first call), else of the installed one."""
    if "torch" in sys.modules:
        return str(sys.modules["torch"].__version__)
    from importlib.metadata import version
    return version("torch")


def _native_target() -> str:
    """What the binding's CPython module is built for: it uses torch's C++ interface, which changes with every release, and Python's."""
    return f"tilefuse native for torch {_torch_version()}, {sys.implementation.cache_tag}"


def native_is_current() -> bool:
    """The module carries its target as a string: no file beside it can get lost or be about another build."""
    if not os.path.exists(NATIVE):
        return False
    with open(NATIVE, "rb") as f:
        return _native_target().encode() + b"\0" in f.read()


def _compile_native() -> None:
    """The binding's CPython module: host code only, against the headers of Python and of torch."""
    import sysconfig

    from importlib.util import find_spec
    torch = os.path.dirname(find_spec("torch").origin)
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    include = [sysconfig.get_paths()["include"], os.path.join(torch, "include"),
               os.path.join(torch, "include", "torch", "csrc", "api", "include"), os.path.join(cuda, "include")]
    cmd = ["g++", "-std=c++17", "-O2", "-fPIC", "-shared", "-fvisibility=hidden", f'-DTF_NATIVE_TARGET="{_native_target()}"',
           os.path.join(CSRC, "native.cpp"), "-o", NATIVE,
           *[a for d in include for a in ("-isystem", d)], "-L" + PKG, "-l:libtilefuse.so", "-Wl,-rpath,$ORIGIN",
           "-L" + os.path.join(torch, "lib"), "-ltorch_python", "-lc10_cuda", "-lc10", "-ltorch_cpu"]
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        raise RuntimeError(f"g++ failed on native.cpp:\n{res.stdout}\n{res.stderr}")


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile every source for sm_100a and link the shared library; returns its path."""
    newest = _deps_mtime()
    fresh = [not force and os.path.exists(p) and os.path.getmtime(p) >= newest for p in (LIB, NATIVE)]
    if not fresh[0]:
        _compile_library(verbose)
    if not (all(fresh) and native_is_current()):
        _compile_native()
    return LIB


def _compile_library(verbose: bool) -> None:
    from concurrent.futures import ThreadPoolExecutor
    os.makedirs(OBJ, exist_ok=True)
    with ThreadPoolExecutor(max_workers=len(SOURCES)) as pool:
        objs = list(pool.map(lambda s: _compile(s, verbose), SOURCES))
    cmd = [_nvcc(), "-gencode", "arch=compute_100a,code=sm_100a", "--shared", "-cudart", "static",
           "-o", LIB, *objs]
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        raise RuntimeError(f"link failed:\n{res.stdout}\n{res.stderr}")


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
