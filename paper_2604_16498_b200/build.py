"""Builds the CUDA library in-tree: ``paper_2604_16498_b200/libforge.so`` (sm_100a only), and the native half of
the Python binding, ``host_calls``.

``python -m paper_2604_16498_b200.build`` or ``build()`` from Python.  nvcc cross-compiles
without a GPU.  Each is rebuilt when one of its sources or headers is newer than it, ``host_calls`` also when it was
built for another torch.  Without what ``host_calls`` needs (torch's and Python's headers, g++) the library is built all the
same: the binding works without it, at a few microseconds more per call.
"""
from __future__ import annotations

import glob
import os
import subprocess
import sys
import sysconfig
from concurrent.futures import ThreadPoolExecutor

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
INCLUDE = os.path.join(os.path.dirname(HERE), "include")
LIB = os.path.join(HERE, "libforge.so")
HOST_CALLS = os.path.join(HERE, "host_calls" + (sysconfig.get_config_var("EXT_SUFFIX") or ".so"))  # importable by this Python only
OBJ_DIR = os.path.join(HERE, "_build")

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
    "-Xcompiler", "-fPIC",
]


def _nvcc() -> str:
    cand = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "bin", "nvcc")
    return cand if os.path.exists(cand) else "nvcc"


def host_calls_stamp() -> str:
    """What host_calls is built for: it reads tensors through torch's inline accessors, whose layouts are those of one build of torch."""
    import torch
    return f"torch {torch.__version__} {torch.version.git_version} python {sysconfig.get_config_var('EXT_SUFFIX')}"


def _older(path: str, deps) -> bool:
    return not os.path.exists(path) or any(os.path.getmtime(d) > os.path.getmtime(path) for d in deps)


def _headers() -> list:
    return glob.glob(os.path.join(INCLUDE, "*.h"))


def _stale() -> bool:
    return _older(LIB, glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh")) + _headers())


def _host_calls_stale() -> bool:
    if _older(HOST_CALLS, [os.path.join(CSRC, "host_calls.cpp"), *_headers()]):
        return True
    try:
        stamp = host_calls_stamp()
    except ImportError:  # no torch, no binding
        return False
    with open(HOST_CALLS, "rb") as f:
        return stamp.encode() not in f.read()


def _build_host_calls() -> None:
    import torch
    t = os.path.dirname(torch.__file__)
    tmp = HOST_CALLS + f".tmp{os.getpid()}"
    cuda = os.path.dirname(os.path.dirname(_nvcc())) or "/usr/local/cuda"
    inc = [os.path.join(t, "include"), os.path.join(t, "include", "torch", "csrc", "api", "include"),
           os.path.join(cuda, "include"), sysconfig.get_paths()["include"]]
    r = subprocess.run(["g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-fvisibility=hidden",
                        f"-D_GLIBCXX_USE_CXX11_ABI={int(torch.compiled_with_cxx11_abi())}",
                        f'-DFORGE_HOST_CALLS_STAMP="{host_calls_stamp()}"', *(f"-I{i}" for i in inc),
                        os.path.join(CSRC, "host_calls.cpp"), "-o", tmp, "-L" + os.path.join(t, "lib"),
                        "-ltorch_python", "-ltorch_cpu", "-lc10", "-lc10_cuda"], capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"g++ failed for host_calls.cpp:\n{r.stdout}\n{r.stderr}")
    os.replace(tmp, HOST_CALLS)


def _try_host_calls() -> None:
    """Builds host_calls, or says why not; one that is out of date does not stay."""
    for old in {os.path.join(HERE, "host_calls.so"), HOST_CALLS}:
        if os.path.exists(old):
            os.remove(old)
    try:
        _build_host_calls()
    except Exception as e:  # whatever is missing: the library does not depend on it
        print(f"host_calls was not built, the binding's calls go the general way: {e}", file=sys.stderr)


def build(force: bool = False, verbose: bool = False) -> str:
    lib, host = force or _stale(), force or _host_calls_stale()
    with ThreadPoolExecutor(max_workers=1) as pool:
        done = pool.submit(_try_host_calls) if host else None
        if lib:
            _build_lib(verbose)
        if done:
            done.result()
    return LIB


def _build_lib(verbose: bool) -> None:
    os.makedirs(OBJ_DIR, exist_ok=True)
    sources = sorted(glob.glob(os.path.join(CSRC, "*.cu")))
    objs = [os.path.join(OBJ_DIR, os.path.basename(s)[:-3] + ".o") for s in sources]
    extra = ["-Xptxas", "-v"] if verbose else []

    def compile_one(pair):
        src, obj = pair
        cmd = [_nvcc(), *NVCC_FLAGS, *extra, "-I", INCLUDE, "-c", src, "-o", obj]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError(f"nvcc failed for {src}:\n{r.stdout}\n{r.stderr}")
        if verbose:
            sys.stderr.write(r.stderr)

    with ThreadPoolExecutor(max_workers=min(8, len(sources))) as pool:
        list(pool.map(compile_one, zip(sources, objs)))
    tmp = LIB + f".tmp{os.getpid()}"
    r = subprocess.run([_nvcc(), "-shared", "-o", tmp, *objs, "-gencode", "arch=compute_100a,code=sm_100a"],
                       capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"link failed:\n{r.stdout}\n{r.stderr}")
    os.replace(tmp, LIB)


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
