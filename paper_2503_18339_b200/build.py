"""In-tree build of the GranQ CUDA library for sm_100a (nvcc cross-compiles without a GPU) and of the binding's native calls."""
from __future__ import annotations

import os
import shutil
import subprocess
import sys
import sysconfig
from concurrent.futures import ThreadPoolExecutor

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
INCLUDE = os.path.join(os.path.dirname(HERE), "include")
LIB = os.path.join(HERE, "libgranq.so")
HOST = os.path.join(HERE, "_host.so")               # the binding's calls in native code, an extension module of this package
HOST_SOURCE = os.path.join(CSRC, "granq_host.cpp")
OBJ_DIR = os.path.join(HERE, "_build")
HOST_RECORD = os.path.join(OBJ_DIR, "host_record")  # host_record() of that module, which holds the same text
SOURCES = ["granq_api.cu", "granq_flat.cu", "granq_staged.cu", "granq_l2wave.cu", "granq_colwalk.cu", "granq_colteam.cu",
           "granq_cluster.cu", "granq_hold.cu", "granq_accumulate.cu", "granq_rows.cu", "granq_weights.cu", "granq_selftest.cu", "granq_noalloc.cu"]
HEADERS = ["granq_device.cuh", "granq_internal.h"]
NVCC_FLAGS = ["-O3", "-std=c++17", "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo",
              "-Xcompiler", "-fPIC"]


def _deps():
    return [os.path.join(CSRC, f) for f in HEADERS] + [os.path.join(INCLUDE, "granq.h")]


def _newer(path: str, than: float) -> bool:
    return os.path.getmtime(path) > than


def _stale() -> bool:
    if not os.path.exists(LIB):
        return True
    t = os.path.getmtime(LIB)
    return any(_newer(d, t) for d in [os.path.join(CSRC, f) for f in SOURCES] + _deps())


def host_record() -> str:
    """What _host.so depends on besides its source: it reads torch's objects and Python's in place."""
    import torch
    return f"torch {torch.__version__}, cxx11 abi {int(torch.compiled_with_cxx11_abi())}, python {sys.version_info[0]}.{sys.version_info[1]}"


def _host_stale() -> bool:
    try:
        with open(HOST_RECORD) as f:
            same = f.read() == host_record()
    except (OSError, ImportError):
        same = False
    return not same or not os.path.exists(HOST) or any(_newer(d, os.path.getmtime(HOST)) for d in (HOST_SOURCE, os.path.join(INCLUDE, "granq.h")))


def _build_host() -> None:
    import torch
    record, home = host_record(), os.path.dirname(torch.__file__)
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(_which_nvcc()))), "include")
    tmp = HOST + f".tmp{os.getpid()}"
    subprocess.check_call([os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-fPIC", "-shared", HOST_SOURCE, "-o", tmp,
                           f'-DGRANQ_HOST_RECORD="{record}"', f"-D_GLIBCXX_USE_CXX11_ABI={int(torch.compiled_with_cxx11_abi())}",
                           f"-I{home}/include", f"-I{home}/include/torch/csrc/api/include", f"-I{cuda}",
                           f"-I{sysconfig.get_paths()['include']}", f"-L{home}/lib", "-ltorch", "-ltorch_cpu", "-ltorch_python",
                           "-lc10", "-lc10_cuda"])
    os.replace(tmp, HOST)
    os.makedirs(OBJ_DIR, exist_ok=True)
    with open(HOST_RECORD, "w") as f:
        f.write(record)


def _which_nvcc() -> str:
    nvcc = os.environ.get("NVCC", "nvcc")
    return shutil.which(nvcc) or nvcc


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile csrc/*.cu (one object per source, in parallel) and link libgranq.so beside this file, and _host.so with
    it; returns the library's path.  Objects are kept in _build/ and reused while their source and the headers are older.
    The library needs nvcc alone.  Where _host.so cannot be built (no C++ compiler, no torch, no Python headers) one line says
    so and the binding marshals its calls in Python."""
    with ThreadPoolExecutor(max_workers=1) as beside:
        host = beside.submit(_build_host) if force or _host_stale() else None
        if force or _stale():
            _build_lib(force, verbose)
        try:
            if host is not None:
                host.result()
        except Exception as e:
            if os.path.exists(HOST):
                os.remove(HOST)          # of an older source, which may call the library otherwise than it is now
            print(f"_host.so has not been built, the binding's calls are marshalled in Python: {type(e).__name__}: {e}", file=sys.stderr)
    return LIB


def _build_lib(force: bool, verbose: bool) -> None:
    nvcc = os.environ.get("NVCC", "nvcc")
    os.makedirs(OBJ_DIR, exist_ok=True)

    def compile_one(src: str) -> str:
        obj = os.path.join(OBJ_DIR, src.replace(".cu", ".o"))
        path = os.path.join(CSRC, src)
        if not force and not verbose and os.path.exists(obj):
            t = os.path.getmtime(obj)
            if not any(_newer(d, t) for d in [path] + _deps()):
                return obj
        cmd = [nvcc, *NVCC_FLAGS, "-I", INCLUDE, "-c", path, "-o", obj]
        if verbose:
            cmd.insert(1, "-Xptxas=-v")
        subprocess.check_call(cmd)
        return obj

    with ThreadPoolExecutor(max_workers=min(len(SOURCES), os.cpu_count() or 1)) as pool:
        objs = list(pool.map(compile_one, SOURCES))
    tmp = LIB + f".tmp{os.getpid()}"
    subprocess.check_call([nvcc, "-shared", "-cudart", "static", "-gencode", "arch=compute_100a,code=sm_100a",
                           "-o", tmp] + objs)
    os.replace(tmp, LIB)


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
