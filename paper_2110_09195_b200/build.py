"""Builds libsnnconv.so (the C-ABI CUDA library) in-tree with nvcc for sm_100a, and _snn_fast (the binding's checks as a
Python module in C++) with the host compiler.  The library needs neither torch nor the module; the module needs torch."""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig
from concurrent.futures import ThreadPoolExecutor
from pathlib import Path

PKG = Path(__file__).resolve().parent
CSRC = PKG / "csrc"
INCLUDE = PKG.parent / "include"
LIB = PKG / "libsnnconv.so"
FAST = PKG / ("_snn_fast" + (sysconfig.get_config_var("EXT_SUFFIX") or ".so"))
FAST_SOURCE = CSRC / "snn_fast.cpp"
FAST_TORCH = PKG / "_build" / "_snn_fast.torch"   # the version of torch it was built for
SOURCES = ["snn_api.cu", "snn_decode.cu", "snn_popc.cu", "snn_reuse.cu", "snn_reuse_f16.cu", "snn_tcg.cu", "snn_microbench.cu", "snn_static.cu"]
NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
    "-Xcompiler", "-fPIC", "-Xcompiler", "-fvisibility=hidden", f"-I{INCLUDE}", f"-I{CSRC}",
]


def _nvcc() -> str:
    cand = os.environ.get("NVCC") or "/usr/local/cuda/bin/nvcc"
    return cand if os.path.exists(cand) else "nvcc"


def _stale() -> bool:
    if not LIB.exists():
        return True
    t = LIB.stat().st_mtime
    deps = list(CSRC.glob("*.cu")) + list(CSRC.glob("*.h")) + list(CSRC.glob("*.cuh")) + list(INCLUDE.glob("*.h"))
    return any(d.stat().st_mtime > t for d in deps)


def build_fast(force: bool = False, verbose: bool = False) -> Path:
    """The module reads torch's tensors by the layout in torch's headers: it is built for the torch that will call it."""
    import torch
    deps = (FAST_SOURCE, INCLUDE / "snn_conv.h")
    if (not force and FAST.exists() and all(d.stat().st_mtime <= FAST.stat().st_mtime for d in deps)
            and FAST_TORCH.exists() and FAST_TORCH.read_text() == torch.__version__):
        return FAST
    root = Path(torch.__file__).resolve().parent
    tmp = FAST.with_name(f"_snn_fast.tmp{os.getpid()}.so")
    cuda = Path(_nvcc()).parent.parent / "include"
    cmd = [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-shared", "-fPIC", "-fvisibility=hidden", "-w",
           f'-DSNN_TORCH_VERSION="{torch.__version__}"',
           f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}", f"-I{INCLUDE}", f"-I{root}/include",
           f"-I{root}/include/torch/csrc/api/include", f"-I{sysconfig.get_paths()['include']}", f"-I{cuda}", str(FAST_SOURCE),
           "-o", str(tmp), f"-L{root}/lib", "-lc10", "-lc10_cuda", "-ltorch_cpu", "-ltorch_python"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if verbose or r.returncode:
        sys.stderr.write(r.stdout + r.stderr)
    if r.returncode:
        raise RuntimeError(f"{cmd[0]} failed on {FAST_SOURCE.name}")
    os.replace(tmp, FAST)
    FAST_TORCH.parent.mkdir(exist_ok=True)
    FAST_TORCH.write_text(torch.__version__)
    return FAST


def build_library(force: bool = False, verbose: bool = False) -> Path:
    if not force and not _stale():
        return LIB
    objdir = PKG / "_build"
    objdir.mkdir(exist_ok=True)
    extra = ["-Xptxas", "-v"] if verbose else []
    extra += os.environ.get("SNN_NVCC_FLAGS", "").split()   # e.g. -DSNN_TRACE (per-role wait counters)

    def compile_one(src: str) -> Path:
        obj = objdir / (src + ".o")
        cmd = [_nvcc(), *NVCC_FLAGS, *extra, "-c", str(CSRC / src), "-o", str(obj)]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if verbose or r.returncode:
            sys.stderr.write(r.stdout + r.stderr)
        if r.returncode:
            raise RuntimeError(f"nvcc failed on {src}")
        return obj

    with ThreadPoolExecutor(max_workers=min(8, len(SOURCES))) as ex:
        objs = list(ex.map(compile_one, SOURCES))
    tmp = LIB.with_suffix(f".tmp{os.getpid()}.so")
    cmd = [_nvcc(), "-shared", "-o", str(tmp), *map(str, objs), "-lcudart_static", "-lcuda",
           "-Xlinker", "--exclude-libs,ALL"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode:
        sys.stderr.write(r.stdout + r.stderr)
        raise RuntimeError("link failed")
    os.replace(tmp, LIB)
    return LIB


def build(force: bool = False, verbose: bool = False) -> Path:
    """The library, and the module where torch is there and the host compiler takes its headers."""
    lib = build_library(force, verbose)
    try:
        build_fast(force, verbose)
    except (ImportError, OSError, RuntimeError) as e:
        sys.stderr.write(f"{FAST.name} was not built ({e})\n")
    return lib


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
