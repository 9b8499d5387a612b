"""Builds the CUDA library (sm_100a only) in-tree with nvcc: one object per
translation unit, compiled in parallel, linked into one shared library; and the
CPython modules with the per-pass entry points (csrc/wino_python*), linked against it."""
from __future__ import annotations

import os
import subprocess
import sysconfig
from concurrent.futures import ThreadPoolExecutor

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
OBJ = os.path.join(HERE, "_build")
LIB = os.path.join(HERE, "libwino_b200.so")
NATIVE = os.path.join(HERE, "_native.so")
NATIVE_TORCH = os.path.join(HERE, "_native_torch.so")
NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-O3", "-lineinfo", "-std=c++17",
    "-fmad=false", "--expt-relaxed-constexpr", "-Xcompiler", "-fPIC",
]


def _units():
    return sorted(f for f in os.listdir(CSRC) if f.endswith(".cu"))


def _headers():
    hs = [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith((".h", ".cuh"))]
    return hs + [os.path.join(ROOT, "include", "wino.h")]


def build(force: bool = False, verbose: bool = False) -> str:
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    os.makedirs(OBJ, exist_ok=True)
    hdr_time = max(os.path.getmtime(h) for h in _headers())
    jobs = []
    for u in _units():
        src = os.path.join(CSRC, u)
        obj = os.path.join(OBJ, u[:-3] + ".o")
        if force or not os.path.exists(obj) or os.path.getmtime(obj) < max(os.path.getmtime(src), hdr_time):
            cmd = [nvcc, *NVCC_FLAGS, "-I", os.path.join(ROOT, "include"), "-I", CSRC, "-c", src, "-o", obj]
            if verbose:
                cmd[1:1] = ["-Xptxas", "-v"]
            jobs.append(cmd)
    if jobs:
        with ThreadPoolExecutor(max_workers=min(len(jobs), os.cpu_count() or 4)) as ex:
            for rc in ex.map(lambda c: subprocess.run(c).returncode, jobs):
                if rc != 0:
                    raise RuntimeError("nvcc failed")
    objs = [os.path.join(OBJ, u[:-3] + ".o") for u in _units()]
    if jobs or not os.path.exists(LIB) or os.path.getmtime(LIB) < max(os.path.getmtime(o) for o in objs):
        tmp = LIB + f".tmp{os.getpid()}"
        subprocess.check_call([nvcc, "-gencode", "arch=compute_100a,code=sm_100a", "-shared",
                               "-cudart", "static", *objs, "-o", tmp])
        os.replace(tmp, LIB)
    _build_native(force)
    return LIB


def _stale(target: str, abi: str, *sources: str) -> bool:
    """Missing, older than a source, or built for another interpreter or torch (the note beside it)."""
    if not os.path.exists(target) or os.path.getmtime(target) < max(os.path.getmtime(f) for f in sources):
        return True
    try:
        with open(target + ".abi") as f:
            return f.read() != abi
    except OSError:
        return True


def _install(tmp: str, target: str, abi: str) -> None:
    if os.path.exists(target + ".abi"):
        os.remove(target + ".abi")      # no moment at which the note belongs to another file
    os.replace(tmp, target)
    with open(target + ".abi", "w") as f:
        f.write(abi)


def _build_native(force: bool) -> None:
    """The CPython modules: plain C, and the one compiled against torch (layer.py's)."""
    header = os.path.join(ROOT, "include", "wino.h")
    common = ["-O2", "-Wall", "-Wextra", "-fPIC", "-shared", "-I", sysconfig.get_paths()["include"],
              "-I", os.path.join(ROOT, "include")]
    link = ["-L", HERE, "-l:" + os.path.basename(LIB), "-Wl,-rpath,$ORIGIN"]
    python_abi = sysconfig.get_config_var("SOABI")
    src = os.path.join(CSRC, "wino_python.c")
    if force or _stale(NATIVE, python_abi, src, header):
        tmp = NATIVE + f".tmp{os.getpid()}"
        subprocess.check_call([os.environ.get("CC", "gcc"), "-std=c11", *common, src, *link, "-o", tmp])
        _install(tmp, NATIVE, python_abi)
    import torch
    torch_abi = f"{python_abi} torch {torch.__version__} abi {int(torch._C._GLIBCXX_USE_CXX11_ABI)}"
    src = os.path.join(CSRC, "wino_python_torch.cpp")
    if force or _stale(NATIVE_TORCH, torch_abi, src, header):
        from torch.utils.cpp_extension import include_paths, library_paths
        tmp = NATIVE_TORCH + f".tmp{os.getpid()}"
        cuda = os.path.join(os.path.dirname(os.path.dirname(os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc"))), "include")
        subprocess.check_call(
            [os.environ.get("CXX", "g++"), "-std=c++17", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
             *common, *[f for d in include_paths() for f in ("-isystem", d)], "-isystem", cuda, src, *link,
             *[f for d in library_paths() for f in ("-L", d)], "-lc10", "-lc10_cuda", "-ltorch_cpu", "-ltorch_cuda",
             "-ltorch", "-ltorch_python", "-o", tmp])
        _install(tmp, NATIVE_TORCH, torch_abi)


if __name__ == "__main__":
    import sys
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
