"""Builds, in-tree, the CUDA library with nvcc for sm_100a and the CPython extension that marshals its arguments with g++
(no JIT cache)."""
from __future__ import annotations

import os
import shutil
import subprocess
import sys

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
LIB = os.path.join(PKG, "libspectre.so")
NATIVE = os.path.join(PKG, "_native.so")
NATIVE_SRC = os.path.join(CSRC, "native.cpp")
OBJ = os.path.join(PKG, "build")
NATIVE_ABI = os.path.join(OBJ, "native_abi")
SOURCES = ["reg_grad.cu", "reg_mix.cu", "reg_inverse.cu", "reg_forward.cu", "api.cu", "mixer.cu", "mixer_tc.cu", "mixer_tc64.cu",
           "mixer_tc4k.cu", "gate.cu", "cache.cu", "wavelet.cu", "backward.cu", "project.cu"]
FLAGS = ["-std=c++17", "-O3", "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo",
         "-Xcompiler", "-fPIC", "-shared"]


def _nvcc() -> str:
    exe = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(exe):
        raise RuntimeError("nvcc not found; the library cannot be built")
    return exe


def sources() -> list[str]:
    extra = sorted(f for f in os.listdir(CSRC) if f.endswith(".cu") and f not in SOURCES)
    return [os.path.join(CSRC, f) for f in SOURCES + extra]


def is_stale() -> bool:
    if not os.path.exists(LIB):
        return True
    t = os.path.getmtime(LIB)
    deps = sources() + [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith((".cuh", ".h"))]
    deps.append(os.path.join(ROOT, "include", "spectre.h"))
    return any(os.path.getmtime(d) > t for d in deps)


def _compile(src: str, obj: str, verbose: bool) -> str:
    cmd = [_nvcc()] + [f for f in FLAGS if f != "-shared"] + ["-I", os.path.join(ROOT, "include"), "-I", CSRC, "-c", "-o", obj, src]
    if verbose:
        cmd[1:1] = ["-Xptxas", "-v"]
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        raise RuntimeError("nvcc failed on " + src + ":\n" + res.stdout + res.stderr)
    return res.stderr


def native_abi() -> str:
    """What the extension is compiled against beside its sources: another torch or Python has another ABI."""
    import sysconfig

    import torch
    return f"torch {torch.__version__} {sysconfig.get_config_var('SOABI')}"


def native_is_stale() -> bool:
    if not os.path.exists(NATIVE) or not os.path.exists(NATIVE_ABI):
        return True
    with open(NATIVE_ABI) as f:
        if f.read() != native_abi():
            return True
    return os.path.getmtime(NATIVE) < max(os.path.getmtime(f) for f in (NATIVE_SRC, os.path.join(ROOT, "include", "spectre.h")))


def build_native(force: bool = False) -> str:
    """The extension links against torch's libraries (loaded with torch itself) and, by $ORIGIN, against libspectre.so."""
    if not force and not native_is_stale():
        return NATIVE
    import sysconfig

    import torch
    t = os.path.dirname(torch.__file__)
    cmd = ["g++", "-std=c++17", "-O2", "-fPIC", "-shared", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
           "-I", os.path.join(ROOT, "include"), "-I", os.path.join(t, "include"),
           "-I", os.path.join(t, "include", "torch", "csrc", "api", "include"), "-I", "/usr/local/cuda/include",
           "-I", sysconfig.get_paths()["include"], "-o", NATIVE, NATIVE_SRC, "-L", os.path.join(t, "lib"), "-ltorch_python", "-ltorch",
           "-ltorch_cpu", "-ltorch_cuda", "-lc10", "-lc10_cuda", "-L", PKG, "-l:libspectre.so", "-Wl,-rpath,$ORIGIN"]
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        raise RuntimeError("g++ failed on " + NATIVE_SRC + ":\n" + res.stdout + res.stderr)
    os.makedirs(OBJ, exist_ok=True)
    with open(NATIVE_ABI, "w") as f:
        f.write(native_abi())
    return NATIVE


def build(force: bool = False, verbose: bool = False) -> str:
    """The library, then the extension over it."""
    lib = build_library(force, verbose)
    build_native(force)
    return lib


def build_library(force: bool = False, verbose: bool = False) -> str:
    """One object per source file (compiled side by side, only the stale ones), then one link."""
    if not force and not is_stale():
        return LIB
    from concurrent.futures import ThreadPoolExecutor
    os.makedirs(OBJ, exist_ok=True)
    headers = [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith((".cuh", ".h"))]
    headers.append(os.path.join(ROOT, "include", "spectre.h"))
    newest_header = max(os.path.getmtime(h) for h in headers)
    jobs, objs = [], []
    for src in sources():
        obj = os.path.join(OBJ, os.path.basename(src)[:-3] + ".o")
        objs.append(obj)
        if force or verbose or not os.path.exists(obj) or os.path.getmtime(obj) < max(os.path.getmtime(src), newest_header):
            jobs.append((src, obj))
    with ThreadPoolExecutor(max_workers=max(1, min(len(jobs), os.cpu_count() or 1))) as pool:
        logs = list(pool.map(lambda j: _compile(j[0], j[1], verbose), jobs))
    if verbose:
        print("".join(logs))
    res = subprocess.run([_nvcc(), "-shared", "-gencode", "arch=compute_100a,code=sm_100a", "-o", LIB] + objs,
                         capture_output=True, text=True)
    if res.returncode != 0:
        raise RuntimeError("link failed:\n" + res.stdout + res.stderr)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
