"""Builds libgsd.so (the C-ABI CUDA library, nvcc for sm_100a) and the CPython extension that
marshals the calls, both in-tree."""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig
from concurrent.futures import ThreadPoolExecutor

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
LIB = os.path.join(PKG, "libgsd.so")
LIB_CHECK = os.path.join(PKG, "libgsd_check.so")
NATIVE = os.path.join(PKG, "_native.so")
OBJ_DIR = os.path.join(PKG, "_build")
SOURCES = ["gsd_api.cu", "gsd_accept.cu", "gsd_accept_sampled.cu", "gsd_draft.cu", "gsd_attn_mma.cu", "gsd_attn_tc.cu", "gsd_attn_plan.cu", "gsd_attn_merge.cu", "gsd_commit.cu", "gsd_mask.cu", "gsd_unmerge.cu"]
NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-O3", "-std=c++17", "-lineinfo",
              "-Xcompiler", "-fPIC", "-I", os.path.join(ROOT, "include"), "-I", CSRC]


def _nvcc() -> str:
    for cand in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    return "nvcc"


def _stale(target: str, deps) -> bool:
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    return any(os.path.getmtime(d) > t for d in deps)


def build_native(force: bool = False) -> str:
    """Compile csrc/gsd_native.cpp (host code only) against the installed torch and CPython."""
    import torch
    src = os.path.join(CSRC, "gsd_native.cpp")
    built_for = os.path.join(OBJ_DIR, "native_torch_version")
    same = os.path.exists(built_for) and open(built_for).read() == torch.__version__
    if not force and same and not _stale(NATIVE, [src, os.path.join(CSRC, "gsd_binding.h"), os.path.join(ROOT, "include", "gsd.h")]):
        return NATIVE
    os.makedirs(OBJ_DIR, exist_ok=True)
    base = os.path.dirname(torch.__file__)
    cuda = os.path.dirname(os.path.dirname(_nvcc())) if os.path.sep in _nvcc() else "/usr/local/cuda"
    tmp = NATIVE + f".tmp{os.getpid()}"
    cmd = [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-fPIC", "-shared",
           f'-DGSD_TORCH_VERSION="{torch.__version__}"', f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
           "-I", os.path.join(ROOT, "include"), "-I", CSRC, "-isystem", os.path.join(base, "include"),
           "-isystem", os.path.join(base, "include", "torch", "csrc", "api", "include"),
           "-isystem", os.path.join(cuda, "include"), "-isystem", sysconfig.get_paths()["include"],
           src, "-o", tmp, "-L", os.path.join(base, "lib"), "-Wl,-rpath," + os.path.join(base, "lib"),
           "-ltorch_python", "-ltorch_cpu", "-lc10_cuda", "-lc10"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        sys.stderr.write(r.stdout + r.stderr)
        raise RuntimeError("c++ failed: " + " ".join(cmd))
    os.replace(tmp, NATIVE)
    with open(built_for, "w") as f:
        f.write(torch.__version__)
    return NATIVE


def build(force: bool = False, verbose: bool = False, checked: bool = False) -> str:
    """Compile the sources that changed and link libgsd.so next to this file.  With `checked`
    the same sources are compiled with -DGSD_BOUNDS_CHECK into libgsd_check.so: the build whose
    kernels check the indices they form and report GSD_DEV_BOUNDS instead of accessing memory
    outside a tensor (used by the tests in place of a memory sanitizer)."""
    obj_dir = OBJ_DIR + ("_check" if checked else "")
    lib = LIB_CHECK if checked else LIB
    extra = ["-DGSD_BOUNDS_CHECK"] if checked else []
    os.makedirs(obj_dir, exist_ok=True)
    headers = [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith((".cuh", ".h"))]
    headers.append(os.path.join(ROOT, "include", "gsd.h"))
    jobs, objs = [], []
    for src in SOURCES:
        s = os.path.join(CSRC, src)
        o = os.path.join(obj_dir, src.replace(".cu", ".o"))
        objs.append(o)
        if force or _stale(o, [s] + headers):
            jobs.append([_nvcc()] + NVCC_FLAGS + extra + (["-Xptxas", "-v"] if verbose else [])
                        + ["-c", s, "-o", o])

    def run(cmd):
        r = subprocess.run(cmd, capture_output=True, text=True)
        if verbose or r.returncode != 0:
            sys.stderr.write(r.stdout + r.stderr)
        if r.returncode != 0:
            raise RuntimeError("nvcc failed: " + " ".join(cmd))

    with ThreadPoolExecutor(max_workers=4) as ex:
        list(ex.map(run, jobs))
    if force or jobs or _stale(lib, objs):
        tmp = lib + f".tmp{os.getpid()}"
        run([_nvcc(), "-shared", "-o", tmp] + objs
            + ["-gencode", "arch=compute_100a,code=sm_100a", "-Xcompiler", "-fPIC"])
        os.replace(tmp, lib)
    return lib


if __name__ == "__main__":
    print(build_native(force="--force" in sys.argv))
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv, checked="--checked" in sys.argv))
