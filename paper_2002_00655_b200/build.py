"""Builds the CUDA library in-tree for sm_100a (Blackwell B200) with nvcc.

`python -m paper_2002_00655_b200.build` compiles every `csrc/*.cu` into
`libps_b200.so` next to this file.  The library is plain C-ABI (include/ps.h);
it links the CUDA runtime statically and depends on nothing else.  Beside it,
`csrc/native.cpp` becomes `_native`, the part of the Python binding that is
called per batch (it links torch, whose tensors it takes).
"""
from __future__ import annotations

import glob
import os
import shutil
import subprocess
import sys
import sysconfig
from concurrent.futures import ThreadPoolExecutor

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
OBJ = os.path.join(PKG, "_build")
LIB = os.path.join(PKG, "libps_b200.so")

NATIVE = os.path.join(PKG, "_native" + sysconfig.get_config_var("EXT_SUFFIX"))

NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "-Xcompiler", "-fPIC", "-I", os.path.join(ROOT, "include"), "-I", CSRC]


def _nvcc() -> str:
    for cand in (shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found: the CUDA library cannot be built")


def _stale(target: str, deps) -> bool:
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    return any(os.path.getmtime(d) > t for d in deps)


def build(force: bool = False, verbose: bool = False) -> str:
    nvcc = _nvcc()
    os.makedirs(OBJ, exist_ok=True)
    sources = sorted(glob.glob(os.path.join(CSRC, "*.cu")))
    headers = glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(ROOT, "include", "*.h"))
    extra = ["-Xptxas", "-v"] if verbose else []

    def compile_one(src):
        obj = os.path.join(OBJ, os.path.basename(src)[:-3] + ".o")
        if force or verbose or _stale(obj, [src] + headers):
            out = subprocess.run([nvcc, *NVCC_FLAGS, *extra, "-c", src, "-o", obj], capture_output=True, text=True)
            if out.returncode != 0:
                raise RuntimeError(f"nvcc failed on {src}:\n{out.stdout}\n{out.stderr}")
            if verbose:
                sys.stderr.write(out.stderr)
        return obj

    with ThreadPoolExecutor(max_workers=5) as pool:
        native = pool.submit(build_native, force)
        objs = list(pool.map(compile_one, sources))
        native.result()
    if force or _stale(LIB, objs):
        tmp = LIB + f".tmp{os.getpid()}"
        subprocess.check_call([nvcc, "-shared", "-o", tmp, *objs, "-gencode", "arch=compute_100a,code=sm_100a"])
        os.replace(tmp, LIB)
    return LIB


def _built_for(path: str, version: str) -> bool:
    """Was the module built for this torch?  (It carries the version it was compiled against.)"""
    with open(path, "rb") as f:
        return b"\0" + version.encode() + b"\0" in f.read()


def build_native(force: bool = False) -> str:
    src = os.path.join(CSRC, "native.cpp")
    import torch
    if not force and not _stale(NATIVE, [src, os.path.join(ROOT, "include", "ps.h")]) and _built_for(NATIVE, torch.__version__):
        return NATIVE
    troot = os.path.dirname(torch.__file__)
    cuda = os.path.dirname(os.path.dirname(os.path.realpath(_nvcc())))
    inc = [os.path.join(ROOT, "include"), os.path.join(troot, "include"),
           os.path.join(troot, "include", "torch", "csrc", "api", "include"), sysconfig.get_paths()["include"],
           os.path.join(cuda, "include")]
    tmp = NATIVE + f".tmp{os.getpid()}"
    cmd = ["g++", "-shared", "-fPIC", "-O2", "-std=c++17", "-Wall", "-Wextra", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
           f'-DPS_TORCH_VERSION="{torch.__version__}"',
           *(x for i in inc for x in ("-isystem", i)), src, "-o", tmp, "-L", os.path.join(troot, "lib"),
           "-lc10", "-lc10_cuda", "-ltorch_cpu", "-ltorch_python"]
    out = subprocess.run(cmd, capture_output=True, text=True)
    if out.returncode != 0:
        raise RuntimeError(f"g++ failed on {src}:\n{out.stdout}\n{out.stderr}")
    os.replace(tmp, NATIVE)
    return NATIVE


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
