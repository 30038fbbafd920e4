"""Compile the CUDA sources into paper_2412_14468_b200/libhashattn.so for sm_100a (in-tree), and the native argument
marshalling of the binding into paper_2412_14468_b200/_hostcall.so, which links against it.

Every .cu file becomes an object under csrc/build/ (compiled in parallel, recompiled only when it or a header
changed), then the objects are linked into the shared library.  The marshalling is recompiled as well when torch or Python is
another one than it was compiled against."""
from __future__ import annotations

import glob
import os
import subprocess
import sys
import sysconfig
from concurrent.futures import ThreadPoolExecutor

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
OBJ = os.path.join(CSRC, "build")
LIB = os.path.join(HERE, "libhashattn.so")
HOST_SRC = os.path.join(CSRC, "host", "ha_hostcall.cpp")
HOST_LIB = os.path.join(HERE, "_hostcall.so")
HOST_STAMP = os.path.join(OBJ, "_hostcall.key")     # what HOST_LIB was compiled against

NVCC_FLAGS = [
    "-std=c++17", "-O3", "-lineinfo",
    "-gencode", "arch=compute_100a,code=sm_100a",
    "-Xcompiler", "-fPIC",
    "-I", os.path.join(ROOT, "include"), "-I", CSRC,
]


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _headers():
    return glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(ROOT, "include", "*.h"))


def _obj(src: str) -> str:
    return os.path.join(OBJ, os.path.basename(src)[:-3] + ".o")


def _stale(target: str, deps) -> bool:
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    return any(os.path.getmtime(d) > t for d in deps)


def _hostcall_key() -> str:
    """The headers and the interpreter that the extension module is bound to: it fits no other torch and no other Python."""
    import torch
    return "\n".join([torch.__version__, os.path.dirname(torch.__file__), str(torch._C._GLIBCXX_USE_CXX11_ABI), sys.version,
                      sysconfig.get_paths()["include"]])


def _hostcall_stale() -> bool:
    if _stale(HOST_LIB, [HOST_SRC, os.path.join(ROOT, "include", "hashattn.h")]) or not os.path.exists(HOST_STAMP):
        return True
    with open(HOST_STAMP) as f:
        return f.read() != _hostcall_key()


def _build_hostcall() -> None:
    """The extension module over torch's own C++ headers; g++ is enough, it has no device code."""
    import torch
    root = os.path.dirname(torch.__file__)
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    inc = [os.path.join(ROOT, "include"), os.path.join(root, "include"),
           os.path.join(root, "include", "torch", "csrc", "api", "include"), sysconfig.get_paths()["include"],
           os.path.join(cuda, "include")]
    cmd = [os.environ.get("CXX", "g++"), "-std=c++17", "-O2", "-fPIC", "-shared", HOST_SRC, "-o", HOST_LIB]
    cmd += [x for d in inc for x in ("-I", d)]
    cmd += ["-L", HERE, "-l:" + os.path.basename(LIB), "-L", os.path.join(root, "lib"), "-lc10", "-lc10_cuda", "-ltorch_cpu",
            "-ltorch_python", "-Wl,-rpath,$ORIGIN"]
    subprocess.run(cmd, check=True)
    with open(HOST_STAMP, "w") as f:
        f.write(_hostcall_key())


def build(force: bool = False, verbose: bool = False) -> str:
    nvcc = os.environ.get("NVCC", "nvcc")
    os.makedirs(OBJ, exist_ok=True)
    hdrs = _headers()
    todo = [s for s in sources() if force or _stale(_obj(s), [s] + hdrs)]

    def compile_one(src):
        cmd = [nvcc] + NVCC_FLAGS + (["-Xptxas", "-v"] if verbose else []) + ["-c", src, "-o", _obj(src)]
        subprocess.run(cmd, check=True)

    if todo:
        with ThreadPoolExecutor(max_workers=min(len(todo), os.cpu_count() or 4)) as ex:
            list(ex.map(compile_one, todo))
    objs = [_obj(s) for s in sources()]
    for stale in set(glob.glob(os.path.join(OBJ, "*.o"))) - set(objs):   # objects of sources that no longer exist
        os.remove(stale)
    if todo or force or _stale(LIB, objs):
        subprocess.run([nvcc, "-shared", "-gencode", "arch=compute_100a,code=sm_100a", "-o", LIB] + objs, check=True)
    if force or _hostcall_stale():
        _build_hostcall()
    return LIB


if __name__ == "__main__":
    print(build(force="-f" in sys.argv or "--force" in sys.argv, verbose="-v" in sys.argv))
