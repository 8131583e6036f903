"""Builds libbsp.so (the C-ABI CUDA library) in-tree with nvcc for sm_100a.

Every .cu under csrc/ is compiled to an object of its own (in parallel, rebuilt only when it or a header is
newer) under _build/, then the objects are linked into paper_2407_09453_b200/libbsp.so.  The marshalling of the Python
calls, csrc/bsp_call.cpp, is compiled by the host compiler into paper_2407_09453_b200/_bspcall.so.
"""
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
OBJ = os.path.join(HERE, "_build")
LIB = os.path.join(HERE, "libbsp.so")
CALL_SOURCE = os.path.join(CSRC, "bsp_call.cpp")
CALL = os.path.join(HERE, "_bspcall.so")


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _headers():
    return glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(ROOT, "include", "*.h"))


def _newer(deps, target) -> bool:
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    return any(os.path.getmtime(d) > t for d in deps)


def _stale() -> bool:
    return _newer(sources() + _headers(), LIB)


def _flags(verbose: bool):
    f = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
         "-I" + os.path.join(ROOT, "include"), "-Xcompiler", "-fPIC"]
    if verbose:
        f += ["-Xptxas", "-v"]
    return f


def call_stamp() -> str:
    """What the marshalling is compiled against: it reads tensors in place, so another PyTorch or Python needs another build."""
    import torch
    return "%s %s %d" % (torch.__version__, sysconfig.get_config_var("SOABI"), int(torch.compiled_with_cxx11_abi()))


def call_is_current() -> bool:
    """Whether the built marshalling is one for the Python and PyTorch that run: the stamp stands behind the file's own contents."""
    stamp = call_stamp().encode()
    try:
        with open(CALL, "rb") as f:
            f.seek(0, os.SEEK_END)
            f.seek(max(0, f.tell() - len(stamp) - 1))
            return f.read() == b"\n" + stamp
    except OSError:
        return False


def build_call(force: bool = False) -> str:
    """Compile the marshalling of the Python calls against the installed Python and PyTorch; returns its path."""
    if not force and call_is_current() and not _newer([CALL_SOURCE] + _headers(), CALL):
        return CALL
    import torch
    root = os.path.dirname(os.path.abspath(torch.__file__))
    cuda = os.path.dirname(os.path.dirname(os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")))
    include = [os.path.join(ROOT, "include"), sysconfig.get_paths()["include"], os.path.join(root, "include"), os.path.join(cuda, "include")]
    tmp = CALL + ".tmp%d" % os.getpid()
    subprocess.check_call([os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-shared", "-fPIC",
                           "-D_GLIBCXX_USE_CXX11_ABI=%d" % int(torch.compiled_with_cxx11_abi())] + ["-I" + d for d in include] +
                          [CALL_SOURCE, "-o", tmp, "-L" + os.path.join(root, "lib"), "-ltorch_python", "-lc10", "-lc10_cuda"])
    with open(tmp, "ab") as f:
        f.write(b"\n" + call_stamp().encode())
    os.replace(tmp, CALL)
    return CALL


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile every .cu under csrc/ and link them into one shared library; returns its path.  Builds the marshalling too."""
    build_call(force)
    if not force and not _stale():
        return LIB
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    os.makedirs(OBJ, exist_ok=True)
    hdrs = _headers()
    jobs = []
    for src in sources():
        obj = os.path.join(OBJ, os.path.basename(src)[:-3] + ".o")
        if force or verbose or _newer([src] + hdrs, obj):
            jobs.append([nvcc] + _flags(verbose) + ["-c", src, "-o", obj])

    def run(cmd):
        subprocess.check_call(cmd)

    with ThreadPoolExecutor(max_workers=max(1, min(len(jobs), os.cpu_count() or 1))) as ex:
        list(ex.map(run, jobs))
    objs = [os.path.join(OBJ, os.path.basename(s)[:-3] + ".o") for s in sources()]
    tmp = LIB + ".tmp%d" % os.getpid()
    subprocess.check_call([nvcc, "-gencode", "arch=compute_100a,code=sm_100a", "-shared", "-o", tmp] + objs)
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
