"""Builds ``libkvq.so`` in-tree with nvcc for sm_100a (cross-compiles without a GPU).

    python -m paper_2605_05699_b200.build [--force]
"""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig
import warnings
from concurrent.futures import ThreadPoolExecutor

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
OBJ = os.path.join(HERE, "_build")
LIB = os.path.join(HERE, "libkvq.so")
CALL_SRC = os.path.join(CSRC, "kvq_call.cpp")
# the binding's native half: a Python extension on torch's own headers and libraries, good for the Python in its name and the torch it says
CALL = os.path.join(HERE, "kvq_call" + sysconfig.get_config_var("EXT_SUFFIX"))
INCLUDE = os.path.join(os.path.dirname(HERE), "include")

NVCC_FLAGS = [
    "-std=c++17", "-O3", "-lineinfo", "--expt-relaxed-constexpr",
    "-gencode", "arch=compute_100a,code=sm_100a",
    "-Xcompiler", "-fPIC", "-Xptxas", "-v",
]


def _sources():
    return sorted(f for f in os.listdir(CSRC) if f.endswith(".cu"))


def _deps_mtime():
    m = 0.0
    for d in (CSRC, INCLUDE):
        for f in os.listdir(d):
            if f.endswith((".cu", ".cuh", ".h")):
                m = max(m, os.path.getmtime(os.path.join(d, f)))
    return m


def _compile(src: str, force: bool, newest: float) -> str:
    obj = os.path.join(OBJ, src[:-3] + ".o")
    if not force and os.path.exists(obj) and os.path.getmtime(obj) >= newest:
        return obj
    cmd = ["nvcc", *NVCC_FLAGS, "-I", INCLUDE, "-c", os.path.join(CSRC, src), "-o", obj]
    res = subprocess.run(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)
    with open(obj + ".log", "w") as f:
        f.write(" ".join(cmd) + "\n" + res.stdout)
    if res.returncode:
        sys.stderr.write(res.stdout)
        raise RuntimeError("nvcc failed on %s" % src)
    return obj


def _build_call(force: bool) -> None:
    import torch

    stamp = os.path.join(OBJ, os.path.basename(CALL) + ".torch")   # the torch that CALL was compiled against
    built_for = None
    if os.path.exists(CALL) and os.path.exists(stamp):
        with open(stamp) as f:
            built_for = f.read()
    if not force and built_for == torch.__version__ and os.path.getmtime(CALL) >= max(os.path.getmtime(CALL_SRC), os.path.getmtime(os.path.join(INCLUDE, "kvq.h"))):
        return
    root = os.path.dirname(torch.__file__)
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    tmp = CALL + ".tmp.%d" % os.getpid()
    try:
        subprocess.check_call([
            "g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-D_GLIBCXX_USE_CXX11_ABI=%d" % int(torch._C._GLIBCXX_USE_CXX11_ABI),
            '-DKVQ_TORCH="%s"' % torch.__version__,
            "-I", os.path.join(root, "include"), "-I", os.path.join(root, "include", "torch", "csrc", "api", "include"),
            "-I", sysconfig.get_paths()["include"], "-I", os.path.join(cuda, "include"), CALL_SRC, "-o", tmp,
            "-L", os.path.join(root, "lib"), "-lc10", "-lc10_cuda", "-ltorch_cpu", "-ltorch_python"])
    except Exception:
        if os.path.exists(CALL):   # out of date: not left behind
            os.remove(CALL)
        raise
    os.replace(tmp, CALL)
    with open(stamp, "w") as f:
        f.write(torch.__version__)


def _build_library(force: bool) -> str:
    os.makedirs(OBJ, exist_ok=True)
    newest = _deps_mtime()
    srcs = _sources()
    if not force and os.path.exists(LIB) and os.path.getmtime(LIB) >= newest:
        return LIB
    with ThreadPoolExecutor(max_workers=min(8, len(srcs))) as ex:
        objs = list(ex.map(lambda s: _compile(s, force, newest), srcs))
    tmp = LIB + ".tmp.%d" % os.getpid()
    subprocess.check_call(["nvcc", "-shared", "-o", tmp, *objs, "-gencode", "arch=compute_100a,code=sm_100a"])
    os.replace(tmp, LIB)
    return LIB


def build(force: bool = False) -> str:
    """The library; then the binding's native half, which the library does not need: what it lacks (g++, torch or Python headers) is a
    warning, and calls take the binding's general way."""
    path = _build_library(force)
    try:
        _build_call(force)
    except Exception as e:
        warnings.warn("kvq_call has not been built, calls from Python take the general way: %s" % e, RuntimeWarning, stacklevel=2)
    return path


if __name__ == "__main__":
    print(build(force="--force" in sys.argv))
