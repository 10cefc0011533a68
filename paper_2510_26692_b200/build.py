"""Build step: compiles the CUDA sources under ``csrc/`` into ``libkda_b200.so`` and the native argument
marshalling of the Python binding (``csrc/marshal.cpp``) into ``_marshal.so`` (both in-tree)."""
from __future__ import annotations

import glob
import os
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libkda_b200.so")
MARSHAL = os.path.join(HERE, "_marshal.so")
MARSHAL_SRC = os.path.join(CSRC, "marshal.cpp")

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
    "-Xcompiler", "-fPIC", "-cudart", "static",
]


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _older(target, deps) -> bool:
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    return any(os.path.getmtime(p) > t for p in deps)


def _headers():
    return glob.glob(os.path.join(ROOT, "include", "*.h")) + [os.path.abspath(__file__)]


def needs_build() -> bool:
    return _older(LIB, sources() + glob.glob(os.path.join(CSRC, "*.cuh")) + _headers())


def marshal_fits() -> bool:
    """Whether ``_marshal.so`` was built for this Python and this torch, by the text it carries."""
    try:
        with open(MARSHAL, "rb") as f:
            return _built_for().encode() in f.read()
    except OSError:
        return False


def _built_for() -> str:
    import torch
    return "kda marshalling for python %d.%d, torch %s;" % (sys.version_info[:2] + (torch.__version__,))


def _build_marshal() -> None:
    import sysconfig

    import torch
    t = os.path.dirname(os.path.abspath(torch.__file__))
    cuda = os.path.dirname(os.path.dirname(os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")))
    tmp = MARSHAL + ".tmp.%d" % os.getpid()
    cmd = [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-fPIC", "-shared",
           "-D_GLIBCXX_USE_CXX11_ABI=%d" % int(torch._C._GLIBCXX_USE_CXX11_ABI),
           "-DKDA_BUILT_FOR=\"%s\"" % _built_for()]
    for d in (os.path.join(t, "include"), os.path.join(t, "include", "torch", "csrc", "api", "include"),
              os.path.join(cuda, "include"), sysconfig.get_paths()["include"], os.path.join(ROOT, "include")):
        cmd += ["-I", d]
    cmd += [MARSHAL_SRC, "-o", tmp, "-L", os.path.join(t, "lib"), "-ltorch_python", "-ltorch_cpu", "-lc10", "-lc10_cuda"]
    subprocess.run(cmd, check=True)
    os.replace(tmp, MARSHAL)


def build(force: bool = False, verbose: bool = False) -> str:
    if force or _older(MARSHAL, [MARSHAL_SRC] + _headers()) or not marshal_fits():
        _build_marshal()
    if not force and not needs_build():
        return LIB
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    tmp = LIB + ".tmp.%d" % os.getpid()
    # one object per source, compiled side by side
    objs, procs = [], []
    for src in sources():
        obj = "%s.%s.o" % (tmp, os.path.basename(src))
        cmd = [nvcc] + NVCC_FLAGS + ["-c", "-I", os.path.join(ROOT, "include"), "-I", CSRC]
        cmd += os.environ.get("KDA_NVCC_EXTRA", "").split()
        if verbose:
            cmd += ["-Xptxas", "-v"]
        objs.append(obj)
        procs.append(subprocess.Popen(cmd + ["-o", obj, src]))
    try:
        if any([p.wait() for p in procs]):
            raise RuntimeError("nvcc failed")
        subprocess.run([nvcc] + NVCC_FLAGS + ["-shared", "-o", tmp] + objs, check=True)
    finally:
        for obj in objs:
            if os.path.exists(obj):
                os.remove(obj)
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
