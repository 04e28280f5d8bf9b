"""Builds libl4l.so (the C-ABI library) in-tree with nvcc for sm_100a.

Run as ``python -m paper_2608_21836_b200.build``. nvcc cross-compiles, so no GPU is needed.
"""
from __future__ import annotations

import os
import shutil
import subprocess
import sys
import sysconfig
from concurrent.futures import ThreadPoolExecutor

PKG = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(PKG, "csrc")
OBJ = os.path.join(PKG, "csrc", "build")
LIB = os.path.join(PKG, "libl4l.so")
# the Python module that marshals the per-step calls: for one interpreter (by its name) and one torch (by its tag)
MARSHAL = os.path.join(PKG, "_l4l_marshal" + sysconfig.get_config_var("EXT_SUFFIX"))
MARSHAL_FLAGS = ["-O2", "-std=c++17", "-fPIC", "-shared"]

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
    "-Xcompiler", "-fPIC", "-Wno-deprecated-gpu-targets",
]


def sources():
    return sorted(f for f in os.listdir(CSRC) if f.endswith(".cu"))


def _stale(target: str, deps) -> bool:
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    return any(os.path.getmtime(d) > t for d in deps)


MARSHAL_SRC = [os.path.join(CSRC, "l4l_marshal.cpp"), os.path.join(PKG, "..", "include", "l4l.h")]


def marshal_tag() -> str:
    """What the module's layout of tensors and of the interpreter depends on; compiled into it, and compared when it is loaded."""
    import torch

    return f"torch {torch.__version__}, {sysconfig.get_config_var('SOABI')}, {' '.join(MARSHAL_FLAGS)}"


def marshal_is_stale() -> bool:
    if _stale(MARSHAL, MARSHAL_SRC):
        return True
    with open(MARSHAL, "rb") as f:
        return marshal_tag().encode() not in f.read()


def build(force: bool = False, verbose: bool = False) -> str:
    os.makedirs(OBJ, exist_ok=True)
    headers = [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith((".cuh", ".h"))]
    headers.append(os.path.join(PKG, "..", "include", "l4l.h"))
    jobs = []
    objs = []
    for src in sources():
        s = os.path.join(CSRC, src)
        o = os.path.join(OBJ, src[:-3] + ".o")
        objs.append(o)
        if force or _stale(o, [s] + headers):
            cmd = ["nvcc"] + NVCC_FLAGS + (["-Xptxas", "-v"] if verbose else []) + ["-c", s, "-o", o]
            jobs.append(cmd)

    def run(cmd):
        r = subprocess.run(cmd, capture_output=True, text=True)
        if verbose or r.returncode != 0:
            sys.stderr.write(r.stdout + r.stderr)
        if r.returncode != 0:
            raise RuntimeError("nvcc failed: " + " ".join(cmd))

    with ThreadPoolExecutor(max_workers=min(8, max(1, len(jobs)))) as ex:
        list(ex.map(run, jobs))
    if force or jobs or _stale(LIB, objs):
        tmp = LIB + f".tmp{os.getpid()}"
        run(["nvcc", "-shared", "-Wno-deprecated-gpu-targets", "-o", tmp] + objs)
        os.replace(tmp, LIB)
    if force or marshal_is_stale():
        import torch

        home = os.path.dirname(torch.__file__)
        cuda = os.path.dirname(os.path.dirname(os.path.realpath(shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc")))
        tmp = MARSHAL + f".tmp{os.getpid()}"
        run(["g++", *MARSHAL_FLAGS, f"-D_GLIBCXX_USE_CXX11_ABI={int(torch.compiled_with_cxx11_abi())}", f'-DL4L_BUILT_FOR="{marshal_tag()}"',
             f"-I{home}/include", f"-I{home}/include/torch/csrc/api/include", f"-I{cuda}/include",
             "-I" + sysconfig.get_paths()["include"], MARSHAL_SRC[0], "-o", tmp, f"-L{PKG}", "-l:libl4l.so", f"-L{home}/lib",
             "-ltorch_python", "-ltorch", "-ltorch_cpu", "-lc10", "-lc10_cuda", "-Wl,-rpath,$ORIGIN"])
        os.replace(tmp, MARSHAL)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
