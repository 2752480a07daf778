"""In-tree build of libxpiler_repair.so for sm_100a with nvcc (no JIT cache is used)."""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libxpiler_repair.so")
LIB_CHECKED = os.path.join(HERE, "libxpiler_repair_checked.so")       # the same sources with -DXP_CHECKS (index checks)
LIB_MARSHAL = os.path.join(HERE, "_marshal.so")                       # CPython extension of the binding (csrc/xp_marshal.c)
SOURCES = ["xp_api.cu", "xp_kernels.cu", "xp_pair.cu", "xp_joint.cu", "xp_behaviour.cu"]
FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
         "-Xcompiler", "-fPIC", "-I" + os.path.join(ROOT, "include"), "-I" + CSRC]


def _stale(lib: str = LIB) -> bool:
    if not os.path.exists(lib):
        return True
    t = os.path.getmtime(lib)
    deps = [os.path.join(CSRC, f) for f in os.listdir(CSRC)] + [os.path.join(ROOT, "include", "xp.h"), __file__]
    return any(os.path.getmtime(d) > t for d in deps)


def build_marshal(force: bool = False) -> str:
    """Compiles the binding's CPython extension next to this file; returns its path."""
    src = os.path.join(CSRC, "xp_marshal.c")
    deps = [src, os.path.join(ROOT, "include", "xp.h")]
    if not force and os.path.exists(LIB_MARSHAL) and all(os.path.getmtime(d) <= os.path.getmtime(LIB_MARSHAL) for d in deps):
        return LIB_MARSHAL
    tmp = LIB_MARSHAL + f".{os.getpid()}.tmp"
    subprocess.check_call(["gcc", "-O2", "-fPIC", "-shared", "-std=gnu11", "-I" + sysconfig.get_paths()["include"],
                           "-I" + os.path.join(ROOT, "include"), src, "-o", tmp])
    os.replace(tmp, LIB_MARSHAL)
    return LIB_MARSHAL


def build(force: bool = False, verbose: bool = False, checked: bool = False) -> str:
    """Compiles the CUDA sources into the shared library next to this file; returns its path.
    ``checked``: the variant with index checks compiled in (a library of its own beside the normal one)."""
    LIB = LIB_CHECKED if checked else globals()["LIB"]
    build_marshal(force)
    if not force and not _stale(LIB):
        return LIB
    objs = []
    procs = []
    for src in SOURCES:
        obj = os.path.join(CSRC, src.replace(".cu", ".checked.o" if checked else ".o"))
        cmd = ["nvcc", *FLAGS, *(["-DXP_CHECKS"] if checked else []), "-c", os.path.join(CSRC, src), "-o", obj]
        if verbose:
            cmd.insert(1, "-Xptxas"); cmd.insert(2, "-v")
        procs.append((src, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)))
        objs.append(obj)
    for src, p in procs:
        out, _ = p.communicate()
        if verbose or p.returncode:
            sys.stderr.write(out)
        if p.returncode:
            raise RuntimeError(f"nvcc failed on {src}")
    tmp = LIB + f".{os.getpid()}.tmp"
    subprocess.check_call(["nvcc", "-gencode", "arch=compute_100a,code=sm_100a", "-shared", "-o", tmp, *objs])
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv, checked="--checked" in sys.argv))
