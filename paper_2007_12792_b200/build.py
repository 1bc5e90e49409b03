"""Builds ``libdn.so`` (the C-ABI CUDA library) in-tree with nvcc for sm_100a.

    python -m paper_2007_12792_b200.build [--force] [--verbose]
"""
from __future__ import annotations

import os
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libdn.so")
NATIVE = os.path.join(HERE, "_native.so")      # native marshalling for Python (dn_py.cpp), linked to libdn.so
# (source, object name, extra flags): the 2D marching kernel and the mirrored-pair 3D kernel are compiled in parts (their template
# instantiations for different numbers of KL modes), which run side by side
SOURCES = [(f, f.replace(".cu", ".o"), []) for f in
           ["dn_api.cu", "dn_aux.cu", "dn_generic.cu", "dn_tiled2d.cu", "dn_march2d.cu", "dn_tiled3d.cu",
            "dn_pair3d.cu", "dn_strip3d.cu", "dn_static.cu", "dn_burgers.cu", "dn_cg.cu",
            "dn_multigrid.cu"]]
SOURCES += [("dn_march2d.cu", f"dn_march2d_{k}.o", [f"-DDN_M2_PART={k}"]) for k in (1, 2, 3)]
SOURCES += [("dn_pair3d.cu", f"dn_pair3d_{k}.o", [f"-DDN_P3_PART={k}"]) for k in (1, 2, 3)]
HEADERS = [os.path.join(CSRC, "dn_internal.cuh"), os.path.join(ROOT, "include", "dn.h")]
NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "-Xcompiler", "-fPIC", "-I" + os.path.join(ROOT, "include"), "-I" + CSRC]


def _native_command():
    import sysconfig
    import torch
    from torch.utils import cpp_extension
    lib = os.path.join(os.path.dirname(torch.__file__), "lib")
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    inc = [sysconfig.get_paths()["include"], os.path.join(ROOT, "include"), os.path.join(cuda, "include")] + cpp_extension.include_paths()
    return (["g++", "-O2", "-std=c++17", "-fPIC", "-shared", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}", "-w"]
            + ["-I" + i for i in inc] + [os.path.join(CSRC, "dn_py.cpp"), "-o", NATIVE, "-L" + lib, "-L" + HERE]
            + ["-ltorch_python", "-ltorch", "-ltorch_cpu", "-lc10", "-lc10_cuda", "-l:libdn.so", "-Wl,-rpath,$ORIGIN", "-Wl,-rpath," + lib])


def _stale(target, deps):
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    return any(os.path.getmtime(d) > t for d in deps)


def build(force: bool = False, verbose: bool = False) -> str:
    nvcc = os.environ.get("NVCC", "nvcc")
    objdir = os.path.join(HERE, "_build")
    os.makedirs(objdir, exist_ok=True)
    objs = []
    procs = []
    for src, objname, extra in SOURCES:
        path = os.path.join(CSRC, src)
        obj = os.path.join(objdir, objname)
        objs.append(obj)
        if force or _stale(obj, [path] + HEADERS):
            cmd = [nvcc] + NVCC_FLAGS + extra + (["-Xptxas", "-v"] if verbose else []) + ["-c", path, "-o", obj]
            procs.append((objname, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)))
    failed = False
    for src, p in procs:
        out, _ = p.communicate()
        if p.returncode != 0 or verbose:
            sys.stderr.write(f"--- {src}\n{out}\n")
        failed |= p.returncode != 0
    if failed:
        raise RuntimeError("nvcc failed")
    if force or procs or _stale(LIB, objs):
        subprocess.run([nvcc, "-shared", "-o", LIB] + objs + ["-lcudart"], check=True)
    if force or _stale(NATIVE, [os.path.join(CSRC, "dn_py.cpp"), HEADERS[1]]):
        subprocess.run(_native_command(), check=True)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="--verbose" in sys.argv))
