"""Compile libspeca.so (the CUDA library behind the C ABI) for sm_100a with nvcc, and the binding's argument
marshalling (against torch's headers, speca_marshal.*.so) with the host compiler.

Run as ``python -m paper_2607_16673_b200.build``.  The shared objects are written
next to this file, so they travel with the source tree.  nvcc cross-compiles without a GPU.
"""
from __future__ import annotations

import os
import shutil
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libspeca.so")
SOURCES = ["api.cu", "plan.cu", "serial.cu", "commit_mma.cu", "direct.cu", "factorized.cu", "effective.cu"]
ARCH = ["-gencode", "arch=compute_100a,code=sm_100a"]


def _nvcc() -> str:
    for cand in (os.environ.get("NVCC"), shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found")


def _newest_source_mtime() -> float:
    deps = [os.path.join(CSRC, f) for f in os.listdir(CSRC)]
    deps.append(os.path.join(os.path.dirname(HERE), "include", "speca.h"))
    return max(os.path.getmtime(d) for d in deps)


def _start_marshal(tmp: str) -> subprocess.Popen:
    import sysconfig

    from torch.utils import cpp_extension
    cuda = os.path.dirname(os.path.dirname(os.path.realpath(_nvcc())))
    inc = [sysconfig.get_paths()["include"], *cpp_extension.include_paths(), os.path.join(cuda, "include")]
    cmd = [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-fPIC", "-shared", "-DUSE_CUDA", *[f"-I{d}" for d in inc],
           os.path.join(CSRC, "marshal.cpp"), "-o", tmp, *[f"-L{d}" for d in cpp_extension.library_paths()],
           "-lc10", "-lc10_cuda", "-ltorch_cpu", "-ltorch_python"]
    return subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)


def build(force: bool = False, verbose: bool = False) -> str:
    from .binding import MARSHAL_PATH as MARSHAL               # named after this Python and this torch
    newest = _newest_source_mtime()
    if not force and all(os.path.exists(f) and os.path.getmtime(f) >= newest for f in (LIB, MARSHAL)):
        return LIB
    nvcc = _nvcc()
    marshal_tmp = MARSHAL + f".tmp{os.getpid()}"
    marshal = _start_marshal(marshal_tmp)
    objdir = os.path.join(HERE, "build")
    os.makedirs(objdir, exist_ok=True)
    # no --use_fast_math: IEEE fp32 arithmetic everywhere, parity is judged on it
    flags = ["-O3", "-std=c++17", "-lineinfo", "-Xcompiler", "-fPIC"] + ARCH
    if verbose:
        flags += ["-Xptxas", "-v"]
    flags += os.environ.get("SPECA_NVCC_FLAGS", "").split()
    objs = []
    procs = []
    for src in SOURCES:
        obj = os.path.join(objdir, src.replace(".cu", ".o"))
        objs.append(obj)
        procs.append((src, subprocess.Popen([nvcc, *flags, "-c", os.path.join(CSRC, src), "-o", obj],
                                            stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)))
    failed = False
    for src, pr in procs + [("marshal.cpp", marshal)]:
        out, _ = pr.communicate()
        if out.strip():
            print(f"--- {src}\n{out}", file=sys.stderr)
        failed |= pr.returncode != 0
    if failed:
        raise RuntimeError("compilation failed")
    tmp = LIB + f".tmp{os.getpid()}"
    subprocess.run([nvcc, "-shared", *ARCH, "-o", tmp, *objs, "-lcudart"], check=True)
    os.replace(marshal_tmp, MARSHAL)
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
