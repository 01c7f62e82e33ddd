"""Builds the C-ABI CUDA library (libsaki.so) in-tree with nvcc for sm_100a, and the tensor side of the Python
binding (_saki_torch.so) with the host compiler.

    python -m paper_2609_36601_b200.build [--verbose]
"""
from __future__ import annotations

import os
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libsaki.so")
TORCH_SOURCE = os.path.join(CSRC, "saki_torch.cpp")
TORCH_LIB = os.path.join(HERE, "_saki_torch.so")
SOURCES = ("saki_api.cu", "saki_general.cu", "saki_cluster.cu", "saki_rowsm.cu", "saki_rowsm_half.cu", "saki_rowsm_quarter.cu", "saki_rowsm_pair.cu", "saki_rowsm_wide.cu", "saki_meta.cu",
           "saki_select.cu", "saki_propose.cu", "saki_vshard.cu", "saki_lmhead.cu")
FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
         "-Xcompiler", "-fPIC", "-Xcompiler", "-fvisibility=hidden"]


def _nvcc():
    for c in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", "nvcc"):
        if c and (os.path.isabs(c) and os.path.exists(c) or not os.path.isabs(c)):
            return c
    raise RuntimeError("nvcc not found")


def host_tag() -> str:
    """What the tensor side of the binding is compiled against: it is of use to no other torch or interpreter."""
    import torch
    return f"saki tensor side for torch {torch.__version__}, python {sys.version_info.major}.{sys.version_info.minor};"


def host_matches() -> bool:
    """Whether the built file is for the torch and the interpreter at hand (looked up in the file: loading it may crash)."""
    with open(TORCH_LIB, "rb") as f:
        return host_tag().encode() in f.read()


def _host_command():
    """The compiler call for the tensor side of the binding, against the installed torch."""
    import sysconfig
    import torch
    from torch.utils import cpp_extension
    inc = [*cpp_extension.include_paths(), sysconfig.get_paths()["include"], os.path.join(os.path.dirname(os.path.dirname(_nvcc())), "include")]
    libdir = os.path.join(os.path.dirname(torch.__file__), "lib")
    return [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-fPIC", "-shared", "-fvisibility=hidden", "-Wall",
            f'-DSAKI_BUILT_FOR="{host_tag()}"', f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}", *(a for d in inc for a in ("-isystem", d)),
            TORCH_SOURCE, "-o", TORCH_LIB, f"-L{libdir}", "-ltorch_python", "-ltorch", "-ltorch_cpu", "-ltorch_cuda", "-lc10", "-lc10_cuda"]


def _host_needs_build() -> bool:
    deps = (TORCH_SOURCE, os.path.join(HERE, "..", "include", "saki.h"), os.path.abspath(__file__))
    return not os.path.exists(TORCH_LIB) or not host_matches() or any(os.path.getmtime(d) > os.path.getmtime(TORCH_LIB) for d in deps)


def needs_build() -> bool:
    if not os.path.exists(LIB):
        return True
    t = os.path.getmtime(LIB)
    deps = [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith((".cu", ".cuh"))] + [
        os.path.join(HERE, "..", "include", "saki.h"), os.path.abspath(__file__)]
    return any(os.path.getmtime(d) > t for d in deps)


def build(verbose: bool = False, force: bool = False) -> str:
    objs = []
    procs = []
    host = force or _host_needs_build()
    if host:
        procs.append((TORCH_SOURCE, subprocess.Popen(_host_command(), stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)))
    library = force or needs_build()
    flags = list(FLAGS)
    for src in SOURCES if library else ():
        obj = os.path.join(CSRC, src.replace(".cu", ".o"))
        cmd = [_nvcc(), *flags, "-c", os.path.join(CSRC, src), "-o", obj]
        if verbose:
            cmd.insert(1, "-Xptxas=-v")
        procs.append((src, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)))
        objs.append(obj)
    for src, p in procs:
        out, _ = p.communicate()
        if verbose or p.returncode:
            sys.stderr.write(out)
        if p.returncode:
            raise RuntimeError(f"nvcc failed on {src}")
    if not library:
        return LIB
    cmd = [_nvcc(), "-shared", "-o", LIB, *objs, "-gencode", "arch=compute_100a,code=sm_100a"]
    r = subprocess.run(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)
    if r.returncode:
        sys.stderr.write(r.stdout)
        raise RuntimeError("link failed")
    return LIB


if __name__ == "__main__":
    print(build(verbose="--verbose" in sys.argv, force="--force" in sys.argv))
