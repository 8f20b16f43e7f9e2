"""Builds libavsa.so and the two host extensions of its binding in-tree with nvcc for sm_100a (cross-compiles without a GPU)."""
from __future__ import annotations

import os
import shutil
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libavsa.so")
HOST = os.path.join(HERE, "_avsa_host" + sysconfig.get_config_var("EXT_SUFFIX"))      # marshalling for this interpreter
ALLOC = os.path.join(HERE, "_avsa_alloc" + sysconfig.get_config_var("EXT_SUFFIX"))    # tensors for the wrappers
ALLOC_FOR = os.path.join(HERE, "build", "alloc_built_for.txt")      # the PyTorch that ALLOC was compiled against
SOURCES = ["api.cu", "mask.cu", "sparse_attn.cu", "cross_attn.cu", "protected_rows.cu", "cache_indicators.cu"]
HEADERS = sorted(f for f in os.listdir(CSRC) if f.endswith(".cuh")) + [os.path.join("..", "..", "include", "avsa.h")]
NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-O3", "-lineinfo", "-std=c++17",
              "-Xcompiler", "-fPIC", "-Xcompiler", "-fvisibility=hidden"]


def _nvcc() -> str:
    exe = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(exe):
        raise RuntimeError("nvcc not found: libavsa.so cannot be built")
    return exe


def _torch_abi() -> str:
    """What the allocating extension is bound to besides its source."""
    import torch
    return f"torch {torch.__version__} cxx11 abi {int(torch.compiled_with_cxx11_abi())}"


def _stale() -> bool:
    outputs = (LIB, HOST, ALLOC)
    if not all(os.path.exists(o) for o in outputs + (ALLOC_FOR,)):
        return True
    with open(ALLOC_FOR) as f:
        if f.read() != _torch_abi():
            return True
    t = min(os.path.getmtime(o) for o in outputs)
    deps = [os.path.join(CSRC, s) for s in SOURCES + HEADERS + ["host_call.cc", "host_alloc.cc"]]
    return any(os.path.getmtime(p) > t for p in deps)


def _start_host_builds():
    """g++ on the two host extensions: (source, process) each."""
    import torch
    base = torch.__path__[0]
    include = [os.path.join(base, "include"), os.path.join(base, "include", "torch", "csrc", "api", "include")]
    common = ["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-fvisibility=hidden", "-I" + sysconfig.get_paths()["include"]]
    host = common + ["-Wall", "-Wno-cast-function-type", os.path.join(CSRC, "host_call.cc"), "-o", HOST]
    alloc = common + [f"-D_GLIBCXX_USE_CXX11_ABI={int(torch.compiled_with_cxx11_abi())}"]
    alloc += [flag for path in include for flag in ("-isystem", path)]
    alloc += [os.path.join(CSRC, "host_alloc.cc"), "-o", ALLOC, "-L" + os.path.join(base, "lib"),
              "-ltorch_python", "-ltorch_cpu", "-ltorch", "-lc10"]
    return [(name, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True))
            for name, cmd in (("host_call.cc", host), ("host_alloc.cc", alloc))]


def build_library(force: bool = False, verbose: bool = False) -> str:
    """Compiles every .cu of the library, links libavsa.so and builds the host extensions; returns the library's path."""
    if not force and not _stale():
        return LIB
    nvcc = _nvcc()
    objdir = os.path.join(HERE, "build")
    os.makedirs(objdir, exist_ok=True)
    procs = []      # (source, object or None, process), all at once
    for name, pr in _start_host_builds():
        procs.append((name, None, pr))
    for s in SOURCES:
        obj = os.path.join(objdir, s.replace(".cu", ".o"))
        cmd = [nvcc] + NVCC_FLAGS + (["-Xptxas", "-v"] if verbose else []) + ["-c", os.path.join(CSRC, s), "-o", obj]
        procs.append((s, obj, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)))
    outputs = [pr.communicate()[0] for _, _, pr in procs]      # (all of them end before the first failure is reported)
    for (name, obj, pr), out in zip(procs, outputs):
        if verbose and out and obj is not None:
            print(out)
        if pr.returncode != 0:
            raise RuntimeError(f"{'g++' if obj is None else 'nvcc'} failed on {name}:\n{out}")
    objs = [obj for _, obj, _ in procs if obj is not None]
    cmd = [nvcc, "-shared", "-o", LIB] + objs + ["-gencode", "arch=compute_100a,code=sm_100a"]
    r = subprocess.run(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"link failed:\n{r.stdout}")
    with open(ALLOC_FOR, "w") as f:
        f.write(_torch_abi())
    return LIB


if __name__ == "__main__":
    print(build_library(force="--force" in sys.argv, verbose="-v" in sys.argv))
