"""Builds the C-ABI shared library (``liblinattn.so``) in-tree with nvcc for sm_100a, and ``_binding.so``, the short way of the
Python calls to it, with g++ against the installed torch.

    python -m paper_2509_24695_b200.build [--force] [--verbose]

nvcc cross-compiles without a GPU.  The library links the CUDA runtime statically and
looks the driver's tensor-map encoder up at run time, so it has no link-time dependency
on libcuda.
"""
from __future__ import annotations

import glob
import hashlib
import importlib.util
import os
import subprocess
import sys
import sysconfig

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
LIB = os.path.join(PKG, "liblinattn.so")
STAMP = os.path.join(PKG, "_build", "stamp")
BINDING_SRC = os.path.join(CSRC, "binding.cpp")
BINDING = os.path.join(PKG, "_binding.so")

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a",
    "-O3", "-std=c++17", "-lineinfo",
    "-Xcompiler", "-fPIC", "-Xcompiler", "-fvisibility=hidden",
    "--expt-relaxed-constexpr",
    "--diag-error", "2809",   # the result of a [[nodiscard]] function (a bounded wait) is dropped
]


def sources() -> list[str]:
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _torch_dir() -> str | None:
    spec = importlib.util.find_spec("torch")   # (found, not imported)
    return os.path.dirname(spec.origin) if spec and spec.origin else None


def _binding_command(out: str) -> list[str] | None:
    torch = _torch_dir()
    if torch is None:
        return None
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    include = [os.path.join(ROOT, "include"), os.path.join(torch, "include"), os.path.join(torch, "include", "torch", "csrc", "api", "include"),
               sysconfig.get_paths()["include"], os.path.join(cuda, "include")]
    return ["g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-fvisibility=hidden", *(f"-I{i}" for i in include), BINDING_SRC, "-o", out,
            f"-L{os.path.join(torch, 'lib')}", "-ltorch_python", "-ltorch_cpu", "-lc10", "-lc10_cuda"]


def _fingerprint() -> str:
    h = hashlib.sha256()
    files = sources() + sorted(glob.glob(os.path.join(CSRC, "*.cuh"))) + sorted(glob.glob(os.path.join(ROOT, "include", "*.h"))) + [BINDING_SRC]
    if _torch_dir():
        files.append(os.path.join(_torch_dir(), "version.py"))
    for f in files:
        h.update(f.encode())
        h.update(open(f, "rb").read())
    h.update(" ".join(NVCC_FLAGS).encode())
    return h.hexdigest()


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile every .cu under csrc/ into liblinattn.so (skipped when sources are unchanged)."""
    fp = _fingerprint()
    if not force and os.path.exists(LIB) and (os.path.exists(BINDING) or _torch_dir() is None) and os.path.exists(STAMP) and open(STAMP).read() == fp:
        return LIB
    os.makedirs(os.path.dirname(STAMP), exist_ok=True)
    objs = []
    procs = []
    for src in sources():
        obj = os.path.join(os.path.dirname(STAMP), os.path.basename(src)[:-3] + ".o")
        cmd = ["nvcc", *NVCC_FLAGS, "-I", os.path.join(ROOT, "include"), "-I", CSRC, "-c", src, "-o", obj]
        if verbose:
            cmd.insert(1, "-Xptxas")
            cmd.insert(2, "-v")
        procs.append((cmd, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)))
        objs.append(obj)
    binding_tmp = BINDING + f".tmp{os.getpid()}"
    binding_cmd = _binding_command(binding_tmp)
    if binding_cmd:
        procs.append((binding_cmd, subprocess.Popen(binding_cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)))
    failed = False
    for cmd, p in procs:
        out, _ = p.communicate()
        if p.returncode != 0 or verbose:
            sys.stderr.write(" ".join(cmd) + "\n" + out + "\n")
        failed |= p.returncode != 0
    if failed:
        raise RuntimeError("the compiler failed")
    tmp = LIB + f".tmp{os.getpid()}"
    subprocess.check_call(["nvcc", "-shared", "-gencode", "arch=compute_100a,code=sm_100a", "-o", tmp, *objs,
                           "-Xlinker", "--exclude-libs=ALL"])
    os.replace(tmp, LIB)
    if binding_cmd:
        os.replace(binding_tmp, BINDING)
    with open(STAMP, "w") as f:
        f.write(fp)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="--verbose" in sys.argv))
