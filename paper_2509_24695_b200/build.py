"""Builds the C-ABI shared library (``liblinattn.so``) in-tree with nvcc for sm_100a, and ``_binding``, the short way of the
Python calls to it, with g++ against the installed torch.  The library needs no torch: where the binding cannot be built (no torch, one
without CUDA, no headers) a warning says so, and the calls go the general way.

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
import runpy
import subprocess
import sys
import sysconfig

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
LIB = os.path.join(PKG, "liblinattn.so")
STAMP = os.path.join(PKG, "_build", "stamp")
BINDING_SRC = os.path.join(CSRC, "binding.cpp")
BINDING = os.path.join(PKG, "_binding" + sysconfig.get_config_var("EXT_SUFFIX"))   # (another Python does not see it)
WITHOUT_BINDING = " without binding"   # in the stamp of a build whose binding failed

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


def _torch_version() -> str | None:
    """``torch.__version__`` of the torch that is installed, not imported."""
    path = os.path.join(_torch_dir() or "", "version.py")
    return runpy.run_path(path)["__version__"] if os.path.exists(path) else None


def _binding_command(out: str) -> list[str] | None:
    torch, version = _torch_dir(), _torch_version()
    if version is None:
        return None
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    include = [os.path.join(ROOT, "include"), os.path.join(torch, "include"), os.path.join(torch, "include", "torch", "csrc", "api", "include"),
               sysconfig.get_paths()["include"], os.path.join(cuda, "include")]
    return ["g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-fvisibility=hidden", f'-DBUILT_AGAINST="{version}"', *(f"-I{i}" for i in include), BINDING_SRC, "-o", out,
            f"-L{os.path.join(torch, 'lib')}", "-ltorch_python", "-ltorch_cpu", "-lc10", "-lc10_cuda"]


def _fingerprint() -> str:
    h = hashlib.sha256()
    files = sources() + sorted(glob.glob(os.path.join(CSRC, "*.cuh"))) + sorted(glob.glob(os.path.join(ROOT, "include", "*.h"))) + [BINDING_SRC]
    for f in files:
        h.update(f.encode())
        h.update(open(f, "rb").read())
    h.update(f"{_torch_version()} {sys.version_info[:2]}".encode())
    h.update(" ".join(NVCC_FLAGS).encode())
    return h.hexdigest()


def _start_binding(out: str):
    """(the compiler at work on the binding, or why there is none; the command; its output file)."""
    cmd = _binding_command(out)
    if cmd is None:
        return "no torch is installed", [], out
    try:
        return subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True), cmd, out
    except OSError as e:
        return str(e), cmd, out


def _finish_binding(compiler, cmd, out, verbose) -> bool:
    """Puts the binding in place; False where it could not be built (an older one, of other sources or another torch, then goes too)."""
    text = compiler if isinstance(compiler, str) else compiler.communicate()[0]
    ok = not isinstance(compiler, str) and compiler.returncode == 0
    if cmd and (verbose or not ok):
        sys.stderr.write(" ".join(cmd) + "\n" + text + "\n")
    if ok:
        os.replace(out, BINDING)
        return True
    sys.stderr.write("warning: the short way from torch tensors to the library is not built; calls take the general way\n")
    for stale in (out, BINDING):
        if os.path.exists(stale):
            os.remove(stale)
    return False


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile every .cu under csrc/ into liblinattn.so (skipped when sources are unchanged)."""
    fp = _fingerprint()
    built = fp if os.path.exists(BINDING) else fp + WITHOUT_BINDING
    if not force and os.path.exists(LIB) and os.path.exists(STAMP) and open(STAMP).read() == built:
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
    binding = _start_binding(BINDING + f".tmp{os.getpid()}")
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
    built = fp if _finish_binding(*binding, verbose) else fp + WITHOUT_BINDING
    with open(STAMP, "w") as f:
        f.write(built)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="--verbose" in sys.argv))
