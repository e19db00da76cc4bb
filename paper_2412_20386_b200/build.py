"""Build ``libptq_linear.so`` in-tree with nvcc for sm_100a, and ``_ptq_torch.so`` (the binding's calls on torch tensors)
with the host compiler against the headers of the installed torch.

    python -m paper_2412_20386_b200.build [--force] [--verbose]

nvcc cross-compiles without a GPU.  The CUDA runtime is linked statically and the
driver API is reached through the runtime's entry-point query, so the library
loads (and exports its symbols) on machines that have no NVIDIA driver.  It does not depend on torch.
"""
from __future__ import annotations

import importlib.metadata
import os
import shutil
import subprocess
import sys
import sysconfig
from concurrent.futures import ThreadPoolExecutor

_HERE = os.path.dirname(os.path.abspath(__file__))
_CSRC = os.path.join(_HERE, "csrc")
_SO = os.path.join(_HERE, "libptq_linear.so")
_SOURCES = ["ptq_api.cu"]
_DEPS = ["ptq_api.cu", "ptq_gemm.cuh", "ptq_fused.cuh", "ptq_small.cuh", "ptq_short_k.cuh", "ptq_quantize.cuh", "ptq_quantize_dynamic.cuh",
         "ptq_calibrate.cuh", "ptq_probe.cuh", "ptx_sm100.cuh",
         os.path.join("..", "..", "include", "ptq_linear.h")]


def nvcc_path() -> str:
    for cand in (os.environ.get("NVCC"), shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found")


_EXT = os.path.join(_HERE, "_ptq_torch.so")
_EXT_STAMP = os.path.join(_HERE, "_build", "_ptq_torch.versions")     # what the extension was compiled against
_EXT_DEPS = ["ptq_torch.cpp", os.path.join("..", "..", "include", "ptq_linear.h")]


def up_to_date(target: str = _SO, deps=_DEPS) -> bool:
    if not os.path.exists(target):
        return False
    t = os.path.getmtime(target)
    return all(os.path.getmtime(os.path.join(_CSRC, d)) <= t for d in deps)


def _ext_versions() -> str:
    """The extension uses torch's C++ classes and Python's C API: another version of either is another layout."""
    return "torch %s, python %s" % (importlib.metadata.version("torch"), sys.version.split()[0])


def extension_up_to_date() -> bool:
    if not up_to_date(_EXT, _EXT_DEPS) or not os.path.exists(_EXT_STAMP):
        return False
    with open(_EXT_STAMP) as f:
        return f.read() == _ext_versions()


def _run(cmd, target: str, verbose: bool) -> None:
    tmp = target + ".tmp.%d" % os.getpid()
    res = subprocess.run(cmd + ["-o", tmp], stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)
    if verbose or res.returncode != 0:
        sys.stderr.write(res.stdout)
    if res.returncode != 0:
        if os.path.exists(tmp):
            os.remove(tmp)
        raise RuntimeError("%s failed (exit %d)" % (os.path.basename(cmd[0]), res.returncode))
    os.replace(tmp, target)


def _build_library(verbose: bool) -> None:
    cmd = [nvcc_path(), "-gencode", "arch=compute_100a,code=sm_100a", "-O3", "-lineinfo", "-std=c++17",
           "-shared", "-Xcompiler", "-fPIC", "-cudart", "static",
           "-Xptxas", "-v" if verbose else "-warn-spills"]
    _run(cmd + [os.path.join(_CSRC, s) for s in _SOURCES], _SO, verbose)


def _build_extension(verbose: bool) -> None:
    import torch
    root = os.path.dirname(os.path.abspath(torch.__file__))
    cuda = os.path.dirname(os.path.dirname(nvcc_path()))
    cmd = [os.environ.get("CXX") or shutil.which("g++") or "g++", "-O2", "-std=c++20", "-shared", "-fPIC",
           "-D_GLIBCXX_USE_CXX11_ABI=%d" % int(torch.compiled_with_cxx11_abi()), "-DUSE_CUDA",
           "-isystem", os.path.join(root, "include"),
           "-isystem", os.path.join(root, "include", "torch", "csrc", "api", "include"),
           "-isystem", os.path.join(cuda, "include"), "-isystem", sysconfig.get_paths()["include"],
           os.path.join(_CSRC, "ptq_torch.cpp"), "-L" + os.path.join(root, "lib"),
           "-Wl,-rpath," + os.path.join(root, "lib"),
           "-ltorch_python", "-ltorch_cuda", "-ltorch_cpu", "-lc10_cuda", "-lc10"]
    _run(cmd, _EXT, verbose)
    os.makedirs(os.path.dirname(_EXT_STAMP), exist_ok=True)
    with open(_EXT_STAMP, "w") as f:
        f.write(_ext_versions())


def build(force: bool = False, verbose: bool = False) -> str:
    jobs = []
    if force or not up_to_date():
        jobs.append(_build_library)
    if force or not extension_up_to_date():
        jobs.append(_build_extension)
    with ThreadPoolExecutor(2) as pool:
        for f in [pool.submit(j, verbose) for j in jobs]:
            f.result()
    return _SO


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="--verbose" in sys.argv))
