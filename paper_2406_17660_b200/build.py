"""Build the C-ABI library in-tree with nvcc for sm_100a.

    python -m paper_2406_17660_b200.build

Produces libgrass_b200.so (the CUDA library, nvcc) and the binding's scan of torch tensors (g++ against
torch's and Python's headers, whose object layouts it is built for: its file name carries both versions)
next to this file.  nvcc cross-compiles without a GPU, so this runs on any box with the CUDA toolkit.
"""
from __future__ import annotations

import os
import shutil
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libgrass_b200.so")
SOURCES = ["common.cu", "row_norms.cu", "select.cu", "project.cu", "adam.cu", "scatter.cu",
           "adam_scatter.cu", "selftest.cu"]


def _nvcc() -> str:
    for cand in (os.environ.get("NVCC"), shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found; set NVCC or install the CUDA toolkit")


def scan_path() -> str:
    """The scan module for the torch and the Python that run now."""
    import torch
    return os.path.join(HERE, f"_scan.{sysconfig.get_config_var('SOABI')}.torch-{torch.__version__}.so")


def _stale() -> bool:
    scan = scan_path()
    if not (os.path.exists(LIB) and os.path.exists(scan)):
        return True
    t = min(os.path.getmtime(LIB), os.path.getmtime(scan))
    deps = [os.path.join(CSRC, f) for f in os.listdir(CSRC)]
    deps += [os.path.join(ROOT, "include", f) for f in os.listdir(os.path.join(ROOT, "include"))]
    return any(os.path.getmtime(d) > t for d in deps)


def _scan_command() -> list:
    import torch
    from torch.utils.cpp_extension import include_paths
    cmd = [shutil.which("g++") or "g++", "-O2", "-std=c++17", "-shared", "-fPIC",
           f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}"]
    for path in include_paths():
        cmd += ["-isystem", path]
    return cmd + ["-I", sysconfig.get_paths()["include"], "-I", os.path.join(ROOT, "include"), "-o", scan_path(),
                  os.path.join(CSRC, "scan.cpp"), "-L", os.path.join(os.path.dirname(torch.__file__), "lib"),
                  "-ltorch_python", "-ltorch_cpu", "-lc10"]


def build(force: bool = False, verbose: bool = False) -> str:
    if not force and not _stale():
        return LIB
    cmd = [_nvcc(), "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3",
           "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "-I", os.path.join(ROOT, "include"),
           "-I", CSRC, "-o", LIB] + [os.path.join(CSRC, s) for s in SOURCES]
    if verbose:
        cmd[1:1] = ["-Xptxas", "-v"]
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        sys.stderr.write(res.stdout + res.stderr)
        raise RuntimeError("nvcc failed building libgrass_b200.so")
    if verbose:
        sys.stderr.write(res.stderr)
    res = subprocess.run(_scan_command(), capture_output=True, text=True)
    if res.returncode != 0:
        sys.stderr.write(res.stdout + res.stderr)
        raise RuntimeError("g++ failed building the scan module")
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
