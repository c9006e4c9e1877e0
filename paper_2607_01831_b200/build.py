"""Builds liblynx.so (the C-ABI CUDA library) in-tree with nvcc for sm_100a, and _native.so (the Python calls that go straight
to it, against the installed torch) with g++."""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig
import warnings

_HERE = os.path.dirname(os.path.abspath(__file__))
_ROOT = os.path.dirname(_HERE)
CSRC = os.path.join(_HERE, "csrc")
LIB = os.path.join(_HERE, "liblynx.so")
NATIVE = os.path.join(_HERE, "_native.so")
SOURCES = ["api.cu", "split_quantize.cu", "attention.cu", "bf16_attention.cu", "hier_quantize.cu", "token_verify.cu", "lse_merge.cu", "bit_split.cu"]
NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "-Xcompiler", "-fPIC", "--expt-relaxed-constexpr"]


def _stale(target: str = LIB) -> bool:
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    deps = [os.path.join(CSRC, f) for f in os.listdir(CSRC) if not f.endswith(".o")] + [os.path.join(_ROOT, "include", "lynx.h")]
    return any(os.path.getmtime(d) > t for d in deps)


def _native_stale() -> bool:
    """Also where it was compiled against another torch (whose name it carries)."""
    import torch
    if _stale(NATIVE):
        return True
    with open(NATIVE, "rb") as f:
        return torch.__version__.encode() + b"\0" not in f.read()


def _native_cmd(out: str) -> list:
    """The extension is linked to liblynx.so beside it; torch's own libraries are there once torch is imported."""
    import torch
    from torch.utils.cpp_extension import include_paths, library_paths
    cxx = os.environ.get("CXX", "g++")
    cmd = [cxx, "-O2", "-std=c++17", "-fPIC", "-shared", "-I", os.path.join(_ROOT, "include"), "-I", sysconfig.get_paths()["include"]]
    for p in include_paths(device_type="cuda"):
        cmd += ["-isystem", p]
    cmd += [f'-DLYNX_TORCH_VERSION="{torch.__version__}"', os.path.join(CSRC, "native.cpp"), "-o", out]
    for p in library_paths(device_type="cuda"):
        cmd += ["-L", p]
    return cmd + ["-ltorch_python", "-ltorch", "-ltorch_cpu", "-lc10", "-lc10_cuda", "-L", _HERE, "-l:liblynx.so", "-Wl,-rpath,$ORIGIN"]


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile every .cu under csrc/ into liblynx.so and csrc/native.cpp into _native.so; returns the former's path.  The library
    works without the extension (calls then cost more host time), whose failure to compile is a warning."""
    if force or _stale():
        _build_library(verbose)
    if force or _native_stale():
        tmp = NATIVE + f".tmp{os.getpid()}"
        try:
            subprocess.run(_native_cmd(tmp), check=True)
            os.replace(tmp, NATIVE)
        except (OSError, subprocess.CalledProcessError) as e:
            warnings.warn(f"_native.so was not built ({e}): Python calls go through ctypes")
    return LIB


def _build_library(verbose: bool) -> None:
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    objs = []
    procs = []
    for src in SOURCES:
        obj = os.path.join(CSRC, src.replace(".cu", ".o"))
        cmd = [nvcc, *NVCC_FLAGS, "-I", os.path.join(_ROOT, "include"), "-I", CSRC, "-c",
               os.path.join(CSRC, src), "-o", obj]
        if verbose:
            cmd.insert(1, "-Xptxas=-v")
        procs.append((src, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT,
                                            text=True)))
        objs.append(obj)
    for src, pr in procs:
        out, _ = pr.communicate()
        if verbose or pr.returncode != 0:
            sys.stderr.write(out)
        if pr.returncode != 0:
            raise RuntimeError(f"nvcc failed on {src}")
    tmp = LIB + f".tmp{os.getpid()}"
    subprocess.run([nvcc, "-shared", "-o", tmp, *objs], check=True)   # static cudart (nvcc default)
    os.replace(tmp, LIB)


if __name__ == "__main__":
    print(build(force=True, verbose="-v" in sys.argv))
