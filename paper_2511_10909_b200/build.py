"""Builds libmmasim.so (nvcc, sm_100a) and the Python call path _mmasim_py.so (g++, against torch) in-tree."""
from __future__ import annotations

import os
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libmmasim.so")
PY_EXT = os.path.join(HERE, "_mmasim_py.so")
SOURCES = ["mmasim_api.cpp", "mmasim_registry.cpp", "mmasim_generic.cu", "mmasim_tfdpa_fast.cu",
           "mmasim_tfdpa_fast_lut8.cu", "mmasim_tfdpa_fast_f16.cu", "mmasim_tfdpa_fast_bf16.cu", "mmasim_direct_8.cu", "mmasim_direct_16.cu", "mmasim_direct_32.cu", "mmasim_direct_amd.cu", "mmasim_trfdpa_f64.cu", "mmasim_efdpa_f64.cu", "mmasim_fp_fast.cu", "mmasim_gst_fast.cu", "mmasim_umma.cu", "mmasim_warp_mma.cu",
           "mmasim_dot_stream.cu", "mmasim_peak.cu", "mmasim_hw_mma.cu", "mmasim_hw_umma.cu", "mmasim_stats.cu"]
HEADERS = ["mmasim_internal.h", "mmasim_device.cuh", "mmasim_tfdpa_fast.cuh", "mmasim_tfdpa_f64.cuh", "mmasim_tfdpa_trop.cuh", "mmasim_direct.cuh", "mmasim_tma.cuh", "mmasim_stats.cuh", os.path.join("..", "..", "include", "mmasim.h")]
NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "-Xcompiler", "-fPIC", "--fmad=false"]


def _nvcc() -> str:
    for cand in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", "nvcc"):
        if cand and (os.path.isabs(cand) and os.path.exists(cand) or not os.path.isabs(cand)):
            return cand
    raise RuntimeError("nvcc not found")


def built_against() -> str:
    """What the extension module carries to say which torch it belongs to (its classes have no stable layout)."""
    from importlib.metadata import version
    return "torch " + version("torch")


def _stale() -> bool:
    if not (os.path.exists(LIB) and os.path.exists(PY_EXT)):
        return True
    with open(PY_EXT, "rb") as f:
        if built_against().encode() + b"\0" not in f.read():
            return True
    t = min(os.path.getmtime(LIB), os.path.getmtime(PY_EXT))
    deps = [os.path.join(CSRC, s) for s in SOURCES + HEADERS + ["mmasim_py.cpp"]] + [__file__]
    return any(os.path.getmtime(d) > t for d in deps)


def _py_ext_cmd() -> list[str]:
    import sysconfig
    import torch
    root = os.path.dirname(torch.__file__)
    inc = [os.path.join(root, "include"), os.path.join(root, "include", "torch", "csrc", "api", "include"), "/usr/local/cuda/include",
           sysconfig.get_paths()["include"]]
    return ["g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-fvisibility=hidden", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
            f'-DMMASIM_BUILT_AGAINST="{built_against()}"', *(f"-I{d}" for d in inc), os.path.join(CSRC, "mmasim_py.cpp"), "-o", PY_EXT, "-L" + os.path.join(root, "lib"),
            "-ltorch_python", "-ltorch_cpu", "-lc10", "-lc10_cuda"]


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile every source for sm_100a and link libmmasim.so next to this file; returns its path."""
    if not force and not _stale():
        return LIB
    objs = []
    procs = []
    for src in SOURCES:
        obj = os.path.join(CSRC, os.path.splitext(src)[0] + ".o")
        cmd = [_nvcc(), *NVCC_FLAGS, "-x", "cu", "-c", os.path.join(CSRC, src), "-o", obj]
        if verbose:
            cmd.insert(1, "-Xptxas=-v")
        procs.append((src, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)))
        objs.append(obj)
    procs.append(("mmasim_py.cpp", subprocess.Popen(_py_ext_cmd(), stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)))
    for src, p in procs:
        out, _ = p.communicate()
        if verbose or p.returncode:
            sys.stderr.write(out)
        if p.returncode:
            raise RuntimeError(f"compiling {src} failed:\n{out}")
    link = [_nvcc(), "-gencode", "arch=compute_100a,code=sm_100a", "-shared", "-o", LIB, *objs, "-lcudart"]
    subprocess.run(link, check=True)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
