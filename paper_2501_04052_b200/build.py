"""Build librazer.so (CUDA kernels + C ABI) in-tree for sm_100a with nvcc.

    python -m paper_2501_04052_b200.build [--force] [--verbose]

The library is written next to this file; cudart is linked statically and the driver API
is reached through cudaGetDriverEntryPoint, so the file loads on a machine without a GPU.
razer_call.so beside it is the compiled part of the Python binding, built against the installed
torch and this interpreter's headers; where it cannot be built the binding goes through ctypes.
"""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "librazer.so")
CALL = os.path.join(HERE, "razer_call.so")
SOURCES = ["razer_api.cu", "razer_pack.cu", "razer_quant.cu", "razer_gemv_simt.cu", "razer_gemm_umma.cu", "razer_gemm_fp4.cu", "razer_gemv_stream.cu",
           "razer_static_scratch.cu"]
NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "-Xcompiler", "-fPIC", "--expt-relaxed-constexpr"]


def _deps():
    out = [os.path.join(CSRC, f) for f in os.listdir(CSRC)]
    out.append(os.path.join(os.path.dirname(HERE), "include", "razer.h"))
    return out


def needs_build() -> bool:
    if not os.path.exists(LIB) or not os.path.exists(CALL):
        return True
    t = os.path.getmtime(LIB)
    return any(os.path.getmtime(p) > t for p in _deps())


def build_call(verbose: bool = False) -> None:
    import torch
    root = os.path.dirname(torch.__file__)
    inc = [os.path.join(root, "include"), os.path.join(root, "include", "torch", "csrc", "api", "include"), sysconfig.get_paths()["include"],
           os.path.join(os.path.dirname(os.path.dirname(os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc"))), "include")]
    lib = os.path.join(root, "lib")
    cmd = [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-fPIC", "-shared", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
           *("-I" + d for d in inc), os.path.join(CSRC, "razer_call.cpp"), "-o", CALL, "-L" + lib, "-lc10", "-lc10_cuda", "-ltorch_cpu",
           "-ltorch_python", "-Wl,-rpath," + lib]
    try:
        r = subprocess.run(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)
        failed, out = r.returncode != 0, r.stdout
    except OSError as e:
        failed, out = True, str(e)
    if failed or verbose:
        sys.stderr.write(f"--- razer_call.cpp\n{out}\n")
    if failed:
        sys.stderr.write("razer_call.so was not built: the binding will go through ctypes\n")


def build(force: bool = False, verbose: bool = False) -> str:
    if not force and not needs_build():
        return LIB
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    objs = []
    procs = []
    for src in SOURCES:
        obj = os.path.join(CSRC, src.replace(".cu", ".o"))
        cmd = [nvcc, *NVCC_FLAGS, "-c", os.path.join(CSRC, src), "-o", obj]
        if verbose:
            cmd.insert(1, "-Xptxas")
            cmd.insert(2, "-v")
        procs.append((src, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)))
        objs.append(obj)
    failed = False
    for src, p in procs:
        out, _ = p.communicate()
        if p.returncode != 0 or verbose:
            sys.stderr.write(f"--- {src}\n{out}\n")
        failed |= p.returncode != 0
    if failed:
        raise RuntimeError("nvcc failed")
    cmd = [nvcc, "-shared", "-o", LIB, *objs, "-gencode", "arch=compute_100a,code=sm_100a"]
    build_call(verbose)
    subprocess.run(cmd, check=True)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="--verbose" in sys.argv))
