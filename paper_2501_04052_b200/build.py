"""Build librazer.so (CUDA kernels + C ABI) in-tree for sm_100a with nvcc.

    python -m paper_2501_04052_b200.build [--force] [--verbose]

The library is written next to this file; cudart is linked statically and the driver API
is reached through cudaGetDriverEntryPoint, so the file loads on a machine without a GPU.
razer_call.<interpreter>.<torch>.so beside it is the compiled part of the Python binding, for the torch
and the interpreter that its name says and no other; where it cannot be built the binding goes through ctypes.
"""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "librazer.so")
SOURCES = ["razer_api.cu", "razer_pack.cu", "razer_quant.cu", "razer_gemv_simt.cu", "razer_gemm_umma.cu", "razer_gemm_fp4.cu", "razer_gemv_stream.cu",
           "razer_static_scratch.cu"]
NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "-Xcompiler", "-fPIC", "--expt-relaxed-constexpr"]


HEADER = os.path.join(os.path.dirname(HERE), "include", "razer.h")
CALL_SOURCE = os.path.join(CSRC, "razer_call.cpp")


def _newer(target: str, deps) -> bool:
    """`target` exists and none of `deps` is newer."""
    return os.path.exists(target) and all(os.path.getmtime(p) <= os.path.getmtime(target) for p in deps)


def call_path(torch_version: str | None = None) -> str:
    """The compiled part for this interpreter and that torch (None: the installed one; "none" where there is none).  Its code has the layout of
    torch's tensors and of the interpreter's objects built in, so that a file for others is not one to be looked at, let alone loaded."""
    if torch_version is None:
        try:
            from torch.version import __version__ as torch_version
        except Exception:
            torch_version = "none"
    tag = "".join(c if c.isalnum() or c in "-_" else "_" for c in torch_version)
    return os.path.join(HERE, f"razer_call.{sysconfig.get_config_var('SOABI')}.torch-{tag}.so")


def needs_build() -> bool:
    """The library: its own sources only, whatever became of the binding's compiled part."""
    return not _newer(LIB, [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith((".cu", ".cuh", ".h"))] + [HEADER])


def needs_call() -> bool:
    """The compiled part: neither built nor, since its sources last changed, found impossible to build."""
    path = call_path()
    return not any(_newer(p, [CALL_SOURCE, HEADER]) for p in (path, path + ".failed"))


def _run(cmd) -> tuple[bool, str]:
    try:
        r = subprocess.run(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)
        return r.returncode == 0, r.stdout
    except OSError as e:
        return False, str(e)


def build_call(verbose: bool = False) -> None:
    """Never fails: without this file the binding goes through ctypes.  What an older build left is gone either way."""
    path = call_path()
    for p in [os.path.join(HERE, f) for f in os.listdir(HERE) if f.startswith("razer_call.")]:
        os.remove(p)
    try:
        import torch
        root = os.path.dirname(torch.__file__)
        inc = [os.path.join(root, "include"), os.path.join(root, "include", "torch", "csrc", "api", "include"), sysconfig.get_paths()["include"],
               os.path.join(os.path.dirname(os.path.dirname(os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc"))), "include")]
        lib = os.path.join(root, "lib")
        ok, out = _run([os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-fPIC", "-shared",
                        f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}", *("-I" + d for d in inc), CALL_SOURCE, "-o", path + ".tmp",
                        "-L" + lib, "-lc10", "-lc10_cuda", "-ltorch_cpu", "-ltorch_python", "-Wl,-rpath," + lib])
    except Exception as e:                               # no torch, or one that does not load
        ok, out = False, repr(e)
    if ok:
        os.replace(path + ".tmp", path)
    else:
        with open(path + ".failed", "w") as f:
            f.write(out)
    if not ok or verbose:
        sys.stderr.write(f"--- razer_call.cpp\n{out}\n")
    if not ok:
        sys.stderr.write("razer_call.cpp was not built: the binding will go through ctypes (--force tries again)\n")


def build_lib(verbose: bool = False) -> None:
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
    # beside it and then in its place: a process that has the library mapped keeps what it mapped
    subprocess.run([nvcc, "-shared", "-o", LIB + ".tmp", *objs, "-gencode", "arch=compute_100a,code=sm_100a"], check=True)
    os.replace(LIB + ".tmp", LIB)


def build(force: bool = False, verbose: bool = False) -> str:
    if force or needs_build():
        build_lib(verbose)
    if force or needs_call():
        build_call(verbose)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="--verbose" in sys.argv))
