"""Builds, in-tree, liblbp.so (the C-ABI library) with nvcc for sm_100a and
_lbp_torch.so (the native part of the Python binding) with the host compiler."""
from __future__ import annotations

import importlib.metadata
import os
import shutil
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "liblbp.so")
BINDING = os.path.join(HERE, "_lbp_torch.so")
BINDING_SOURCE = os.path.join(CSRC, "torch_binding.cpp")
TORCH_STAMP = os.path.join(HERE, "_build", "torch_version")

SOURCES = ["lbp_host.cpp", "lbp_api.cu", "wht_project.cu", "wht_expand.cu",
           "gemm_fp32.cu", "gemm_fp32_split.cu", "gemm_bf16.cu", "lbp_fused.cu", "lbp_static.cu",
           "wht_spectrum.cu", "lbp_extras.cu", "lbp_fused_plan.cu", "wht_project_umma.cu"]


def _nvcc() -> str:
    exe = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(exe):
        raise RuntimeError("nvcc not found")
    return exe


def _torch_version() -> str:
    return importlib.metadata.version("torch")


def _stale() -> bool:
    if not os.path.exists(LIB) or not os.path.exists(BINDING):
        return True
    # the binding is good for the torch it was compiled against only
    if not os.path.exists(TORCH_STAMP) or open(TORCH_STAMP).read() != _torch_version():
        return True
    t = min(os.path.getmtime(LIB), os.path.getmtime(BINDING))
    deps = [os.path.join(CSRC, f) for f in os.listdir(CSRC)]
    deps.append(os.path.join(ROOT, "include", "lbp.h"))
    return any(os.path.getmtime(d) > t for d in deps)


def _binding_command() -> list:
    import sysconfig

    import torch
    root = os.path.dirname(os.path.abspath(torch.__file__))
    cuda = os.path.dirname(os.path.dirname(_nvcc()))
    libs = os.path.join(root, "lib")
    return [shutil.which("g++") or "g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-fvisibility=hidden",
            "-Wall", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
            "-I", os.path.join(ROOT, "include"), "-isystem", os.path.join(root, "include"),
            "-isystem", os.path.join(root, "include", "torch", "csrc", "api", "include"),
            "-isystem", sysconfig.get_paths()["include"], "-isystem", os.path.join(cuda, "include"),
            BINDING_SOURCE, "-o", BINDING, "-L", libs, "-lc10", "-lc10_cuda", "-ltorch_cpu", "-ltorch",
            "-ltorch_python", "-ldl", f"-Wl,-rpath,{libs}"]


def build_library(force: bool = False, verbose: bool = False, extra_flags=(), out: str | None = None) -> str:
    """Compile every CUDA source into paper_2309_15275_b200/liblbp.so, and the binding.

    `extra_flags` (e.g. ["-DLBP_ROLE_TRACE"]) with `out` builds a diagnostic
    variant into another file; the binding loads it when LBP_LIBRARY names it."""
    if out is None and not extra_flags:
        if not force and not _stale():
            return LIB
    lib = out or LIB
    objs = []
    build_dir = os.path.join(HERE, "_build" if out is None else "_build_variant")
    os.makedirs(build_dir, exist_ok=True)
    common = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "-Xcompiler", "-fPIC", "-I", os.path.join(ROOT, "include"), "-I", CSRC, *extra_flags]
    if verbose:
        common += ["-Xptxas", "-v"]
    procs = []
    for src in SOURCES:
        obj = os.path.join(build_dir, os.path.splitext(src)[0] + ".o")
        objs.append(obj)
        cmd = [_nvcc(), *common, "-x", "cu", "-c", os.path.join(CSRC, src), "-o", obj]
        procs.append((src, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT,
                                            text=True)))
    if out is None:
        procs.append((os.path.basename(BINDING_SOURCE),
                      subprocess.Popen(_binding_command(), stdout=subprocess.PIPE, stderr=subprocess.STDOUT,
                                       text=True)))
    failed = False
    for src, p in procs:
        log, _ = p.communicate()
        if verbose or p.returncode != 0:
            sys.stderr.write(f"--- {src} ---\n{log}\n")
        failed |= p.returncode != 0
    if failed:
        raise RuntimeError("nvcc failed")
    link = [_nvcc(), "-shared", "-o", lib, *objs, "-lcudart_static", "-ldl", "-lrt", "-lpthread"]
    subprocess.run(link, check=True)
    if out is None:
        with open(TORCH_STAMP, "w") as f:
            f.write(_torch_version())
    return lib


if __name__ == "__main__":
    print(build_library(force="--force" in sys.argv, verbose="-v" in sys.argv))
