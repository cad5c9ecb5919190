"""Builds libfpq.so (sm_100a only, nvcc) and the torch binding _fpq_torch.so (g++) in-tree."""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
SO = os.path.join(HERE, "libfpq.so")
BINDING = os.path.join(HERE, "_fpq_torch.so")
SOURCES = ["fpq_api.cu", "fpq_quantize.cu", "fpq_gemm.cu", "fpq_pair.cu", "fpq_pair_gemm.cu", "fpq_pair_rows.cu", "fpq_noalloc.cu", "fpq_search.cu", "fpq_smallm.cu", "fpq_fewrows.cu",
           "fpq_roundlearn.cu", "fpq_general.cu", "fpq_tf32.cu", "fpq_tensormap.cu"]


def _newest_source_mtime() -> float:
    paths = [os.path.join(CSRC, f) for f in os.listdir(CSRC)] + [os.path.join(ROOT, "include", "fpq.h")]
    return max(os.path.getmtime(p) for p in paths)


def build(force: bool = False, verbose: bool = False) -> str:
    newest = _newest_source_mtime()
    if not force and all(os.path.exists(p) and os.path.getmtime(p) >= newest for p in (SO, BINDING)):
        return SO
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    cmd = [nvcc, "-gencode", "arch=compute_100a,code=sm_100a", "-O3", "-lineinfo", "-std=c++17",
           "-shared", "-Xcompiler", "-fPIC", "-I", os.path.join(ROOT, "include"), "-I", CSRC,
           "-cudart", "static"]
    if verbose:
        cmd += ["-Xptxas", "-v"]
    cmd += [os.path.join(CSRC, s) for s in SOURCES] + ["-o", SO]
    subprocess.run(cmd, check=True)
    build_binding()
    return SO


def build_binding() -> None:
    """The per-layer calls as a CPython extension over torch tensors (a few headers of torch and its c10 library)."""
    import torch
    inc = os.path.join(os.path.dirname(torch.__file__), "include")
    libs = os.path.join(os.path.dirname(torch.__file__), "lib")
    cmd = ["g++", "-O2", "-std=c++17", "-shared", "-fPIC", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
           "-I", os.path.join(ROOT, "include"), "-I", sysconfig.get_paths()["include"], "-I", inc,
           "-I", os.path.join(inc, "torch", "csrc", "api", "include"), "-I", "/usr/local/cuda/include",
           os.path.join(CSRC, "fpq_torch.cpp"), "-o", BINDING, "-L", HERE, "-l:libfpq.so", "-L", libs,
           "-lc10", "-lc10_cuda", "-ltorch_cpu", "-ltorch_python", "-Wl,-rpath,$ORIGIN", f"-Wl,-rpath,{libs}"]
    subprocess.run(cmd, check=True)


if __name__ == "__main__":
    print(build(force=True, verbose="-v" in sys.argv))
