"""Compile the CUDA sources of this package into librdk_b200.so (sm_100a only), in-tree."""
from __future__ import annotations

import os
import shutil
import subprocess
import sys
import tempfile
from concurrent.futures import ThreadPoolExecutor

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "librdk_b200.so")
HOST = os.path.join(HERE, "_rdk_host.so")        # the binding's native part
SOURCES = ["rdk_api.cu", "rdk_ids.cu", "rdk_row.cu", "rdk_row_cluster.cu", "rdk_row_stream.cu", "rdk_emit.cu", "rdk_affinity.cu", "rdk_affinity_tc.cu", "rdk_exact.cu", "rdk_exact_tc.cu"]


def _nvcc() -> str:
    for cand in (os.environ.get("NVCC"), shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found; the RDK library has no other build route")


def _stale() -> bool:
    if not os.path.exists(LIB) or not os.path.exists(HOST):
        return True
    t = min(os.path.getmtime(LIB), os.path.getmtime(HOST))
    deps = [os.path.join(CSRC, f) for f in os.listdir(CSRC)] + [os.path.join(ROOT, "include", "rdk.h")]
    return any(os.path.getmtime(d) > t for d in deps)


def _host_command():
    """Compiler command of the binding's native part, against the headers and libraries of the torch in use."""
    import sysconfig

    import torch
    from torch.utils import cpp_extension
    cuda = os.path.dirname(os.path.dirname(os.path.realpath(_nvcc())))
    inc = [os.path.join(ROOT, "include"), sysconfig.get_paths()["include"], os.path.join(cuda, "include"), *cpp_extension.include_paths()]
    libdir = os.path.join(os.path.dirname(torch.__file__), "lib")
    return ["g++", "-shared", "-fPIC", "-std=c++17", "-O2", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
            *[f for i in inc for f in ("-isystem" if "torch" in i else "-I", i)], os.path.join(CSRC, "rdk_host.cpp"),
            "-L" + HERE, "-l:librdk_b200.so", "-Wl,-rpath,$ORIGIN", "-L" + libdir, "-ltorch_python", "-ltorch_cpu", "-ltorch", "-lc10", "-lc10_cuda"]


def build(force: bool = False, verbose: bool = False) -> str:
    """Build the shared library if it is missing or older than a source; return its path."""
    if not force and not _stale():
        return LIB
    flags = ["-Xcompiler", "-fPIC", "-std=c++17", "-O3", "-lineinfo", "-gencode", "arch=compute_100a,code=sm_100a",
             "-I", os.path.join(ROOT, "include"), "-I", CSRC]
    if verbose:
        flags += ["-Xptxas", "-v"]
    nvcc = _nvcc()

    def run(cmd):
        res = subprocess.run(cmd, capture_output=True, text=True)
        if res.returncode != 0:
            raise RuntimeError("nvcc failed:\n" + res.stdout + res.stderr)
        return res.stdout + res.stderr

    with tempfile.TemporaryDirectory() as tmp:      # one compiler process per source file, side by side
        objs = [os.path.join(tmp, s + ".o") for s in SOURCES]
        with ThreadPoolExecutor(max_workers=min(len(SOURCES), os.cpu_count() or 1)) as pool:
            logs = list(pool.map(lambda so: run([nvcc, "-c", *flags, os.path.join(CSRC, so[0]), "-o", so[1]]), zip(SOURCES, objs)))
        logs.append(run([nvcc, "-shared", *flags, *objs, "-o", LIB]))
        logs.append(run([*_host_command(), "-o", HOST]))
    if verbose:
        print("".join(logs))
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
