"""Builds liblq.so (the C-ABI CUDA library) in-tree with nvcc for sm_100a, and _native.so, the module that takes torch
tensors to its calls, with the host compiler."""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
OUT = os.path.join(HERE, "liblq.so")
NATIVE = os.path.join(HERE, "_native.so")
# (source, extra flags).  The level fit is compiled without FMA contraction.
SOURCES = [("lq_api.cu", []), ("lq_norm.cu", []), ("lq_quantize.cu", []), ("lq_quantize_small.cu", []), ("lq_quantize_bucket.cu", []), ("lq_decode.cu", []), ("lq_noalloc.cu", []), ("lq_coding.cu", []), ("lq_encode_by_width.cu", []),
           ("lq_fit.cu", ["-fmad=false"]), ("lq_codelen.cu", ["-fmad=false"])]
NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "-Xcompiler", "-fPIC", "-I", os.path.join(ROOT, "include"), "-I", CSRC]


def _stale() -> bool:
    if not os.path.exists(OUT) or not os.path.exists(NATIVE):
        return True
    t = min(os.path.getmtime(OUT), os.path.getmtime(NATIVE))
    deps = [__file__] + [os.path.join(CSRC, f) for f in os.listdir(CSRC)] + [os.path.join(ROOT, "include", "lq.h")]
    return any(os.path.getmtime(d) > t for d in deps)


def _native_compile(obj: str) -> list:
    import torch
    from torch.utils import cpp_extension as ext
    include = [f for d in (*ext.include_paths(), os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include"),
                           sysconfig.get_paths()["include"], os.path.join(ROOT, "include")) for f in ("-isystem", d)]
    return ["g++", "-O2", "-std=c++17", "-fPIC", *include, f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
            "-c", os.path.join(CSRC, "lq_native.cpp"), "-o", obj]


def _native_link(obj: str, out: str) -> list:
    """Against liblq.so beside it (the same file that binding.py opens)."""
    import torch
    return ["g++", "-shared", obj, "-o", out, "-L", HERE, "-l:liblq.so", "-Wl,-rpath,$ORIGIN",
            "-L", os.path.join(os.path.dirname(torch.__file__), "lib"), "-ltorch_python", "-ltorch", "-ltorch_cpu", "-lc10",
            "-lc10_cuda"]


def _outdated(src: str, obj: str, common: float) -> bool:
    """(an object as old as its source counts as outdated: the clock of a file system may be coarse)"""
    return not os.path.exists(obj) or os.path.getmtime(obj) <= max(common, os.path.getmtime(src))


def build(force: bool = False, verbose: bool = False) -> str:
    if not force and not _stale():
        return OUT
    nvcc = os.environ.get("NVCC", "nvcc")
    bdir = os.path.join(HERE, "_build")
    os.makedirs(bdir, exist_ok=True)
    # what every object hangs on: the headers, and this file's flags
    common = max([os.path.getmtime(__file__)] + [os.path.getmtime(os.path.join(d, f)) for d in (CSRC, os.path.join(ROOT, "include"))
                                                 for f in os.listdir(d) if f.endswith((".cuh", ".h"))])
    objs, procs = [], []
    native_obj = os.path.join(bdir, "lq_native.o")
    jobs = [(os.path.join(CSRC, "lq_native.cpp"), native_obj, lambda: _native_compile(native_obj))]
    for src, extra in SOURCES:
        obj = os.path.join(bdir, src.replace(".cu", ".o"))
        cmd = [nvcc, *NVCC_FLAGS, *extra, *(["-Xptxas", "-v"] if verbose else []), "-c", os.path.join(CSRC, src), "-o", obj]
        jobs.append((os.path.join(CSRC, src), obj, lambda cmd=cmd: cmd))
        objs.append(obj)
    for src, obj, command in jobs:
        if force or _outdated(src, obj, common):
            cmd = command()
            procs.append((cmd, obj, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)))
    failed = []
    for cmd, obj, p in procs:
        out, _ = p.communicate()
        if verbose or p.returncode:
            sys.stderr.write(out)
        if p.returncode:
            failed.append(" ".join(cmd))
            if os.path.exists(obj):
                os.remove(obj)
    if failed:
        raise RuntimeError("compiler failed: " + "; ".join(failed))
    tmp = f".{os.getpid()}.tmp"
    subprocess.check_call([nvcc, "-shared", "-o", OUT + tmp, *objs, "-gencode", "arch=compute_100a,code=sm_100a"])
    os.replace(OUT + tmp, OUT)
    subprocess.check_call(_native_link(native_obj, NATIVE + tmp))
    os.replace(NATIVE + tmp, NATIVE)
    return OUT


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
