"""Builds libgnn_b200.so (nvcc, sm_100a only), the Python extension in front of it and the input-generator library, in-tree.

    python -m paper_2412_06354_b200.build [--force]
"""
from __future__ import annotations

import glob
import os
import subprocess
import sys
from concurrent.futures import ThreadPoolExecutor

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
OBJ = os.path.join(ROOT, "_build")
LIB = os.path.join(HERE, "libgnn_b200.so")
NVCC = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-O3", "-lineinfo", "-std=c++17",
         "-Xcompiler", "-fPIC", "-I" + os.path.join(ROOT, "include"), "-I" + CSRC,
         *os.environ.get("GNN_NVCC_FLAGS", "").split()]


BINDING = os.path.join(HERE, "_binding.so")
BINDING_KEY = os.path.join(OBJ, "binding.key")  # what the extension was built against


def _newest(paths):
    return max(os.path.getmtime(p) for p in paths)


def build(force: bool = False, verbose: bool = False) -> str:
    srcs = sorted(glob.glob(os.path.join(CSRC, "*.cu")))
    hdrs = glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(CSRC, "*.h")) + glob.glob(os.path.join(ROOT, "include", "*.h"))
    os.makedirs(OBJ, exist_ok=True)
    dep_time = _newest(hdrs)
    jobs = []
    objs = []
    for s in srcs:
        o = os.path.join(OBJ, os.path.basename(s)[:-3] + ".o")
        objs.append(o)
        if force or not os.path.exists(o) or os.path.getmtime(o) < max(os.path.getmtime(s), dep_time):
            jobs.append([NVCC, *FLAGS, *(["-Xptxas", "-v"] if verbose else []), "-c", s, "-o", o])
    if jobs:
        with ThreadPoolExecutor(max_workers=min(len(jobs), os.cpu_count() or 4)) as ex:
            for r in ex.map(lambda c: subprocess.run(c, capture_output=True, text=True), jobs):
                if verbose or r.returncode != 0:
                    sys.stderr.write(r.stdout + r.stderr)
                if r.returncode != 0:
                    raise RuntimeError("nvcc failed: " + " ".join(r.args))
    if jobs or not os.path.exists(LIB):
        subprocess.check_call([NVCC, "-gencode", "arch=compute_100a,code=sm_100a", "-shared", "-Xlinker=-soname,libgnn_b200.so", "-o", LIB, *objs])
    build_binding(force)
    from . import synth
    synth.build(force)
    return LIB


def build_binding(force: bool = False) -> str:
    """The CPython extension (host code only) that gnn.py calls; linked against libgnn_b200.so beside it and torch."""
    import sysconfig
    import torch
    src = os.path.join(CSRC, "binding.cpp")
    # the extension uses torch's C++ interface, which another version or Python need not share
    key = " ".join(map(str, (torch.__version__, int(torch._C._GLIBCXX_USE_CXX11_ABI), sysconfig.get_config_var("SOABI"))))
    built = open(BINDING_KEY).read() if os.path.exists(BINDING_KEY) else None
    if not force and built == key and os.path.exists(BINDING) and os.path.getmtime(BINDING) >= _newest([src, os.path.join(ROOT, "include", "gnn.h")]):
        return BINDING
    tdir = os.path.dirname(torch.__file__)
    inc = [os.path.join(ROOT, "include"), os.path.join(tdir, "include"), os.path.join(tdir, "include", "torch", "csrc", "api", "include"),
           sysconfig.get_paths()["include"], os.path.join(os.path.dirname(os.path.dirname(NVCC)), "include")]
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-fvisibility=hidden", *["-I" + d for d in inc],
                           f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}", src, "-o", BINDING,
                           "-L" + HERE, "-l:libgnn_b200.so", "-Wl,-rpath,$ORIGIN", "-L" + os.path.join(tdir, "lib"),
                           "-lc10", "-lc10_cuda", "-ltorch_cpu", "-ltorch_cuda", "-ltorch_python"])
    os.makedirs(OBJ, exist_ok=True)
    with open(BINDING_KEY, "w") as f:
        f.write(key)
    return BINDING


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
