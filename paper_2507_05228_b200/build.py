"""Builds the CUDA library (sm_100a) in-tree with nvcc.  `python -m paper_2507_05228_b200.build [--force] [--debug]`.

--debug builds libcascade_b200_debug.so with -DCASCADE_DEBUG: every row index a kernel reads out of a plan array is
checked before it forms an address (a bad one lands in the plan's status word).  Load it by setting the environment
variable CASCADE_B200_LIB to its path before importing the binding."""
from __future__ import annotations

import os
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libcascade_b200.so")
FASTCALL = os.path.join(HERE, "_fastcall.so")
LIB_DEBUG = os.path.join(HERE, "libcascade_b200_debug.so")
SOURCES = ["cascade_api.cu", "merge.cu", "attn_simt.cu", "attn_rows.cu", "attn_tc.cu", "attn_split.cu", "gather.cu", "decode.cu", "decode_static.cu",
           "shard_maps.cu", "rope.cu", "plan_advance.cu"]
NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
    "-Xcompiler", "-fPIC", "-Xptxas", "-v", "-I", os.path.join(ROOT, "include"), "-I", CSRC,
]


def _nvcc() -> str:
    for cand in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", "nvcc"):
        if cand and (os.path.isabs(cand) and os.path.exists(cand) or not os.path.isabs(cand)):
            return cand
    return "nvcc"


def _stale(lib: str = LIB) -> bool:
    if not os.path.exists(lib):
        return True
    t = os.path.getmtime(lib)
    deps = [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f != "fastcall.cpp"] + [os.path.join(ROOT, "include", "cascade.h"), __file__]
    return any(os.path.getmtime(d) > t for d in deps)


def _build_fastcall(force: bool) -> None:
    """Compile csrc/fastcall.cpp (the native side of binding.py) against this interpreter and torch."""
    src = os.path.join(CSRC, "fastcall.cpp")
    if not force and os.path.exists(FASTCALL):
        t = os.path.getmtime(FASTCALL)
        if all(os.path.getmtime(d) <= t for d in (src, os.path.join(ROOT, "include", "cascade.h"), __file__)):
            return
    import sysconfig

    import torch
    base = os.path.dirname(torch.__file__)
    inc = [sysconfig.get_paths()["include"], os.path.join(base, "include"),
           os.path.join(base, "include", "torch", "csrc", "api", "include"),
           os.path.join(os.path.dirname(os.path.dirname(_nvcc())), "include"), os.path.join(ROOT, "include")]
    tmp = FASTCALL + f".{os.getpid()}.tmp"
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-fvisibility=hidden", "-w",
                           f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
                           *[f"-I{i}" for i in inc], src, "-o", tmp, f"-L{os.path.join(base, 'lib')}",
                           "-ltorch_python", "-ltorch", "-ltorch_cpu", "-lc10", "-lc10_cuda", "-ldl"])
    os.replace(tmp, FASTCALL)


def build_library(force: bool = False, verbose: bool = False, debug: bool = False) -> str:
    """Compile every .cu file for sm_100a and link libcascade_b200.so (or the _debug variant) next to this file."""
    _build_fastcall(force and not debug)
    lib = LIB_DEBUG if debug else LIB
    if not force and not _stale(lib):
        return lib
    objdir = os.path.join(HERE, "_build_debug" if debug else "_build")
    os.makedirs(objdir, exist_ok=True)
    objs, procs = [], []
    for src in SOURCES:
        obj = os.path.join(objdir, src.replace(".cu", ".o"))
        objs.append(obj)
        cmd = [_nvcc(), *NVCC_FLAGS, *(["-DCASCADE_DEBUG"] if debug else []), "-c", os.path.join(CSRC, src), "-o", obj]
        procs.append((src, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)))
    log = []
    failed = False
    for src, pr in procs:
        out, _ = pr.communicate()
        log.append(f"== {src}\n{out}")
        failed |= pr.returncode != 0
    with open(os.path.join(objdir, "ptxas.log"), "w") as f:
        f.write("\n".join(log))
    if failed or verbose:
        sys.stderr.write("\n".join(log))
    if failed:
        raise RuntimeError("nvcc failed; see output above")
    tmp = lib + f".{os.getpid()}.tmp"
    subprocess.check_call([_nvcc(), "-shared", "-o", tmp, *objs, "-gencode", "arch=compute_100a,code=sm_100a"])
    os.replace(tmp, lib)
    return lib


if __name__ == "__main__":
    print(build_library(force="--force" in sys.argv, verbose="-v" in sys.argv, debug="--debug" in sys.argv))
