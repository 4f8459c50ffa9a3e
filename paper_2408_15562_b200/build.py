"""Build libfspad.so (sm_100a) in-tree with nvcc.  `python -m paper_2408_15562_b200.build`."""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
LIB = os.path.join(PKG, "libfspad.so")
HEADER = os.path.join(ROOT, "include", "fspad.h")
CALLS_SRC = os.path.join(CSRC, "pycall.cpp")
SOURCES = ["api.cu", "accept_stats.cu", "accept_walk.cu", "kv_compact.cu", "tree_attn.cu", "tree_attn_umma.cu", "tree_build.cu", "draft_expand.cu", "lm_head.cu", "feature_sampler.cu"]
NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "-Xcompiler", "-fPIC", "-I" + os.path.join(ROOT, "include"), "-I" + CSRC]


def _nvcc() -> str:
    for cand in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", "nvcc"):
        if cand and (os.path.isabs(cand) and os.path.exists(cand) or not os.path.isabs(cand)):
            return cand
    return "nvcc"


def _newest_source() -> float:
    files = [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f != os.path.basename(CALLS_SRC)] + [HEADER]
    return max(os.path.getmtime(f) for f in files)


def calls_path() -> str:
    """The Python calls are built for one torch and one interpreter, which the file's name says: another torch lays out its tensors
    in another way, and must not come upon this file."""
    import torch
    return os.path.join(PKG, "_pycall.torch-%s%s" % (torch.__version__, sysconfig.get_config_var("EXT_SUFFIX")))


def _build_calls(force: bool) -> None:
    """The Python calls of the C ABI (g++ against torch's headers), linked with the library beside it.  torch's own libraries are in
    the process by the time it is imported and are found by their names."""
    calls = calls_path()
    if not force and os.path.exists(calls) and os.path.getmtime(calls) >= max(os.path.getmtime(CALLS_SRC), os.path.getmtime(HEADER)):
        return
    import torch
    t = os.path.dirname(torch.__file__)
    tmp = calls + ".tmp.%d" % os.getpid()
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-I" + os.path.dirname(HEADER),
                           "-I" + os.path.join(t, "include"), "-I" + os.path.join(t, "include", "torch", "csrc", "api", "include"),
                           "-I" + sysconfig.get_paths()["include"], "-D_GLIBCXX_USE_CXX11_ABI=%d" % torch._C._GLIBCXX_USE_CXX11_ABI,
                           CALLS_SRC, "-o", tmp, "-L" + PKG, "-l:" + os.path.basename(LIB), "-L" + os.path.join(t, "lib"),
                           "-ltorch_python", "-ltorch_cpu", "-lc10", "-Wl,-rpath,$ORIGIN"])
    os.replace(tmp, calls)
    for f in os.listdir(PKG):
        if f.startswith("_pycall") and f.endswith(".so") and f != os.path.basename(calls):
            os.remove(os.path.join(PKG, f))


def build(force: bool = False, verbose: bool = False) -> str:
    _build_library(force, verbose)
    _build_calls(force)
    return LIB


def _build_library(force: bool, verbose: bool) -> None:
    if not force and os.path.exists(LIB) and os.path.getmtime(LIB) >= _newest_source():
        return
    objdir = os.path.join(PKG, "_build")
    os.makedirs(objdir, exist_ok=True)
    procs = []
    objs = []
    for src in SOURCES:
        obj = os.path.join(objdir, src.replace(".cu", ".o"))
        objs.append(obj)
        cmd = [_nvcc()] + NVCC_FLAGS + (["-Xptxas", "-v"] if verbose else []) + \
              ["-c", os.path.join(CSRC, src), "-o", obj]
        procs.append((src, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)))
    failed = False
    for src, p in procs:
        out, _ = p.communicate()
        if verbose or p.returncode != 0:
            sys.stderr.write("== %s ==\n%s\n" % (src, out))
        failed |= p.returncode != 0
    if failed:
        raise RuntimeError("nvcc failed")
    tmp = LIB + ".tmp.%d" % os.getpid()
    subprocess.check_call([_nvcc(), "-gencode", "arch=compute_100a,code=sm_100a", "-shared", "-o", tmp] + objs)
    os.replace(tmp, LIB)


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
