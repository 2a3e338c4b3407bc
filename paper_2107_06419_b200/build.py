"""Compile libflat_attn.so for sm_100a with nvcc, and the extension module _binding that calls it (in-tree, next to this file)."""
from __future__ import annotations

import os
import shutil
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libflat_attn.so")
SOURCES = ["flat_attn_api.cu", "simt_kernels.cu", "fused_tc.cu", "fused_tc2.cu", "fused_tc3.cu", "fused_rgran.cu", "proj_gemm.cu", "naive_tc.cu", "naive_static.cu", "bwd_tc.cu", "layernorm.cu", "fused_tf32.cu", "fused_small.cu", "fused_decode.cu", "fused_d128.cu"]
HEADERS = ["flat_internal.cuh", "ptx_sm100.cuh", "tc_common.cuh", os.path.join("..", "..", "include", "flat_attn.h")]


def nvcc_path() -> str:
    for cand in (shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found: libflat_attn.so cannot be built")


BINDING = os.path.join(HERE, "_binding" + sysconfig.get_config_var("EXT_SUFFIX"))   # (the name says which Python it is for)
BINDING_FLAGS = ["-O2", "-std=c++17", "-shared", "-fPIC"]


def _older(target: str, deps) -> bool:
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    return any(os.path.getmtime(d) > t for d in deps)


def is_stale() -> bool:
    return _older(LIB, [os.path.join(CSRC, s) for s in SOURCES + HEADERS])


def build_library(verbose: bool = False) -> None:
    tmp = LIB + ".%d.tmp" % os.getpid()
    cmd = [nvcc_path(), "-gencode", "arch=compute_100a,code=sm_100a", "-O3", "-std=c++17", "-lineinfo",
           "-shared", "-Xcompiler", "-fPIC", "-cudart", "static", "--threads", "0"]
    if verbose:
        cmd += ["-Xptxas", "-v"]
    cmd += [os.path.join(CSRC, s) for s in SOURCES] + ["-o", tmp]
    subprocess.check_call(cmd)
    os.replace(tmp, LIB)


def binding_key() -> str:
    """What the extension module is compiled against: it reads torch's tensors through torch's C++ headers and libraries."""
    import torch
    return "flat_attn binding for torch %s, %s" % (torch.__version__, " ".join(BINDING_FLAGS))


def binding_is_stale() -> bool:
    if _older(BINDING, [os.path.join(CSRC, "binding.cpp"), os.path.join(HERE, "..", "include", "flat_attn.h")]):
        return True
    with open(BINDING, "rb") as f:                       # (the module holds its key as a string)
        return binding_key().encode() not in f.read()


def build_binding() -> None:
    """The extension module next to the library, which it is linked against (found through its own folder)."""
    import torch
    root = os.path.dirname(torch.__file__)
    include = [os.path.join(root, "include"), os.path.join(root, "include", "torch", "csrc", "api", "include"),
               os.path.join(os.path.dirname(os.path.dirname(nvcc_path())), "include"), sysconfig.get_paths()["include"]]
    tmp = BINDING + ".%d.tmp" % os.getpid()
    subprocess.check_call(["g++"] + BINDING_FLAGS + ["-I" + d for d in include] + ['-DBINDING_KEY="%s"' % binding_key(),
                          os.path.join(CSRC, "binding.cpp"), "-o", tmp, "-L" + os.path.join(root, "lib"), "-lc10",
                          "-lc10_cuda", "-ltorch_cpu", "-ltorch_python", "-L" + HERE, "-l:libflat_attn.so",
                          "-Wl,-rpath,$ORIGIN"])
    os.replace(tmp, BINDING)


def build(force: bool = False, verbose: bool = False) -> str:
    if force or is_stale():
        build_library(verbose)
    if force or binding_is_stale():
        build_binding()
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
