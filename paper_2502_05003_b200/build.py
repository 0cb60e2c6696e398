"""Builds the CUDA library in-tree: ``python -m paper_2502_05003_b200.build``.

nvcc cross-compiles for sm_100a without a GPU.  The quantizer is compiled with ``-fmad=false``
(its binary32 operation order is part of the contract), and so is the decoding layer that repeats it; everything
else with defaults.
"""
from __future__ import annotations

import os
import re
import shutil
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
INCLUDE = os.path.join(os.path.dirname(HERE), "include")
OBJ_DIR = os.path.join(HERE, "_build")
LIB = os.path.join(HERE, "libquest_b200.so")

ARCH = ["-gencode", "arch=compute_100a,code=sm_100a"]
COMMON = ["-O3", "-std=c++17", "-lineinfo", "-Xcompiler", "-fPIC", "-I", INCLUDE, "-I", CSRC]
UNITS = {
    "quest_api.cu": [],
    "quest_quantize.cu": ["-fmad=false"],
    "quest_decode.cu": ["-fmad=false"],
    "quest_gemm.cu": [],
    "quest_static.cu": [],
    "quest_backward.cu": [],
    "quest_weight_only.cu": [],
}


def _newer(src_paths, target):
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    return any(os.path.getmtime(p) > t for p in src_paths)


def build(force: bool = False, verbose: bool = False) -> str:
    nvcc = os.environ.get("NVCC", "nvcc")
    os.makedirs(OBJ_DIR, exist_ok=True)
    headers = [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith((".cuh", ".h"))]
    headers.append(os.path.join(INCLUDE, "quest.h"))
    objs = []
    for unit, extra in UNITS.items():
        src = os.path.join(CSRC, unit)
        obj = os.path.join(OBJ_DIR, unit.replace(".cu", ".o"))
        objs.append(obj)
        if force or _newer([src] + headers, obj):
            cmd = [nvcc] + ARCH + COMMON + extra + (["-Xptxas", "-v"] if verbose else []) + ["-c", src, "-o", obj]
            subprocess.check_call(cmd)
    if force or _newer(objs, LIB):
        tmp = LIB + f".{os.getpid()}.tmp"
        subprocess.check_call([nvcc] + ARCH + ["-shared", "-o", tmp] + objs)
        os.replace(tmp, LIB)
    build_binding(force)
    return LIB


def binding_name() -> str:
    """Module name of the CPython binding for the installed torch: an object compiled against another one is not found."""
    import torch
    return "_binding_torch_" + re.sub(r"\W", "_", torch.__version__)


def build_binding(force: bool = False):
    """The CPython binding of the per-layer calls: host code over the C ABI, compiled against torch's headers.  Without a
    CUDA build of torch there is none (None is returned): the package goes through ctypes."""
    try:
        import torch
    except ImportError:
        return None
    if torch.version.cuda is None:
        return None
    name = binding_name()
    target = os.path.join(HERE, name + sysconfig.get_config_var("EXT_SUFFIX"))
    src = os.path.join(CSRC, "quest_binding.cpp")
    if not (force or _newer([src, os.path.join(INCLUDE, "quest.h")], target)):
        return target
    root = os.path.dirname(torch.__file__)
    cuda = os.path.dirname(os.path.dirname(os.path.realpath(shutil.which(os.environ.get("NVCC", "nvcc")))))
    includes = [os.path.join(root, "include"), os.path.join(root, "include", "torch", "csrc", "api", "include"),
                sysconfig.get_paths()["include"], os.path.join(cuda, "include"), INCLUDE]
    tmp = target + f".{os.getpid()}.tmp"
    cmd = [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-fPIC", "-shared", "-fvisibility=hidden",
           f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}", f"-DQUEST_BINDING={name}"]
    for inc in includes:
        cmd += ["-isystem", inc]
    cmd += [src, "-o", tmp, "-L", HERE, "-l:libquest_b200.so", "-L", os.path.join(root, "lib"), "-ltorch_python", "-ltorch_cpu",
            "-lc10_cuda", "-lc10", "-Wl,-rpath,$ORIGIN"]
    subprocess.check_call(cmd)
    os.replace(tmp, target)
    return target


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
