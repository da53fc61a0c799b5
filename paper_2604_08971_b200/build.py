"""Build libsentry.so in-tree with nvcc for sm_100a (cross-compiles without a GPU), and the native binding beside it."""
from __future__ import annotations

import glob
import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libsentry.so")
BINDING = os.path.join(HERE, "_binding.so")
BINDING_SRC = os.path.join(CSRC, "binding.cpp")
NVCC = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
         "-Xcompiler", "-fPIC",
         "-shared", "-Xcompiler", "-fvisibility=hidden", "-Xcompiler", "-Wall"]


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _older(target, deps) -> bool:
    return not os.path.exists(target) or any(os.path.getmtime(p) > os.path.getmtime(target) for p in deps)


HEADER = os.path.join(os.path.dirname(HERE), "include", "sentry.h")


def needs_build() -> bool:
    return _older(LIB, sources() + glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(CSRC, "ptx", "*.cuh"))
                  + [HEADER]) or _older(BINDING, [BINDING_SRC, HEADER])


def _compile(cmd, target):
    tmp = target + ".tmp%d" % os.getpid()
    res = subprocess.run(cmd + ["-o", tmp], capture_output=True, text=True)
    if res.returncode != 0:
        raise RuntimeError("%s failed:\n" % cmd[0] + res.stdout + res.stderr)
    os.replace(tmp, target)
    return res.stderr


def build_binding():
    """_binding.so: C++ against the Python and torch headers, linked to libsentry.so beside it."""
    import torch
    root = os.path.dirname(torch.__file__)
    inc = [os.path.join(root, "include"), os.path.join(root, "include", "torch", "csrc", "api", "include"),
           sysconfig.get_paths()["include"], os.path.join(os.path.dirname(os.path.dirname(NVCC)), "include")]
    cmd = ["g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-fvisibility=hidden", "-w",
           "-D_GLIBCXX_USE_CXX11_ABI=%d" % int(torch._C._GLIBCXX_USE_CXX11_ABI)]
    cmd += [f for p in inc for f in ("-isystem", p)] + [BINDING_SRC]
    cmd += ["-L" + HERE, "-l:" + os.path.basename(LIB), "-L" + os.path.join(root, "lib"), "-lc10", "-lc10_cuda", "-ltorch_cpu",
            "-ltorch_python"]
    _compile(cmd + ["-Wl,-rpath,$ORIGIN"], BINDING)


def build(force: bool = False, verbose: bool = False) -> str:
    if not force and not needs_build():
        return LIB
    err = _compile([NVCC] + FLAGS + (["-Xptxas", "-v"] if verbose else []) + sources(), LIB)
    if verbose:
        sys.stderr.write(err)
    build_binding()
    return LIB


if __name__ == "__main__":
    print(build(force=True, verbose="-v" in sys.argv))
