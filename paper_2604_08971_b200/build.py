"""Build libsentry.so in-tree with nvcc for sm_100a (cross-compiles without a GPU), and the native binding beside it."""
from __future__ import annotations

import glob
import os
import subprocess
import sys
import sysconfig
from importlib import metadata

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libsentry.so")
BINDING = os.path.join(HERE, "_binding.so")
BINDING_SRC = os.path.join(CSRC, "binding.cpp")
BINDING_STAMP = BINDING + ".stamp"   # what the binding was compiled against
NVCC = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
         "-Xcompiler", "-fPIC",
         "-shared", "-Xcompiler", "-fvisibility=hidden", "-Xcompiler", "-Wall"]


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _older(target, deps) -> bool:
    return not os.path.exists(target) or any(os.path.getmtime(p) > os.path.getmtime(target) for p in deps)


HEADER = os.path.join(os.path.dirname(HERE), "include", "sentry.h")


def _lib_stale() -> bool:
    return _older(LIB, sources() + glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(CSRC, "ptx", "*.cuh"))
                  + [HEADER])


def _built_against() -> str:
    return "torch %s python %s" % (metadata.version("torch"), sysconfig.get_config_var("EXT_SUFFIX"))


def _binding_stale() -> bool:
    if _older(BINDING, [BINDING_SRC, HEADER]) or not os.path.exists(BINDING_STAMP):
        return True
    with open(BINDING_STAMP) as f:
        return f.read() != _built_against()


def needs_build() -> bool:
    return _lib_stale() or _binding_stale()


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
    cmd = ["g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-fvisibility=hidden", "-Wall", "-Wextra",
           "-D_GLIBCXX_USE_CXX11_ABI=%d" % int(torch._C._GLIBCXX_USE_CXX11_ABI)]
    cmd += [f for p in inc for f in ("-isystem", p)] + [BINDING_SRC]
    cmd += ["-L" + HERE, "-l:" + os.path.basename(LIB), "-L" + os.path.join(root, "lib"), "-lc10", "-lc10_cuda", "-ltorch_cpu",
            "-ltorch_python"]
    err = _compile(cmd + ["-Wl,-rpath,$ORIGIN"], BINDING)
    with open(BINDING_STAMP, "w") as f:
        f.write(_built_against())
    return err


def build(force: bool = False, verbose: bool = False) -> str:
    err = ""
    if force or _lib_stale():
        err += _compile([NVCC] + FLAGS + (["-Xptxas", "-v"] if verbose else []) + sources(), LIB)
    if force or _binding_stale():
        err += build_binding()
    if verbose:
        sys.stderr.write(err)
    return LIB


if __name__ == "__main__":
    print(build(force=True, verbose="-v" in sys.argv))
