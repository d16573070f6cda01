"""Compile the CUDA sources into ``libmassv.so`` for sm_100a with nvcc, and the binding's argument marshalling with g++."""
from __future__ import annotations

import os
import runpy
import subprocess
import sys
import sysconfig

PKG = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(PKG, "csrc")
INCLUDE = os.path.join(os.path.dirname(PKG), "include")
LIB = os.path.join(PKG, "libmassv.so")
SOURCES = ["api.cu", "attn.cu", "attn_umma.cu", "lm_head.cu", "accept.cu", "accept_static.cu", "tensor_map.cu", "tvd.cu", "top_p.cu"]


TEST_LIB = os.path.join(PKG, "libmassv_testhooks.so")
DEBUG_LIB = os.path.join(PKG, "libmassv_debug.so")


def _torch_dir() -> str:
    import importlib.util
    return os.path.dirname(importlib.util.find_spec("torch").origin)          # (without importing torch: that takes seconds)


def marshal_path() -> str:
    """The native module's file.  It is compiled against the layout of torch's and Python's objects, so their versions are in its name:
    after an update of either the old file is not the one that is looked for, and the build makes another."""
    torch_version = runpy.run_path(os.path.join(_torch_dir(), "version.py"))["__version__"]
    return os.path.join(PKG, f"_marshal.torch-{torch_version}{sysconfig.get_config_var('EXT_SUFFIX')}")


def _stale(lib=LIB) -> bool:
    if not os.path.exists(lib):
        return True
    t = os.path.getmtime(lib)
    deps = [os.path.join(CSRC, f) for f in os.listdir(CSRC)] + [os.path.join(INCLUDE, "massv.h")]
    return any(os.path.getmtime(d) > t for d in deps)


def _command(out, extra, verbose=False):
    nvcc = os.environ.get("NVCC", "nvcc")
    cmd = [nvcc, "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
           "-shared", "-Xcompiler", "-fPIC", "-I", INCLUDE, "-I", CSRC] + extra + \
          ["-o", out] + [os.path.join(CSRC, s) for s in SOURCES] + ["-ldl"]
    if verbose:
        cmd.insert(1, "-Xptxas=-v")
    return cmd


def _compile(out, extra, verbose=False):
    subprocess.run(_command(out, extra, verbose), check=True)
    return out


VARIANTS = {LIB: [], TEST_LIB: ["-DMASSV_TEST_HOOKS", "-DMASSV_SPIN_LIMIT=65536u"], DEBUG_LIB: ["-DMASSV_DEBUG"]}


def _marshal_command():
    """The extension module against torch's own headers and libraries."""
    torch_dir = _torch_dir()
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    include = [sysconfig.get_paths()["include"], os.path.join(torch_dir, "include"),
               os.path.join(torch_dir, "include", "torch", "csrc", "api", "include"), os.path.join(cuda, "include")]
    return ([os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-shared", "-fPIC", "-I", INCLUDE] + [x for d in include for x in ("-isystem", d)] +
            ["-o", marshal_path(), os.path.join(CSRC, "marshal.cpp"), "-L", os.path.join(torch_dir, "lib"), "-ltorch_python", "-ltorch_cpu", "-lc10_cuda", "-lc10"])


def build_all(force: bool = False):
    """The library, its two test variants and the marshalling module, the stale ones compiled side by side."""
    commands = {lib: _command(lib, extra) for lib, extra in VARIANTS.items()}
    commands[marshal_path()] = _marshal_command()
    procs = [(out, subprocess.Popen(cmd)) for out, cmd in commands.items() if force or _stale(out)]
    for out, proc in procs:
        if proc.wait() != 0:
            raise subprocess.CalledProcessError(proc.returncode, "compiler -o " + out)
    return list(commands)


def build(force: bool = False, verbose: bool = False) -> str:
    if force or _stale(marshal_path()):
        subprocess.run(_marshal_command(), check=True)
    if not (force or _stale()):
        return LIB
    return _compile(LIB, [], verbose)


def build_test_hooks(force: bool = False) -> str:
    """The same sources with the test hooks compiled in and a short limit on device-side waits: only
    the tests load it (to make a bounded wait run out on purpose, on a tiny problem)."""
    if not (force or _stale(TEST_LIB)):
        return TEST_LIB
    return _compile(TEST_LIB, ["-DMASSV_TEST_HOOKS", "-DMASSV_SPIN_LIMIT=65536u"])


def build_debug(force: bool = False) -> str:
    """The same sources with -DMASSV_DEBUG: index checks on the device that record MASSV_ERR_BOUNDS in the status
    word and skip the access.  The binding loads it instead of the ordinary library when MASSV_DEBUG=1 is set."""
    if not (force or _stale(DEBUG_LIB)):
        return DEBUG_LIB
    return _compile(DEBUG_LIB, VARIANTS[DEBUG_LIB])


if __name__ == "__main__":
    force = "--force" in sys.argv
    print("\n".join([build(force, verbose=True)] if "-v" in sys.argv else build_all(force)))
