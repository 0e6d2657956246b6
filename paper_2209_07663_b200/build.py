"""Build the CUDA shared library (libmono.so) in-tree for sm_100a with nvcc, and the small CPython
extension that hands tensors to it."""
from __future__ import annotations

import glob
import os
import re
import shutil
import subprocess
import sysconfig

PKG = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(PKG, "csrc")
LIB = os.path.join(PKG, "libmono.so")
# the same sources with -DMONO_DEBUG: every index the library computes for itself is range-checked
# on the device and a bad one reported through the status bits (binding: MONO_LIBRARY=checked)
LIB_CHECKED = os.path.join(PKG, "libmono_checked.so")
# the hot calls' Python side; touches no table and needs no nvcc
NATIVE_SOURCE = os.path.join(CSRC, "binding_native.cpp")

NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "-shared", "-Xcompiler", "-fPIC", "--cudart", "static", "-ldl"]


def _sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _newest_input() -> float:
    files = glob.glob(os.path.join(CSRC, "*.cu*")) + [os.path.join(PKG, "..", "include", "mono.h")]
    return max(os.path.getmtime(f) for f in files)


def find_nvcc() -> str:
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        raise RuntimeError("nvcc not found: the CUDA library cannot be built")
    return nvcc


def native_path() -> str:
    """Where the extension for this Python and this torch is, once it is built: it is compiled against both, so a build
    made for others has another name and is neither reused nor loaded."""
    import torch
    tag = f"{sysconfig.get_config_var('SOABI')}-torch-{torch.__version__}"
    return os.path.join(PKG, f"_binding_native.{re.sub('[^0-9A-Za-z._-]', '_', tag)}.so")


def build_native(force: bool = False) -> str:
    """Compile csrc/binding_native.cpp against the torch that is installed, unless it is up to date."""
    native = native_path()
    if not force and os.path.exists(native) and os.path.getmtime(native) >= os.path.getmtime(NATIVE_SOURCE):
        return native
    import torch
    from torch.utils import cpp_extension
    tmp = f"{native}.{os.getpid()}.tmp"
    lib_dir = os.path.join(os.path.dirname(torch.__file__), "lib")
    cmd = [shutil.which("g++") or "g++", "-O2", "-std=c++17", "-shared", "-fPIC",
           f"-D_GLIBCXX_USE_CXX11_ABI={int(torch.compiled_with_cxx11_abi())}",
           *[f"-isystem{d}" for d in cpp_extension.include_paths()], f"-I{sysconfig.get_paths()['include']}",
           NATIVE_SOURCE, "-o", tmp, f"-L{lib_dir}", "-ltorch_python", "-ltorch_cpu", "-ltorch", "-lc10"]
    subprocess.check_call(cmd)
    os.replace(tmp, native)
    return native


def build(force: bool = False, verbose: bool = False, checked: bool = False) -> str:
    """Compile csrc/*.cu into libmono.so (or, with `checked`, into libmono_checked.so) unless it is
    already up to date.  The Python side of the hot calls comes with it."""
    build_native(force=force and not checked)
    lib = LIB_CHECKED if checked else LIB
    if not force and os.path.exists(lib) and os.path.getmtime(lib) >= _newest_input():
        return lib
    tmp = f"{lib}.{os.getpid()}.tmp"
    cmd = [find_nvcc(), *NVCC_FLAGS, *(["-DMONO_DEBUG"] if checked else []), "-o", tmp, *_sources()]
    if verbose:
        cmd.insert(1, "-Xptxas")
        cmd.insert(2, "-v")
    subprocess.check_call(cmd)
    os.replace(tmp, lib)
    return lib


if __name__ == "__main__":
    print(build(force=True, verbose=True))
    print(build(force=True, checked=True))
