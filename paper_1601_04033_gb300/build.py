"""Compile the CUDA library libfasgd.so in-tree (nvcc, sm_103a only).

Each translation unit is compiled in parallel, then linked into one shared
library that exports only the C ABI of include/fasgd.h (the CUDA runtime is
linked statically and kept private).  A rebuild happens only when a source
or header is newer than the library.
"""

from __future__ import annotations

import concurrent.futures
import glob
import os
import shutil
import subprocess
import sysconfig

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
INCLUDE = os.path.join(ROOT, "include")
BUILD = os.path.join(PKG, "_build")
LIB = os.path.join(PKG, "libfasgd.so")

ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
NVCC_FLAGS = ["-O3", "-std=c++17", "-lineinfo", "-Xcompiler", "-fPIC,-fvisibility=hidden",
              "-Xptxas", "-warn-spills", f"-I{INCLUDE}", f"-I{CSRC}"]


def nvcc() -> str:
    exe = shutil.which("nvcc")
    if exe is None:
        cand = "/usr/local/cuda/bin/nvcc"
        if os.path.exists(cand):
            return cand
        raise RuntimeError("nvcc not found: cannot build the CUDA library")
    return exe


def sources() -> list:
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _inputs() -> list:
    return (sources() + glob.glob(os.path.join(CSRC, "*.cuh"))
            + glob.glob(os.path.join(INCLUDE, "*.h")) + [os.path.abspath(__file__)])


def up_to_date() -> bool:
    if not os.path.exists(LIB):
        return False
    t = os.path.getmtime(LIB)
    return all(os.path.getmtime(p) <= t for p in _inputs())


def build(force: bool = False, verbose: bool = False, extra_flags: list | None = None) -> str:
    """Build libfasgd.so (and the binding's module) if needed; returns its path."""
    if not force and up_to_date():
        build_binding()
        return LIB
    os.makedirs(BUILD, exist_ok=True)
    exe = nvcc()
    flags = NVCC_FLAGS + (extra_flags or [])

    def compile_one(src):
        obj = os.path.join(BUILD, os.path.basename(src) + ".o")
        cmd = [exe, *ARCH, *flags, "-c", src, "-o", obj]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError(f"nvcc failed on {src}:\n{r.stdout}\n{r.stderr}")
        if verbose and (r.stdout or r.stderr):
            print(r.stdout + r.stderr)
        return obj

    with concurrent.futures.ThreadPoolExecutor(max_workers=max(1, len(sources()))) as ex:
        objs = list(ex.map(compile_one, sources()))
    vscript = os.path.join(BUILD, "exports.map")
    with open(vscript, "w") as f:
        f.write("{ global: fasgd_*; bfasgd_*; local: *; };\n")
    tmp = LIB + f".tmp{os.getpid()}"
    cmd = [exe, *ARCH, "-shared", "-o", tmp, *objs, "-Xlinker", f"--version-script={vscript}"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"link failed:\n{r.stdout}\n{r.stderr}")
    os.replace(tmp, LIB)
    build_binding(force)
    return LIB


BINDING_SRC = os.path.join(PKG, "binding.c")
# The name carries the interpreter's ABI and machine, so that every Python loads
# only a module that was built for it.
BINDING = os.path.join(PKG, "_binding" + sysconfig.get_config_var("EXT_SUFFIX"))
_UNTAGGED = os.path.join(PKG, "_binding.so")   # what earlier versions built: any Python would load it


def build_binding(force: bool = False) -> str | None:
    """Build the CPython module of the binding's hot calls (binding.c) against
    libfasgd.so; returns its path, or None where Python's headers are not
    installed (the binding then makes every call through ctypes)."""
    if BINDING != _UNTAGGED and os.path.exists(_UNTAGGED):
        os.remove(_UNTAGGED)
    include = sysconfig.get_paths()["include"]
    if not os.path.exists(os.path.join(include, "Python.h")):
        return None
    newest = max(os.path.getmtime(p) for p in (BINDING_SRC, os.path.join(INCLUDE, "fasgd.h")))
    if not force and os.path.exists(BINDING) and os.path.getmtime(BINDING) >= newest:
        return BINDING
    tmp = BINDING + f".tmp{os.getpid()}"
    cmd = ["gcc", "-O2", "-std=c11", "-Wall", "-Wextra", "-shared", "-fPIC", "-fvisibility=hidden",
           BINDING_SRC, f"-I{include}", f"-I{INCLUDE}", f"-L{PKG}", "-lfasgd", "-Wl,-rpath,$ORIGIN",
           "-o", tmp]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"binding build failed:\n{r.stdout}\n{r.stderr}")
    os.replace(tmp, BINDING)
    return BINDING


DRIVER_SRC = os.path.join(PKG, "abi_latency.c")
DRIVER = os.path.join(BUILD, "abi_latency")


def build_latency_driver(force: bool = False) -> str:
    """Build the C timing driver of the ABI (abi_latency.c) against
    libfasgd.so and the CUDA runtime; returns the executable's path."""
    lib = build()
    if (not force and os.path.exists(DRIVER)
            and os.path.getmtime(DRIVER) >= max(os.path.getmtime(DRIVER_SRC),
                                                os.path.getmtime(lib))):
        return DRIVER
    os.makedirs(BUILD, exist_ok=True)
    cuda = os.path.dirname(os.path.dirname(nvcc()))
    tmp = DRIVER + f".tmp{os.getpid()}"
    cmd = ["gcc", "-O2", "-std=c11", "-Wall", "-Wextra", DRIVER_SRC, f"-I{INCLUDE}",
           f"-I{os.path.join(cuda, 'include')}", f"-L{PKG}", "-lfasgd",
           f"-L{os.path.join(cuda, 'lib64')}", "-lcudart", f"-Wl,-rpath,{PKG}",
           f"-Wl,-rpath,{os.path.join(cuda, 'lib64')}", "-o", tmp]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"abi_latency build failed:\n{r.stdout}\n{r.stderr}")
    os.replace(tmp, DRIVER)
    return DRIVER


if __name__ == "__main__":
    import sys
    print(build(force="--force" in sys.argv, verbose=True,
                extra_flags=["-Xptxas", "-v"] if "-v" in sys.argv else None))
