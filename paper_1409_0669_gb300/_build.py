"""In-tree build of the CUDA library ``liblak_gb300.so`` for sm_103a and of the
Python extension ``_fast`` that calls it.

Each translation unit under ``csrc/`` is compiled by nvcc in parallel into
``_build/`` and linked (static CUDA runtime) into a shared library beside this
file; the extension (``csrc/py_fast.cpp``) is compiled by g++ against the
installed torch's headers and linked against that library.  A rebuild happens
only when a source or header is newer than the results, or the installed torch is
another one than the extension was compiled for, unless ``force`` is set.  An
extension that cannot be compiled is left out with a warning: the package works
without it, through ctypes.
"""
from __future__ import annotations

import concurrent.futures
import importlib.util
import os
import re
import shutil
import subprocess
import sysconfig
import tempfile
import warnings

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
INCLUDE = os.path.join(ROOT, "include")
OBJDIR = os.path.join(PKG, "_build")
LIB = os.path.join(PKG, "liblak_gb300.so")
FAST = os.path.join(PKG, "_fast" + sysconfig.get_config_var("EXT_SUFFIX"))
FAST_STAMP = os.path.join(OBJDIR, "py_fast.torch")    # torch it was last compiled (or tried) for
ARCH = "-gencode=arch=compute_103a,code=sm_103a"
SOURCES = ["lak_api.cu", "k_vec.cu", "k_gemv.cu", "k_gemv_wide.cu", "k_spmv.cu", "k_dot_noalloc.cu", "k_batch.cu", "k_grad.cu", "k_transpose.cu", "k_vec_ext.cu", "k_sell.cu", "k_csr_bin.cu", "k_probe.cu"]


def nvcc_path() -> str:
    for cand in (os.environ.get("CUDA_HOME"), os.environ.get("CUDA_PATH"), "/usr/local/cuda"):
        if cand and os.path.exists(os.path.join(cand, "bin", "nvcc")):
            return os.path.join(cand, "bin", "nvcc")
    found = shutil.which("nvcc")
    if not found:
        raise RuntimeError("nvcc not found (set CUDA_HOME)")
    return found


def _deps():
    files = [os.path.join(CSRC, f) for f in os.listdir(CSRC)]
    files.append(os.path.join(INCLUDE, "lak.h"))
    files.append(os.path.abspath(__file__))
    return files


def up_to_date() -> bool:
    if not os.path.exists(LIB) or not os.path.exists(FAST_STAMP):
        return False
    with open(FAST_STAMP) as fh:
        version, _, failed = fh.read().partition(" ")
    if version != torch_version() or (not failed and not os.path.exists(FAST)):
        return False
    t = min(os.path.getmtime(f) for f in ([LIB, FAST_STAMP] if failed else [LIB, FAST_STAMP, FAST]))
    return all(os.path.getmtime(f) <= t for f in _deps())


def compile_flags():
    return [ARCH, "-lineinfo", "-O3", "-std=c++17", "-Xcompiler", "-fPIC",
            "-Xcompiler", "-fvisibility=hidden", "-I", INCLUDE, "-I", CSRC]


def torch_dir() -> str:
    spec = importlib.util.find_spec("torch")
    if spec is None or not spec.submodule_search_locations:
        raise RuntimeError("torch not found")
    return list(spec.submodule_search_locations)[0]


def torch_version() -> str:
    """The installed torch's version, read without importing it."""
    with open(os.path.join(torch_dir(), "version.py")) as fh:
        found = re.search(r"""^__version__\s*=\s*['"]([^'"]+)""", fh.read(), re.M)
    if not found:
        raise RuntimeError("torch/version.py names no version")
    return found.group(1)


def compile_fast() -> str:
    """Object file of the Python extension."""
    inc = os.path.join(torch_dir(), "include")
    cuda = os.path.join(os.path.dirname(os.path.dirname(nvcc_path())), "include")
    obj = os.path.join(OBJDIR, "py_fast.o")
    cmd = ["g++", "-O2", "-std=c++17", "-fPIC", "-fvisibility=hidden",
           f'-DLAK_TORCH_VERSION="{torch_version()}"', "-I", INCLUDE, "-I", inc,
           "-I", os.path.join(inc, "torch", "csrc", "api", "include"), "-I", cuda, "-I",
           sysconfig.get_paths()["include"], "-c", os.path.join(CSRC, "py_fast.cpp"), "-o", obj]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"g++ failed on py_fast.cpp:\n{r.stderr}")
    return obj


def link_fast(obj: str):
    lib = os.path.join(torch_dir(), "lib")
    fd, tmp = tempfile.mkstemp(suffix=".so", dir=PKG)
    os.close(fd)
    cmd = ["g++", "-shared", "-o", tmp, obj, "-L", lib, "-lc10", "-lc10_cuda", "-ltorch_cpu",
           "-ltorch_python", "-L", PKG, "-l:" + os.path.basename(LIB), "-Wl,-rpath,$ORIGIN"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        os.unlink(tmp)
        raise RuntimeError(f"link of the Python extension failed:\n{r.stderr}")
    os.replace(tmp, FAST)


def build(force: bool = False, verbose: bool = False, ptxas_verbose: bool = False) -> str:
    if not force and up_to_date():
        return LIB
    nvcc = nvcc_path()
    os.makedirs(OBJDIR, exist_ok=True)
    flags = compile_flags() + (["-Xptxas", "-v"] if ptxas_verbose else [])

    def one(src):
        obj = os.path.join(OBJDIR, os.path.splitext(src)[0] + ".o")
        cmd = [nvcc, *flags, "-c", os.path.join(CSRC, src), "-o", obj]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError(f"nvcc failed on {src}:\n{r.stderr}")
        return obj, r.stderr

    with concurrent.futures.ThreadPoolExecutor(max_workers=len(SOURCES) + 1) as ex:
        fast = ex.submit(compile_fast)
        results = list(ex.map(one, SOURCES))
    if verbose or ptxas_verbose:
        for _, log in results:
            if log:
                print(log)
    fd, tmp = tempfile.mkstemp(suffix=".so", dir=PKG)
    os.close(fd)
    cmd = [nvcc, ARCH, "-shared", "-o", tmp, *[o for o, _ in results]]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        os.unlink(tmp)
        raise RuntimeError(f"link failed:\n{r.stderr}")
    os.replace(tmp, LIB)
    stamp = torch_version()
    try:
        link_fast(fast.result())
    except Exception as e:              # g++, torch's headers or its libraries
        warnings.warn(f"built without the Python extension: {e}")
        stamp += " failed"
        if os.path.exists(FAST):        # of other sources or another torch
            os.unlink(FAST)
    with open(FAST_STAMP, "w") as fh:
        fh.write(stamp)
    return LIB


if __name__ == "__main__":
    import sys
    print(build(force="--force" in sys.argv, verbose=True, ptxas_verbose="-v" in sys.argv))
