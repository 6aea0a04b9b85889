"""Build ``libtk.so`` (the CUDA library behind include/tk.h) in-tree for sm_103a.

Each ``csrc/*.cu`` is compiled by nvcc in parallel, then linked into
``paper_2603_04427_gb300/libtk.so``; ``csrc/py_binding.cpp`` (the binding's
native argument checks) is compiled by g++ beside them into ``_tkpy.so``.  Either
is skipped when it is newer than its sources and headers and, for ``_tkpy.so``, was
built for this Python and torch.  Run ``python -m paper_2603_04427_gb300.build`` (or
``__graft_entry__.build()``).
"""

from __future__ import annotations

import concurrent.futures as cf
import glob
import os
import platform
import shutil
import subprocess
import sys
import sysconfig

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
INCLUDE = os.path.join(ROOT, "include")
BUILD = os.path.join(PKG, "_build")
LIB = os.path.join(PKG, "libtk.so")
PY_SRC = os.path.join(CSRC, "py_binding.cpp")
PY_LIB = os.path.join(PKG, "_tkpy.so")
PY_TAG = os.path.join(BUILD, "_tkpy.tag")   # what _tkpy.so was built for

ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
NVCC_FLAGS = ["-std=c++17", "-O3", "-lineinfo", "-Xcompiler", "-fPIC", "-Xcompiler", "-O2",
              "--expt-relaxed-constexpr", "-I", INCLUDE, "-I", CSRC]


def nvcc() -> str:
    for cand in (os.environ.get("NVCC"), shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found (set NVCC or put the CUDA toolkit on PATH)")


def _sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _deps():
    return _sources() + glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(
        os.path.join(CSRC, "*.h")) + _headers()


def _headers():
    return glob.glob(os.path.join(INCLUDE, "*.h"))


def _newer(lib: str, deps) -> bool:
    if not os.path.exists(lib):
        return False
    t = os.path.getmtime(lib)
    return all(os.path.getmtime(f) <= t for f in [*deps, __file__])


def lib_up_to_date() -> bool:
    return _newer(LIB, _deps())


def py_tag() -> str:
    """What _tkpy.so depends on beside its sources: CPython's and torch's C++ interfaces."""
    import torch
    return (f"{sys.implementation.cache_tag} {platform.machine()} torch {torch.__version__} "
            f"cxx11_abi {int(torch.compiled_with_cxx11_abi())}")


def py_matches() -> bool:
    """_tkpy.so exists and was built for this Python and torch."""
    if not os.path.exists(PY_LIB) or not os.path.exists(PY_TAG):
        return False
    with open(PY_TAG) as f:
        return f.read() == py_tag()


def py_up_to_date() -> bool:
    return _newer(PY_LIB, [PY_SRC] + _headers()) and py_matches()


def up_to_date() -> bool:
    return lib_up_to_date() and py_up_to_date()


def _compile(src: str, extra) -> str:
    obj = os.path.join(BUILD, os.path.basename(src)[:-3] + ".o")
    cmd = [nvcc()] + ARCH + NVCC_FLAGS + list(extra) + ["-c", src, "-o", obj]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"nvcc failed for {src}:\n{' '.join(cmd)}\n{r.stdout}\n{r.stderr}")
    if r.stderr.strip() and "-Xptxas" in " ".join(extra):
        sys.stderr.write(r.stderr)
    return obj


def _build_py() -> None:
    """_tkpy.so: a CPython module over torch's C++ tensors (paths of the installed torch)."""
    import torch
    root = os.path.dirname(os.path.abspath(torch.__file__))
    cuda = os.path.dirname(os.path.dirname(os.path.abspath(nvcc())))
    inc = [sysconfig.get_paths()["include"], os.path.join(root, "include"),
           os.path.join(root, "include", "torch", "csrc", "api", "include"),
           os.path.join(cuda, "include"), INCLUDE]
    tmp = PY_LIB + ".tmp"
    cmd = (["g++", "-std=c++17", "-O2", "-fPIC", "-shared", "-fvisibility=hidden",
            f"-D_GLIBCXX_USE_CXX11_ABI={int(torch.compiled_with_cxx11_abi())}"]
           + [x for d in inc for x in ("-isystem", d)] + [PY_SRC, "-o", tmp, "-L", os.path.join(root, "lib"),
              "-ltorch_python", "-ltorch_cpu", "-lc10_cuda", "-lc10"])
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"g++ failed for {PY_SRC}:\n{' '.join(cmd)}\n{r.stdout}\n{r.stderr}")
    if os.path.exists(PY_TAG):   # no tag beside another module, whatever happens next
        os.remove(PY_TAG)
    os.replace(tmp, PY_LIB)
    with open(PY_TAG + ".tmp", "w") as f:
        f.write(py_tag())
    os.replace(PY_TAG + ".tmp", PY_TAG)


def build(force: bool = False, verbose_ptxas: bool = False) -> str:
    """Compile and link libtk.so and _tkpy.so where they are not up to date; returns libtk.so's path."""
    want_lib, want_py = force or not lib_up_to_date(), force or not py_up_to_date()
    if not want_lib and not want_py:
        return LIB
    os.makedirs(BUILD, exist_ok=True)
    extra = ["-Xptxas", "-v"] if verbose_ptxas else []
    srcs = _sources() if want_lib else []
    with cf.ThreadPoolExecutor(max_workers=max(1, min(len(srcs) + 1, os.cpu_count() or 1))) as ex:
        py = ex.submit(_build_py) if want_py else None
        objs = list(ex.map(lambda s: _compile(s, extra), srcs))
    if want_lib:
        tmp = LIB + ".tmp"
        cmd = [nvcc()] + ARCH + ["-shared", "-o", tmp] + objs
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError(f"link failed:\n{' '.join(cmd)}\n{r.stdout}\n{r.stderr}")
        os.replace(tmp, LIB)
    if py is not None:
        py.result()   # libtk.so, which needs no torch, stands whatever became of _tkpy.so
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose_ptxas="--ptxas-v" in sys.argv))
