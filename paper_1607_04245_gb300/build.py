"""Build libfem (the CUDA C-ABI library) in-tree for sm_103a, and the binding's native
marshalling module.

Each .cu translation unit is compiled in parallel with nvcc, then linked into
``paper_1607_04245_gb300/libfem.so``. No cmake, no torch extension machinery: the
library is a plain shared object with the C ABI of ``include/fem.h``. Beside it,
``fem_marshal.cpp`` is compiled with g++ against the installed torch into the extension
module ``paper_1607_04245_gb300/_marshal`` (host code; it links no libfem).

    python -m paper_1607_04245_gb300.build [--verbose-ptxas]
"""

from __future__ import annotations

import concurrent.futures as cf
import os
import shutil
import subprocess
import sys
import sysconfig

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
OUT = os.path.join(PKG, "libfem.so")
BUILD = os.path.join(PKG, "_build")

ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
SOURCES = ["fem_core.cu", "fem_laplacian.cu", "fem_elasticity.cu", "fem_mesh.cu", "fem_geometry.cu", "fem_reaction.cu",
           "fem_solver.cu", "fem_transpose.cu", "fem_host.cu", "fem_df.cu",
           "fem_arena.cpp", "fem_noalloc.cu", "fem_serve.cu", "fem_pointwise.cu"]


def nvcc() -> str:
    for c in (shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if c and os.path.exists(c):
            return c
    raise RuntimeError("nvcc not found")


def _deps_mtime() -> float:
    files = [os.path.join(CSRC, f) for f in os.listdir(CSRC)] + [os.path.join(ROOT, "include", "fem.h")]
    return max(os.path.getmtime(f) for f in files)


MARSHAL = os.path.join(PKG, "_marshal" + sysconfig.get_config_var("EXT_SUFFIX"))


def marshal_stamp() -> str:
    """What the marshalling module is compiled against (its inlined accessors read torch's own
    structures): recorded in the module, compared before it is kept or used."""
    import torch

    return (f"torch {torch.__version__} abi {int(torch._C._GLIBCXX_USE_CXX11_ABI)} "
            f"python {sysconfig.get_config_var('EXT_SUFFIX')}")


def _marshal_is_current() -> bool:
    if not os.path.exists(MARSHAL) or os.path.getmtime(MARSHAL) < _deps_mtime():
        return False
    with open(MARSHAL, "rb") as f:
        return marshal_stamp().encode() + b"\0" in f.read()


def _build_marshal() -> None:
    """fem_marshal.cpp against this interpreter and the installed torch."""
    import torch

    t = os.path.dirname(torch.__file__)
    cuda = os.path.dirname(os.path.dirname(os.path.realpath(nvcc())))
    cuda_inc = [d for d in (os.path.join(cuda, "include"), "/usr/local/cuda/include") if os.path.isdir(d)]
    tmp = MARSHAL + ".tmp"
    cmd = ["g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-fvisibility=hidden", "-w",
           f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
           f'-DFEM_MARSHAL_BUILT_FOR="{marshal_stamp()}"', "-I", sysconfig.get_path("include"),
           "-I", os.path.join(t, "include"), "-I", os.path.join(t, "include", "torch", "csrc", "api", "include")]
    cmd += [x for d in cuda_inc for x in ("-I", d)]
    cmd += [os.path.join(CSRC, "fem_marshal.cpp"), "-o", tmp, "-L", os.path.join(t, "lib"), "-ltorch_python",
            "-ltorch_cpu", "-ltorch", "-lc10_cuda", "-lc10"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"g++ failed on fem_marshal.cpp:\n{r.stderr}")
    os.replace(tmp, MARSHAL)


def build(force: bool = False, verbose_ptxas: bool = False) -> str:
    if not force and not verbose_ptxas and os.path.exists(OUT) and os.path.getmtime(OUT) >= _deps_mtime():
        if not _marshal_is_current():
            _build_marshal()
        return OUT
    os.makedirs(BUILD, exist_ok=True)
    cc = nvcc()
    flags = ARCH + ["-O3", "-lineinfo", "-std=c++17", "-Xcompiler", "-fPIC", "-I", os.path.join(ROOT, "include")]
    if verbose_ptxas:
        flags += ["-Xptxas", "-v"]

    def compile_one(src):
        obj = os.path.join(BUILD, os.path.splitext(src)[0] + ".o")
        cmd = [cc] + flags + ["-c", os.path.join(CSRC, src), "-o", obj]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError(f"nvcc failed on {src}:\n{r.stderr}")
        return obj, r.stderr

    with cf.ThreadPoolExecutor(max_workers=len(SOURCES) + 1) as ex:
        marshal = ex.submit(_build_marshal)
        results = list(ex.map(compile_one, SOURCES))
    if verbose_ptxas:
        for _, log in results:
            sys.stderr.write(log)
    tmp = OUT + ".tmp"
    cmd = [cc] + ARCH + ["-shared", "-o", tmp] + [o for o, _ in results] + ["-lcudart", "-ldl"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"link failed:\n{r.stderr}")
    os.replace(tmp, OUT)
    marshal.result()  # a failure is raised with the library in place, which works without the module
    return OUT


if __name__ == "__main__":
    print(build(force=True, verbose_ptxas="--verbose-ptxas" in sys.argv))
