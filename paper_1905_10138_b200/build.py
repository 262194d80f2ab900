"""Builds ``libsqnn.so`` (C-ABI library: host encoder + sm_100a kernels) in-tree with nvcc, and
``_sqnn_python.so`` (marshalling of torch tensors for its device entry points) with the host compiler."""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig
from concurrent.futures import ThreadPoolExecutor

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
INCLUDE = os.path.join(os.path.dirname(HERE), "include")
LIB = os.path.join(HERE, "libsqnn.so")
PY_MODULE = os.path.join(HERE, "_sqnn_python.so")
PY_SOURCE = "sqnn_python.cpp"
SOURCES = ["sqnn_host.cpp", "sqnn_api.cu", "sqnn_mma.cu", "sqnn_search.cu"]
SHAPE_SOURCE = "sqnn_shape.cu"
# (n_out, n_in) with compile-time kernels -- the list in csrc/sqnn_shapes.h -- plus the run-time shape (0, 0)
SHAPES = [(40, 12), (40, 16), (60, 12), (80, 8), (80, 16), (100, 10), (200, 10), (0, 0)]
HEADERS = ["sqnn_blob.h", "sqnn_layout.h", "sqnn_decode.cuh", "sqnn_launch.h", "sqnn_kernels.cuh", "sqnn_gemv.cuh", "sqnn_gemv_tc.cuh", "sqnn_gemv_plan.h", "sqnn_tc.cuh", "sqnn_shapes.h", SHAPE_SOURCE]


def _nvcc() -> str:
    for cand in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", "nvcc"):
        if cand and (os.path.sep not in cand or os.path.exists(cand)):
            return cand
    return "nvcc"


def _stale(target: str, sources) -> bool:
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    deps = [os.path.join(CSRC, s) for s in sources] + [os.path.join(INCLUDE, "sqnn.h")]
    return any(os.path.getmtime(d) > t for d in deps)


def _build_python_module(force: bool) -> None:
    """The module uses torch's C++ tensor type, so it is compiled against the headers of the installed torch."""
    if not force and not _stale(PY_MODULE, [PY_SOURCE]):
        return
    from torch.utils import cpp_extension
    import torch
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(_nvcc()))), "include")
    cmd = [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-shared", "-fPIC",
           f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
           "-I", INCLUDE, "-I", sysconfig.get_paths()["include"], "-I", cuda]
    for d in cpp_extension.include_paths():
        cmd += ["-isystem", d]
    for d in cpp_extension.library_paths():
        cmd += ["-L", d]
    cmd += [os.path.join(CSRC, PY_SOURCE), "-o", PY_MODULE, "-lc10", "-lc10_cuda", "-ltorch_cpu", "-ltorch_python"]
    subprocess.run(cmd, check=True)


def build(force: bool = False, verbose: bool = False) -> str:
    _build_python_module(force)
    if not force and not _stale(LIB, SOURCES + HEADERS):
        return LIB
    objdir = os.path.join(HERE, "_build")
    os.makedirs(objdir, exist_ok=True)
    common = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "-I", INCLUDE, "-I", CSRC, "-Xcompiler", "-fPIC,-fopenmp,-O3"]
    if verbose:
        common += ["-Xptxas", "-v"]
    jobs = []
    for no, ni in reversed(SHAPES):               # the longest first
        for part in (2, 1, 0):
            jobs.append(([f"-DSQNN_NO={no}", f"-DSQNN_NI={ni}", f"-DSQNN_PART={part}", os.path.join(CSRC, SHAPE_SOURCE)],
                         os.path.join(objdir, f"sqnn_shape_{no}x{ni}_{part}.o")))
    for s in SOURCES:
        jobs.append(([os.path.join(CSRC, s)], os.path.join(objdir, os.path.splitext(s)[0] + ".o")))
    objs = [o for _, o in jobs]
    with ThreadPoolExecutor(max(1, min(len(jobs), os.cpu_count() or 4))) as pool:
        for _ in pool.map(lambda j: subprocess.run([_nvcc(), *common, "-c", *j[0], "-o", j[1]], check=True), jobs):
            pass
    subprocess.run([_nvcc(), "-shared", "-o", LIB, *objs, "-Xcompiler", "-fopenmp", "-lgomp"], check=True)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
