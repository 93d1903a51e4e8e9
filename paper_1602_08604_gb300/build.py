"""Build liblre.so (the C-ABI library) in-tree with nvcc for sm_103a.

Each translation unit is compiled in parallel, then linked with cuSOLVER and
cuBLAS.  The result lands next to this file; nothing is installed.
"""
import os
import shutil
import subprocess
from concurrent.futures import ThreadPoolExecutor

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
OBJ = os.path.join(HERE, "_build")
LIB = os.path.join(HERE, "liblre.so")
SOURCES = ["abi.cu", "fold.cu", "assemble.cu", "assemble_top.cu", "estimate_small.cu", "project.cu", "project_small.cu", "host.cu", "noalloc.cu", "batch.cu", "fold_mma.cu", "fold_tma.cu", "tridiag.cu", "records.cu", "krylov.cu", "krylov_steps.cu", "krylov_vecs.cu", "slab.cu", "ic4.cu", "stream.cu"]
HEADERS = [os.path.join(CSRC, "lre_internal.cuh"), os.path.join(CSRC, "sm103.cuh"),
           os.path.join(CSRC, "passes.cuh"), os.path.join(CSRC, "dfloat.cuh"), os.path.join(CSRC, "krylov.cuh"),
           os.path.join(CSRC, "tri_minor.cuh"),
           os.path.join(ROOT, "include", "lre.h")]
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]


def cuda_home():
    for c in (os.environ.get("CUDA_HOME"), "/usr/local/cuda"):
        if c and os.path.exists(os.path.join(c, "bin", "nvcc")):
            return c
    nv = shutil.which("nvcc")
    if nv:
        return os.path.dirname(os.path.dirname(nv))
    raise RuntimeError("nvcc not found")


def _stale(target, deps):
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    return any(os.path.getmtime(d) > t for d in deps)


def build(force=False, verbose=False):
    cuda = cuda_home()
    nvcc = os.path.join(cuda, "bin", "nvcc")
    os.makedirs(OBJ, exist_ok=True)
    flags = ["-O3", "-std=c++17", "-lineinfo", "-Xcompiler", "-fPIC", *ARCH,
             "-I", os.path.join(ROOT, "include")]
    if verbose:
        flags += ["-Xptxas", "-v"]

    def compile_one(src):
        s = os.path.join(CSRC, src)
        o = os.path.join(OBJ, src.replace(".cu", ".o"))
        if force or _stale(o, [s] + HEADERS):
            subprocess.check_call([nvcc, *flags, "-c", s, "-o", o])
        return o

    with ThreadPoolExecutor(max_workers=len(SOURCES)) as ex:
        objs = list(ex.map(compile_one, SOURCES))
    if force or _stale(LIB, objs):
        libdir = os.path.join(cuda, "lib64")
        if not os.path.isdir(libdir):
            libdir = os.path.join(cuda, "lib")
        cmd = [nvcc, "-shared", *ARCH, *objs, "-o", LIB + ".tmp", "-L", libdir,
               "-lcusolver", "-lcublas", "-Xlinker", "-rpath=" + libdir]
        subprocess.check_call(cmd)
        os.replace(LIB + ".tmp", LIB)
    return LIB


if __name__ == "__main__":
    import sys
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
