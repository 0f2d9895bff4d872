"""Build the in-tree shared library ``libafqmc_gb300.so`` for sm_103a with nvcc.

Each translation unit is compiled in parallel into ``_build/`` and linked with
the static CUDA runtime; nothing is installed outside the package directory.
"""
import concurrent.futures
import hashlib
import os
import shutil
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
BUILD = os.path.join(ROOT, "_build")
LIB = os.path.join(HERE, "libafqmc_gb300.so")
SOURCES = ["gemm_f64.cu", "gemm_f64e.cu", "energy_f64e.cu", "taylor_f64e.cu", "step_small.cu", "walker_kernels.cu", "setup_kernels.cu", "api.cu", "pair.cu", "stats.cpp",
           "noalloc.cu", "gemm_tc.cu", "mixed_kernels.cu", "walker_fast.cu", "autotune.cu",
           "tangent.cu", "adjoint_kernels.cu", "adjoint.cu",
           "energy_tc.cu", "propagate_f32.cu",
           "propagate_tc.cu", "propagate_tcl.cu", "pes.cu", "multidet.cu"]
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
FLAGS = ["-O3", "-lineinfo", "-std=c++17", "-Xcompiler", "-fPIC", "-Xcompiler", "-O2"]


def _nvcc():
    for cand in (os.environ.get("NVCC"), shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found: the CUDA toolkit is required to build libafqmc_gb300.so")


def _fingerprint():
    h = hashlib.sha256()
    h.update(" ".join(ARCH + FLAGS).encode())
    h.update(os.uname().machine.encode())
    for name in sorted(os.listdir(CSRC)) + ["../../include/afqmc.h"]:
        path = os.path.normpath(os.path.join(CSRC, name))
        if os.path.isfile(path):
            with open(path, "rb") as f:
                h.update(name.encode())
                h.update(f.read())
    return h.hexdigest()


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile (if needed) and return the path of the shared library."""
    stamp = LIB + ".stamp"
    fp = _fingerprint()
    if not force and os.path.exists(LIB) and os.path.exists(stamp):
        with open(stamp) as f:
            if f.read().strip() == fp:
                return LIB
    nvcc = _nvcc()
    os.makedirs(BUILD, exist_ok=True)

    def compile_one(src):
        obj = os.path.join(BUILD, src + ".o")
        cmd = [nvcc] + ARCH + FLAGS + ["-c", os.path.join(CSRC, src), "-o", obj]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError(f"nvcc failed on {src}:\n{r.stderr}")
        if verbose and r.stderr:
            print(r.stderr)
        return obj

    with concurrent.futures.ThreadPoolExecutor(max_workers=len(SOURCES)) as ex:
        objs = list(ex.map(compile_one, SOURCES))
    tmp = LIB + ".tmp"
    cmd = [nvcc] + ARCH + ["-shared", "-cudart", "static", "-o", tmp] + objs
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"link failed:\n{r.stderr}")
    os.replace(tmp, LIB)
    with open(stamp, "w") as f:
        f.write(fp)
    return LIB


if __name__ == "__main__":
    print(build(force=True, verbose=True))
