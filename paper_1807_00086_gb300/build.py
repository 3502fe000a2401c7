"""Builds libhdg.so in-tree with nvcc for sm_103a (no cmake, one nvcc call per unit, in parallel)."""
import concurrent.futures
import os
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
OUT = os.path.join(HERE, "libhdg.so")
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
# -split-compile: the device code of a unit is optimised by several threads (api.cu: 230 -> 77 s)
FLAGS = ["-O3", "-lineinfo", "-std=c++17", "-split-compile=0", "-Xcompiler", "-fPIC", "-Xcompiler", "-O2"]
UNITS = ["api.cu", "vardeg.cu", "svk.cu", "bilu.cu", "noalloc.cu", "reftab.cpp", "mesh.cpp"]


def _nvcc():
    for cand in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", "nvcc"):
        if cand and (os.path.sep not in cand or os.path.exists(cand)):
            return cand
    return "nvcc"


def build(verbose=False):
    nvcc = _nvcc()
    objdir = os.path.join(HERE, "_build")
    os.makedirs(objdir, exist_ok=True)

    # a unit is rebuilt when it, a header of the library or this script is newer than its object
    deps = [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith((".h", ".cuh"))]
    deps += [os.path.join(HERE, "..", "include", "hdg.h"), os.path.abspath(__file__)]
    newest_dep = max(os.path.getmtime(d) for d in deps if os.path.exists(d))

    def compile_unit(u):
        obj = os.path.join(objdir, u + ".o")
        src = os.path.join(CSRC, u)
        if os.path.exists(obj) and os.path.getmtime(obj) > max(newest_dep, os.path.getmtime(src)):
            return obj
        cmd = [nvcc] + ARCH + FLAGS + ["-c", src, "-o", obj]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError("nvcc failed for %s:\n%s\n%s" % (u, " ".join(cmd), r.stderr))
        return obj

    with concurrent.futures.ThreadPoolExecutor(len(UNITS)) as ex:
        objs = list(ex.map(compile_unit, UNITS))
    tmp = OUT + ".tmp"
    cmd = [nvcc] + ARCH + ["-shared", "-o", tmp] + objs
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError("link failed:\n%s\n%s" % (" ".join(cmd), r.stderr))
    os.replace(tmp, OUT)
    if verbose:
        print("built", OUT)
    return OUT


if __name__ == "__main__":
    build(verbose=True)
