"""Build libvlb.so (the CUDA library behind include/vlb.h) in-tree for sm_103a.

Each translation unit compiles in parallel with nvcc, then one link step
produces paper_2401_17183_gb300/libvlb.so. No CMake; portable across the
x86-64 build host and the aarch64 GPU host (no -march flags).
"""
import concurrent.futures as cf
import os
import shutil
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
BUILD = os.path.join(HERE, "_build")
LIB = os.path.join(HERE, "libvlb.so")
SOURCES = ["vlb_api.cu", "vlb_geometry.cu", "vlb_step.cu", "vlb_step_f32.cu", "vlb_step_f16.cu", "vlb_step_bf16.cu",
           "vlb_batch.cu",
           "vlb_moments.cu", "vlb_noalloc.cu", "vlb_nn.cu", "vlb_q39.cu",
           "vlb_small.cu"]
HEADERS = ["vlb_chain.cuh", "vlb_internal.cuh", "vlb_collide.cuh", "vlb_addr.cuh", "vlb_step.cuh", "vlb_q39.cuh",
           "vlb_nn_tc.cuh", "vlb_small.cuh"]
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
FLAGS = ["-O3", "-std=c++17", "-lineinfo", "--expt-relaxed-constexpr", "-Xcompiler", "-fPIC",
         "-Xcompiler", "-O2"]


def nvcc():
    exe = shutil.which("nvcc")
    if exe:
        return exe
    cand = "/usr/local/cuda/bin/nvcc"
    if os.path.exists(cand):
        return cand
    raise RuntimeError("nvcc not found: the CUDA toolkit is required to build libvlb")


def _stale(target, deps):
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    return any(os.path.getmtime(d) > t for d in deps)


def _inc_deps():
    return [os.path.join(CSRC, h) for h in HEADERS] + [
        os.path.join(HERE, "..", "include", "vlb.h"), os.path.join(HERE, "..", "include", "vlb_nn.h"),
        os.path.abspath(__file__)]


def _compile(src, verbose):
    obj = os.path.join(BUILD, src.replace(".cu", ".o"))
    deps = [os.path.join(CSRC, src)] + _inc_deps()
    if not _stale(obj, deps):
        return obj, ""
    cmd = [nvcc()] + ARCH + FLAGS + (["-Xptxas", "-v"] if verbose else []) + [
        "-c", os.path.join(CSRC, src), "-o", obj]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError("nvcc failed for %s:\n%s\n%s" % (src, r.stdout, r.stderr))
    return obj, r.stderr


def build(force=False, verbose=False):
    """Compile every translation unit and link libvlb.so; returns its path."""
    os.makedirs(BUILD, exist_ok=True)
    if force:
        for f in os.listdir(BUILD):
            os.remove(os.path.join(BUILD, f))
    with cf.ThreadPoolExecutor(max_workers=len(SOURCES)) as ex:
        results = list(ex.map(lambda s: _compile(s, verbose), SOURCES))
    objs = [o for o, _ in results]
    if verbose:
        for _, log in results:
            if log:
                sys.stderr.write(log)
    if force or _stale(LIB, objs):
        tmp = LIB + ".tmp%d" % os.getpid()
        cmd = [nvcc()] + ARCH + ["-shared", "-o", tmp] + objs + ["-lcudart"]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError("link failed:\n%s\n%s" % (r.stdout, r.stderr))
        os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
