"""Compile the CUDA sources under csrc/ into paper_2509_10798_b200/libjq.so for sm_100a (in-tree).

build(debug=True) compiles the same sources with -DJQ_DEBUG into libjq_debug.so: the bounds-checked build
(csrc/jq_debug.cuh), in which every index the kernels compute is compared with the extent of what it indexes."""
import glob
import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libjq.so")
LIB_DEBUG = os.path.join(HERE, "libjq_debug.so")
LIB_CALL = os.path.join(HERE, "_jqcall.so")   # the binding's C marshalling (csrc/jq_pycall.c)
OBJDIR = os.path.join(HERE, "_build")

NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "-Xcompiler", "-fPIC", "-I", os.path.join(ROOT, "include"), "-I", CSRC]


def _nvcc():
    for cand in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", "nvcc"):
        if cand and (os.path.sep not in cand or os.path.exists(cand)):
            return cand
    return "nvcc"


def _deps():
    return glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(ROOT, "include", "*.h"))


def _build_call(force: bool):
    src = os.path.join(CSRC, "jq_pycall.c")
    if not force and os.path.exists(LIB_CALL) and os.path.getmtime(LIB_CALL) >= max(os.path.getmtime(p) for p in [src] + _deps()):
        return
    tmp = LIB_CALL + ".tmp%d" % os.getpid()
    subprocess.run([os.environ.get("CC", "gcc"), "-O2", "-std=c11", "-Wall", "-shared", "-fPIC", "-I", sysconfig.get_paths()["include"],
                    "-I", os.path.join(ROOT, "include"), src, "-o", tmp], check=True)
    os.replace(tmp, LIB_CALL)


def build(force: bool = False, verbose: bool = False, debug: bool = False) -> str:
    _build_call(force)
    srcs = sorted(glob.glob(os.path.join(CSRC, "*.cu")))
    objdir = OBJDIR + ("_debug" if debug else "")
    lib = LIB_DEBUG if debug else LIB
    flags = NVCC_FLAGS + (["-DJQ_DEBUG"] if debug else [])
    os.makedirs(objdir, exist_ok=True)
    dep_mtime = max(os.path.getmtime(p) for p in _deps())
    objs, rebuilt = [], False
    procs = []
    for src in srcs:
        obj = os.path.join(objdir, os.path.basename(src)[:-3] + ".o")
        objs.append(obj)
        if force or not os.path.exists(obj) or os.path.getmtime(obj) < max(os.path.getmtime(src), dep_mtime):
            cmd = [_nvcc()] + flags + (["-Xptxas", "-v"] if verbose else []) + ["-c", src, "-o", obj]
            procs.append((src, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)))
            rebuilt = True
    for src, p in procs:
        out, _ = p.communicate()
        if verbose or p.returncode:
            sys.stderr.write(out)
        if p.returncode:
            raise RuntimeError("nvcc failed on %s" % src)
    if rebuilt or not os.path.exists(lib):
        tmp = lib + ".tmp%d" % os.getpid()
        cmd = [_nvcc(), "-shared", "-o", tmp] + objs + ["-gencode", "arch=compute_100a,code=sm_100a"]
        subprocess.run(cmd, check=True)
        os.replace(tmp, lib)
    return lib


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv, debug="--debug" in sys.argv))
