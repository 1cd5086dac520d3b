"""Build libspecdiff.so (the C-ABI library) for sm_103a with nvcc.

Sources are compiled in parallel, one nvcc process per translation unit, and
linked into ``paper_2606_13426_gb300/lib/libspecdiff.so``; the CPython module of the
binding's frequent calls goes beside it.  A rebuild happens only
when a source or header is newer than the library (or ``force=True``).
"""
import os
import shutil
import subprocess
import sys
import sysconfig
from concurrent.futures import ThreadPoolExecutor

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
INCLUDE = os.path.join(ROOT, "include")
LIBDIR = os.path.join(PKG, "lib")
LIBNAME = "libspecdiff.so"
SOURCES = ["sdv_verify.cu", "sdv_chain_f32.cu", "sdv_chain_bf16.cu", "sdv_sampler.cu", "sdv_rounds_c8.cu",
           "sdv_rounds_c16.cu", "sdv_noalloc.cu"]
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
NVCC_FLAGS = ["-O3", "-std=c++17", "-lineinfo", "-Xcompiler", "-fPIC", "-I" + INCLUDE,
              "-I" + CSRC]


def lib_path():
    return os.path.join(LIBDIR, LIBNAME)


def pycall_path():
    return os.path.join(LIBDIR, "_sdvcall.so")


def _build_pycall():
    """The CPython module of sdv_pycall.c; left out where Python's headers are missing (the
    binding then calls through ctypes)."""
    inc = sysconfig.get_paths()["include"]
    if not os.path.exists(os.path.join(inc, "Python.h")):
        return
    out = pycall_path()
    cmd = [os.environ.get("CC") or shutil.which("gcc") or "cc", "-O2", "-shared", "-fPIC", "-I" + INCLUDE, "-I" + inc,
           os.path.join(CSRC, "sdv_pycall.c"), "-o", out + ".tmp"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError("compiling sdv_pycall.c failed:\n%s\n%s" % (" ".join(cmd), r.stderr))
    os.replace(out + ".tmp", out)


def _nvcc():
    for cand in (os.environ.get("NVCC"), shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found: the CUDA toolkit is required to build libspecdiff")


def _sources():
    return [os.path.join(CSRC, s) for s in SOURCES if os.path.exists(os.path.join(CSRC, s))]


def _deps():
    deps = _sources() + [os.path.join(CSRC, "sdv_pycall.c")]
    for d in (CSRC, INCLUDE):
        deps += [os.path.join(d, f) for f in os.listdir(d) if f.endswith((".h", ".cuh"))]
    return deps


def up_to_date():
    out = lib_path()
    if not os.path.exists(out):
        return False
    t = os.path.getmtime(out)
    return all(os.path.getmtime(p) <= t for p in _deps())


def build(force=False, verbose=False):
    """Compile every CUDA source for sm_103a and link libspecdiff.so; returns its path."""
    out = lib_path()
    if not force and up_to_date():
        return out
    nvcc = _nvcc()
    os.makedirs(LIBDIR, exist_ok=True)
    objdir = os.path.join(LIBDIR, "obj")
    os.makedirs(objdir, exist_ok=True)

    def compile_one(src):
        obj = os.path.join(objdir, os.path.basename(src).replace(".cu", ".o"))
        cmd = [nvcc] + ARCH + NVCC_FLAGS + ["-c", src, "-o", obj]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError("nvcc failed for %s:\n%s\n%s" % (src, " ".join(cmd), r.stderr))
        if verbose and r.stderr:
            sys.stderr.write(r.stderr)
        return obj

    srcs = _sources()
    with ThreadPoolExecutor(max_workers=max(1, len(srcs))) as ex:
        objs = list(ex.map(compile_one, srcs))
    _build_pycall()
    tmp = out + ".tmp"
    cmd = [nvcc] + ARCH + ["-shared", "-o", tmp] + objs
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError("link failed:\n%s\n%s" % (" ".join(cmd), r.stderr))
    os.replace(tmp, out)
    return out


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose=True))
