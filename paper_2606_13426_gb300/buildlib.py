"""Build libspecdiff.so (the C-ABI library) for sm_103a with nvcc.

Sources are compiled in parallel, one nvcc process per translation unit, and
linked into ``paper_2606_13426_gb300/lib/libspecdiff.so``; the CPython module of the
binding's frequent calls goes beside it.  Each is rebuilt only when one of its sources or
headers is newer (or ``force=True``).
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
    """The module's file, named for this Python's ABI."""
    return os.path.join(LIBDIR, "_sdvcall" + (sysconfig.get_config_var("EXT_SUFFIX") or ".so"))


def _pycall_source():
    return os.path.join(CSRC, "sdv_pycall.c")


def _python_headers():
    inc = sysconfig.get_paths()["include"]
    return inc if os.path.exists(os.path.join(inc, "Python.h")) else None


def _newer_than(out, deps):
    if not os.path.exists(out):
        return False
    t = os.path.getmtime(out)
    return all(os.path.getmtime(p) <= t for p in deps)


def _build_pycall(force=False):
    """The CPython module of sdv_pycall.c, if it is not up to date; left out where Python's
    headers or a C compiler are missing (the binding then calls through ctypes)."""
    inc, out = _python_headers(), pycall_path()
    cc = os.environ.get("CC") or shutil.which("gcc") or shutil.which("cc")
    if inc is None or cc is None or not force and _newer_than(out, [_pycall_source(), os.path.join(INCLUDE, "specdiff.h")]):
        return
    os.makedirs(LIBDIR, exist_ok=True)
    cmd = [cc, "-O2", "-shared", "-fPIC", "-I" + INCLUDE, "-I" + inc,
           _pycall_source(), "-o", out + ".tmp"]
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
    deps = _sources()
    for d in (CSRC, INCLUDE):
        deps += [os.path.join(d, f) for f in os.listdir(d) if f.endswith((".h", ".cuh"))]
    return deps


def up_to_date():
    return _newer_than(lib_path(), _deps())


def build(force=False, verbose=False):
    """Compile every CUDA source for sm_103a and link libspecdiff.so, and the module of the
    binding's frequent calls; returns the library's path."""
    out = lib_path()
    _build_pycall(force)
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
    tmp = out + ".tmp"
    cmd = [nvcc] + ARCH + ["-shared", "-o", tmp] + objs
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError("link failed:\n%s\n%s" % (" ".join(cmd), r.stderr))
    os.replace(tmp, out)
    return out


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose=True))
