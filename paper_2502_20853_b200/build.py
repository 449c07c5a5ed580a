"""Compile the CUDA sources into the in-tree shared library libmxfp4.so (sm_100a only) and the binding's host module _host."""
import importlib
import os
import subprocess
import sys
import sysconfig
from concurrent.futures import ThreadPoolExecutor

_HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(_HERE, "csrc")
LIB = os.path.join(_HERE, "libmxfp4.so")
SOURCES = ["quantize.cu", "gemm.cu", "linear.cu", "gemm_static.cu", "qramp.cu", "diag.cu"]
NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "-Xcompiler", "-fPIC", "--expt-relaxed-constexpr"]


HOST = os.path.join(_HERE, "_host" + sysconfig.get_config_var("EXT_SUFFIX"))   # for this interpreter alone
HOST_SOURCE = os.path.join(CSRC, "host.cpp")


def build_host(force: bool = False) -> str:
    """Build the host module if missing or stale and load the binding again if it was loaded without it; return its path."""
    path = _build_host(force)
    binding, package = (sys.modules.get(__package__ + s) for s in (".binding", "")) if __package__ else (None, None)
    if binding is not None and isinstance(binding._host, binding._NotBuilt):
        importlib.invalidate_caches()
        importlib.reload(binding)
        importlib.reload(package)
    return path


def _build_host(force):
    header = os.path.join(os.path.dirname(_HERE), "include", "mxfp4.h")
    if not force and os.path.exists(HOST) and os.path.getmtime(HOST) >= max(os.path.getmtime(HOST_SOURCE), os.path.getmtime(header)):
        return HOST
    tmp = HOST + ".tmp.%d" % os.getpid()
    r = subprocess.run([os.environ.get("CXX", "g++"), "-std=c++17", "-O2", "-fPIC", "-shared", "-I", sysconfig.get_paths()["include"],
                        "-o", tmp, HOST_SOURCE], capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError("the host module does not build:\n%s\n%s" % (r.stdout, r.stderr))
    os.replace(tmp, HOST)
    return HOST


def _newest_source_mtime():
    paths = [os.path.join(CSRC, f) for f in os.listdir(CSRC)]
    paths.append(os.path.join(os.path.dirname(_HERE), "include", "mxfp4.h"))
    return max(os.path.getmtime(p) for p in paths)


def build(force: bool = False, verbose: bool = False, extra_flags=()) -> str:
    """Build libmxfp4.so and _host if missing or stale; return the former's path.  nvcc cross-compiles without a GPU."""
    build_host(force)
    if not force and os.path.exists(LIB) and os.path.getmtime(LIB) >= _newest_source_mtime():
        return LIB
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    objdir = os.path.join(_HERE, "_build")
    os.makedirs(objdir, exist_ok=True)
    flags = NVCC_FLAGS + list(extra_flags) + (["-Xptxas", "-v"] if verbose else [])

    def compile_one(src):
        obj = os.path.join(objdir, src.replace(".cu", ".o"))
        r = subprocess.run([nvcc] + flags + ["-c", os.path.join(CSRC, src), "-o", obj],
                           capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError("nvcc failed for %s:\n%s\n%s" % (src, r.stdout, r.stderr))
        if verbose:
            sys.stderr.write(r.stderr)
        return obj

    with ThreadPoolExecutor(max_workers=len(SOURCES)) as ex:
        objs = list(ex.map(compile_one, SOURCES))
    tmp = LIB + ".tmp.%d" % os.getpid()
    r = subprocess.run([nvcc, "-shared", "-o", tmp] + objs + ["-gencode", "arch=compute_100a,code=sm_100a"],
                       capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError("link failed:\n%s\n%s" % (r.stdout, r.stderr))
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build(force=True, verbose="-v" in sys.argv))
