"""Build libclq.so (the sm_103a kernels and the C ABI) in-tree with nvcc, and
_clq_host.so (the native form of a layer's call from Python) with g++.

Each .cu under csrc/ compiles to its own object in parallel; the objects
link into paper_2509_24416_gb300/libclq.so.  Rebuilds only what changed.
"""
import concurrent.futures
import glob
import os
import shutil
import subprocess
import sys
import sysconfig

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
BUILD = os.path.join(ROOT, "_build")
LIB = os.path.join(PKG, "libclq.so")
HOST_SRC = os.path.join(CSRC, "host_layer.cpp")
HOST = os.path.join(PKG, "_clq_host.so")
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
FLAGS = ["-O3", "-lineinfo", "-std=c++17", "-Xcompiler", "-fPIC",
         "--expt-relaxed-constexpr", "-Xptxas", "-O3"]


def _nvcc():
    p = shutil.which("nvcc")
    if p is None and os.path.exists("/usr/local/cuda/bin/nvcc"):
        p = "/usr/local/cuda/bin/nvcc"
    if p is None:
        raise RuntimeError("nvcc not found: cannot build libclq")
    return p


def _deps():
    heads = glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(
        os.path.join(CSRC, "*.h")) + glob.glob(
        os.path.join(ROOT, "include", "*.h"))
    return max((os.path.getmtime(h) for h in heads), default=0.0)


def _compile(src, obj, extra):
    cmd = [_nvcc()] + ARCH + FLAGS + extra + ["-c", src, "-o", obj]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError("nvcc failed for %s:\n%s%s" % (src, r.stdout,
                                                           r.stderr))
    return r.stderr


def _host_object():
    """Object of the host module, named by the torch and the Python it was compiled
    against."""
    import torch
    return os.path.join(BUILD, "host_layer-%s-%s.o" % (torch.__version__,
                                                       sys.implementation.cache_tag))


def _linked_host():
    """Name of the object that _clq_host.so was linked from, or None."""
    try:
        with open(os.path.join(BUILD, "host_layer.linked")) as f:
            return f.read()
    except OSError:
        return None


def _compile_host(obj):
    import torch
    root = os.path.dirname(torch.__file__)
    nvcc = os.path.dirname(os.path.dirname(os.path.realpath(_nvcc())))
    cmd = ["g++", "-O2", "-std=c++17", "-fPIC", "-I" + os.path.join(root, "include"),
           "-I" + os.path.join(root, "include", "torch", "csrc", "api", "include"),
           "-I" + sysconfig.get_paths()["include"], "-I" + os.path.join(nvcc, "include"),
           "-D_GLIBCXX_USE_CXX11_ABI=%d" % int(torch._C._GLIBCXX_USE_CXX11_ABI),
           "-c", HOST_SRC, "-o", obj]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError("g++ failed for %s:\n%s%s" % (HOST_SRC, r.stdout, r.stderr))
    return ""


def _link_host(obj):
    import torch
    lib = os.path.join(os.path.dirname(torch.__file__), "lib")
    cmd = ["g++", "-shared", "-o", HOST, obj, "-L" + lib, "-lc10", "-lc10_cuda", "-ltorch_cpu",
           "-ltorch_python", "-L" + PKG, "-l:" + os.path.basename(LIB),
           "-Wl,-rpath,$ORIGIN", "-Wl,-rpath," + lib]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError("link failed:\n%s%s" % (r.stdout, r.stderr))
    with open(os.path.join(BUILD, "host_layer.linked"), "w") as f:
        f.write(os.path.basename(obj))


def build(verbose=False, force=False, extra_flags=()):
    os.makedirs(BUILD, exist_ok=True)
    host_obj = _host_object()
    host_new = force or not os.path.exists(host_obj) or os.path.getmtime(host_obj) < max(
        os.path.getmtime(HOST_SRC),
        os.path.getmtime(os.path.join(ROOT, "include", "clq.h")))
    srcs = sorted(glob.glob(os.path.join(CSRC, "*.cu")))
    dep_t = _deps()
    jobs = []
    objs = []
    for s in srcs:
        o = os.path.join(BUILD, os.path.basename(s)[:-3] + ".o")
        objs.append(o)
        if force or not os.path.exists(o) or os.path.getmtime(o) < max(
                os.path.getmtime(s), dep_t):
            jobs.append((s, o))
    if jobs or host_new:
        with concurrent.futures.ThreadPoolExecutor(len(jobs) + 1) as ex:
            futs = [ex.submit(_compile, s, o, list(extra_flags))
                    for s, o in jobs]
            if host_new:
                futs.append(ex.submit(_compile_host, host_obj))
            for f in futs:
                msg = f.result()
                if verbose and msg:
                    print(msg)
    if jobs or not os.path.exists(LIB):
        cmd = [_nvcc()] + ARCH + ["-shared", "-o", LIB] + objs
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError("link failed:\n%s%s" % (r.stdout, r.stderr))
    if (host_new or not os.path.exists(HOST) or _linked_host() != os.path.basename(host_obj)
            or os.path.getmtime(HOST) < os.path.getmtime(host_obj)):
        _link_host(host_obj)
    return LIB


if __name__ == "__main__":
    print(build(verbose=True))
