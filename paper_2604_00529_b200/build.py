"""Builds libmxq.so (the CUDA C-ABI library) in-tree with nvcc for sm_100a.

    python -m paper_2604_00529_b200.build [--force] [--debug]

One object per translation unit under ``_build/`` (compiled in parallel), linked into
``paper_2604_00529_b200/libmxq.so``; then ``mxq_abi_timing``, a small C-level caller of the ABI, and ``_mxq_host``,
the native part of the Python binding (for the torch and Python at hand).  A unit is rebuilt when it or any header is
newer than its object.
"""
from __future__ import annotations

import os
import re
import subprocess
import sys
import sysconfig
from concurrent.futures import ThreadPoolExecutor

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
OBJ_DIR = os.path.join(ROOT, "_build")
LIB = os.path.join(HERE, "libmxq.so")
TIMING_EXE = os.path.join(HERE, "mxq_abi_timing")      # C-level caller of the ABI (csrc/abi_timing.cu)
UNITS = ["mxq_api", "mxq_quantize", "mxq_slice_scale", "mxq_dequantize", "mxq_fake_quant", "mxq_static_batch", "mxq_slice_scale_multi", "mxq_slice_scale_multi_fp", "mxq_layout", "mxq_fake_quant_batched"]
NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-std=c++20", "-O3", "-lineinfo",
              "-Xcompiler", "-fPIC", "-Xcompiler", "-fvisibility=hidden"]


def _nvcc() -> str:
    for cand in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", "nvcc"):
        if cand and (os.path.isabs(cand) and os.path.exists(cand) or not os.path.isabs(cand)):
            return cand
    return "nvcc"


def _headers():
    hs = [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith((".cuh", ".h"))]
    hs.append(os.path.join(ROOT, "include", "mxq.h"))
    return hs


def _stale(target: str, deps) -> bool:
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    return any(os.path.getmtime(d) > t for d in deps)


DEBUG_LIB = os.path.join(HERE, "libmxq_debug.so")      # the same sources with -DMXQ_DEBUG (bounds-checked accesses)


def build(force: bool = False, verbose: bool = False, debug: bool = False) -> str:
    """Builds libmxq.so (and mxq_abi_timing); with debug=True builds libmxq_debug.so instead."""
    if debug:
        return _build_library(os.path.join(ROOT, "_build_debug"), DEBUG_LIB, ["-DMXQ_DEBUG"], force, verbose, timing=False)
    lib = _build_library(OBJ_DIR, LIB, [], force, verbose, timing=True)
    if _torch_folder() is None:
        print("no torch with CUDA here: the C library is built, the Python binding's _mxq_host is not", file=sys.stderr)
    else:
        build_host_module(force)
    return lib


def _torch_folder():
    """The folder of a torch that _mxq_host can be built against (its headers and CUDA libraries), or None: users of the C
    library alone need neither."""
    try:
        import torch
    except ImportError:
        return None
    top = os.path.dirname(torch.__file__)
    need = (("include", "torch", "csrc", "autograd", "custom_function.h"), ("lib", "libtorch_python.so"), ("lib", "libc10_cuda.so"))
    return top if all(os.path.exists(os.path.join(top, *n)) for n in need) else None


def host_module_path() -> str:
    """The file of _mxq_host for the torch and the Python that run: it holds the C++ layouts of the one and the ABI of the
    other, so each combination has a module of its own."""
    import torch
    return os.path.join(HERE, "_mxq_host.torch-%s-abi%d%s" % (re.sub(r"[^0-9A-Za-z.]", "_", torch.__version__),
                                                             torch.compiled_with_cxx11_abi(), sysconfig.get_config_var("EXT_SUFFIX")))


def build_host_module(force: bool = False) -> str:
    """Builds _mxq_host, the CPython module of binding.py (csrc/host_calls.cpp), against the installed torch."""
    src, target = os.path.join(CSRC, "host_calls.cpp"), host_module_path()
    if not (force or _stale(target, [src, os.path.join(ROOT, "include", "mxq.h"), os.path.abspath(__file__)])):
        return target
    import torch
    top = _torch_folder()
    if top is None:
        raise RuntimeError("_mxq_host needs a torch with its headers and CUDA libraries; %s has none" % torch.__file__)
    cuda = os.path.dirname(os.path.dirname(_nvcc())) if os.path.isabs(_nvcc()) else "/usr/local/cuda"
    tmp = target + ".tmp.%d" % os.getpid()
    cmd = [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-fPIC", "-shared", "-fvisibility=hidden",
           "-D_GLIBCXX_USE_CXX11_ABI=%d" % int(torch.compiled_with_cxx11_abi())]
    for d in (os.path.join(top, "include"), os.path.join(top, "include", "torch", "csrc", "api", "include"),
              os.path.join(cuda, "include"), sysconfig.get_paths()["include"]):
        cmd += ["-isystem", d]
    # The C++ runtime is named by its shared object: a compiler whose own folder has only libstdc++.a would link a second
    # copy of the runtime into the module, and a stream or an error message made there then crashes the process.
    cmd += [src, "-o", tmp, "-L" + os.path.join(top, "lib"), "-ltorch_python", "-ltorch", "-ltorch_cpu", "-lc10_cuda", "-lc10",
            "-nostdlib++", "-l:libstdc++.so.6"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError("g++ failed: %s\n%s" % (" ".join(cmd), r.stderr))
    os.replace(tmp, target)
    return target


def _build_library(obj_dir: str, lib: str, extra, force: bool, verbose: bool, timing: bool) -> str:
    OBJ_DIR, LIB = obj_dir, lib
    os.makedirs(OBJ_DIR, exist_ok=True)
    headers = _headers()
    units = [u for u in UNITS if os.path.exists(os.path.join(CSRC, u + ".cu"))]
    jobs = []
    for u in units:
        src = os.path.join(CSRC, u + ".cu")
        obj = os.path.join(OBJ_DIR, u + ".o")
        if force or _stale(obj, [src] + headers):
            cmd = [_nvcc()] + NVCC_FLAGS + list(extra) + (["-Xptxas", "-v"] if verbose else []) + ["-c", src, "-o", obj]
            jobs.append(cmd)

    def run(cmd):
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError("nvcc failed: %s\n%s\n%s" % (" ".join(cmd), r.stdout, r.stderr))
        return r.stderr

    if jobs:
        with ThreadPoolExecutor(max_workers=min(len(jobs), os.cpu_count() or 1)) as ex:
            for log in ex.map(run, jobs):
                if verbose and log:
                    sys.stderr.write(log)
    objs = [os.path.join(OBJ_DIR, u + ".o") for u in units]
    if force or jobs or _stale(LIB, objs):
        tmp = LIB + ".tmp.%d" % os.getpid()
        run([_nvcc(), "-shared", "-o", tmp] + objs + ["-gencode", "arch=compute_100a,code=sm_100a"])
        os.replace(tmp, LIB)
    timing_src = os.path.join(CSRC, "abi_timing.cu")
    if timing and os.path.exists(timing_src) and (force or _stale(TIMING_EXE, [timing_src, LIB, os.path.join(ROOT, "include", "mxq.h")])):
        tmp = TIMING_EXE + ".tmp.%d" % os.getpid()
        run([_nvcc(), "-O2", "-std=c++17", "-gencode", "arch=compute_100a,code=sm_100a", timing_src, "-o", tmp,
             "-L" + HERE, "-lmxq", "-Xlinker", "-rpath", "-Xlinker", "$ORIGIN"])
        os.replace(tmp, TIMING_EXE)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv, debug="--debug" in sys.argv))
