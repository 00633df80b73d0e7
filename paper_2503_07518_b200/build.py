"""Builds libtokenbutler.so in-tree with nvcc for sm_100a (no JIT cache, no torch extension), and beside it the
extension module through which binding.py makes the per-step calls."""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libtokenbutler.so")
CALLS = os.path.join(HERE, "_tokenbutler.so")
SOURCES = ["tb_api.cu", "tb_cache.cu", "tb_select.cu", "tb_select_wave.cu", "tb_select_small.cu", "tb_select_stream.cu", "tb_select_aux.cu", "tb_attention.cu", "tb_predictor.cu"]
NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17", "-Xcompiler", "-fPIC",
              "--expt-relaxed-constexpr", "--expt-extended-lambda"]


def calls_abi() -> str:
    """What the extension module is compiled against and cannot be loaded without: torch's and CPython's C++ interfaces."""
    import importlib.metadata
    return "built for torch %s, %s" % (importlib.metadata.version("torch"), sysconfig.get_config_var("SOABI"))


def calls_match() -> bool:
    """Whether the extension module was built for the torch and Python that are running (it carries their names)."""
    with open(CALLS, "rb") as f:
        return calls_abi().encode() + b"\0" in f.read()


def _stale() -> bool:
    if not os.path.exists(LIB) or not os.path.exists(CALLS) or not calls_match():
        return True
    t = min(os.path.getmtime(LIB), os.path.getmtime(CALLS))
    deps = [os.path.join(CSRC, f) for f in os.listdir(CSRC)] + [os.path.join(HERE, "..", "include", "tokenbutler.h")]
    return any(os.path.getmtime(d) > t for d in deps)


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile the sources that changed and link the library.  Safe to call from several processes at
    once (every rank of a multi-GPU run, parallel test workers): one builds under a file lock, the others
    wait for it and find the library up to date."""
    if not force and not _stale():
        return LIB
    import fcntl
    with open(os.path.join(HERE, ".build.lock"), "w") as lock:
        fcntl.flock(lock, fcntl.LOCK_EX)
        try:
            if not force and not _stale():      # another process built it while this one waited
                return LIB
            return _build_locked(verbose)
        finally:
            fcntl.flock(lock, fcntl.LOCK_UN)


def _build_locked(verbose: bool) -> str:
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    import torch
    cxx = os.environ.get("CXX", "g++")
    torch_dir = os.path.dirname(torch.__file__)
    calls_obj = os.path.join(CSRC, "tb_python.o")
    calls = subprocess.Popen([cxx, "-O2", "-std=c++17", "-fPIC", '-DTB_CALLS_ABI="%s"' % calls_abi(), "-D_GLIBCXX_USE_CXX11_ABI=%d" % torch._C._GLIBCXX_USE_CXX11_ABI,
                              "-I" + sysconfig.get_paths()["include"], "-I" + os.path.join(torch_dir, "include"),
                              "-I" + os.path.join(torch_dir, "include", "torch", "csrc", "api", "include"),
                              "-I" + os.path.join(os.path.dirname(os.path.dirname(nvcc)), "include"), "-c", os.path.join(CSRC, "tb_python.cpp"),
                              "-o", calls_obj], stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)
    objs = []
    procs = []
    for src in SOURCES:
        obj = os.path.join(CSRC, src.replace(".cu", ".o"))
        cmd = [nvcc, *NVCC_FLAGS, "-c", os.path.join(CSRC, src), "-o", obj]
        if verbose:
            cmd.insert(1, "-Xptxas=-v")
        procs.append((src, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)))
        objs.append(obj)
    for src, p in procs:
        out, _ = p.communicate()
        if verbose or p.returncode:
            sys.stderr.write(out)
        if p.returncode:
            raise RuntimeError("nvcc failed on %s" % src)
    tmp = LIB + ".%d.tmp" % os.getpid()
    subprocess.check_call([nvcc, "-shared", "-o", tmp, *objs, "-gencode", "arch=compute_100a,code=sm_100a"])
    os.replace(tmp, LIB)
    out, _ = calls.communicate()
    if calls.returncode:
        sys.stderr.write(out)
        raise RuntimeError("compiling tb_python.cpp failed")
    # the library is found beside the module ($ORIGIN), under the name it has there; torch's are loaded when it is imported
    tmp = CALLS + ".%d.tmp" % os.getpid()
    subprocess.check_call([cxx, "-shared", calls_obj, "-o", tmp, "-L" + HERE, "-l:" + os.path.basename(LIB), "-L" + os.path.join(torch_dir, "lib"),
                           "-lc10", "-lc10_cuda", "-ltorch_cpu", "-ltorch_python", "-Wl,-rpath,$ORIGIN"])
    os.replace(tmp, CALLS)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
