"""Builds libtdq.so (the C-ABI CUDA library) in-tree with nvcc for sm_100a, and _tdq_host.so (the Python binding's host
side, which reads torch tensors in C++) with g++, where there is a PyTorch and a C++ compiler for it.

    python -m paper_2604_16855_b200.build [--force] [--verbose]

nvcc cross-compiles without a GPU.  The shared object lands next to this file so that it
travels with the source tree; nothing is installed into site-packages.
"""
from __future__ import annotations

import os
import shutil
import subprocess
import sys
from concurrent.futures import ThreadPoolExecutor

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
OBJ = os.path.join(HERE, "_build")
LIB = os.path.join(HERE, "libtdq.so")
HOST = os.path.join(HERE, "_tdq_host.so")
HOST_SOURCE = "tdq_host.cpp"
SOURCES = ["tdq_quantize_act.cu", "tdq_quantize_act_wide.cu", "tdq_quantize_weight.cu", "tdq_linear.cu", "tdq_linear_g32.cu", "tdq_linear_pair.cu", "tdq_linear_defer.cu", "tdq_linear_solo.cu", "tdq_linear_strip.cu", "tdq_linear_one.cu", "tdq_fused.cu", "tdq_api.cu", "tdq_peak.cu"]
NVCC = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
         "-Xcompiler", "-fPIC", "--ftz=false", "--prec-div=true", "--prec-sqrt=true"]


def _newest(keep) -> float:
    """When the newest file of the two source folders that `keep` names, or this one, was written."""
    newest = os.path.getmtime(os.path.abspath(__file__))
    for root in (CSRC, os.path.join(os.path.dirname(HERE), "include")):
        for name in os.listdir(root):
            if keep(name):
                newest = max(newest, os.path.getmtime(os.path.join(root, name)))
    return newest


def _fresh(path: str, newest: float) -> bool:
    return os.path.exists(path) and os.path.getmtime(path) >= newest


def _host_missing() -> str:
    """What the extension module needs and this machine has not got ("" when it has everything)."""
    try:
        import torch
    except ImportError:
        return "PyTorch"
    if torch.version.cuda is None:
        return "a PyTorch with CUDA"
    cxx = os.environ.get("CXX", "g++")
    return "" if shutil.which(cxx) else cxx


def _compile_host():
    """The extension module: torch's headers and libraries, nothing of CUDA but its headers."""
    import sysconfig
    import torch
    tdir = os.path.dirname(torch.__file__)
    tmp = HOST + ".tmp.%d" % os.getpid()
    inc = [os.path.join(tdir, "include"), os.path.join(tdir, "include", "torch", "csrc", "api", "include"),
           sysconfig.get_paths()["include"], os.path.join(os.path.dirname(os.path.dirname(NVCC)), "include")]
    cmd = [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-fPIC", "-shared", "-fvisibility=hidden",
           "-D_GLIBCXX_USE_CXX11_ABI=%d" % int(torch._C._GLIBCXX_USE_CXX11_ABI)]
    cmd += ["-I" + d for d in inc] + [os.path.join(CSRC, HOST_SOURCE), "-o", tmp, "-L" + HERE, "-l:libtdq.so",
                                      "-L" + os.path.join(tdir, "lib"), "-lc10", "-lc10_cuda", "-ltorch_cpu", "-ltorch_cuda", "-ltorch_python",
                                      "-ltorch", "-Wl,-rpath,$ORIGIN"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode:
        sys.stderr.write(r.stdout + r.stderr)
        raise RuntimeError("g++ failed on %s" % HOST_SOURCE)
    os.replace(tmp, HOST)


def build(force: bool = False, verbose: bool = False) -> str:
    """Builds what is older than its sources and returns the path of libtdq.so.  The library needs nvcc alone; where PyTorch
    or a C++ compiler is missing, the binding's extension module is left out (and an older one removed, so that it
    cannot be loaded against another library): callers of the C ABI do not need it."""
    if force or not _fresh(LIB, _newest(lambda name: not name.endswith(".cpp"))):
        _compile_lib(force, verbose)
    if force or not _fresh(HOST, _newest(lambda name: not name.endswith((".cu", ".cuh", ".inc")))):
        missing = _host_missing()
        if not missing:
            _compile_host()
        else:
            if os.path.exists(HOST):
                os.remove(HOST)
            sys.stderr.write("%s is missing: %s is not built, the C library is complete without it\n" % (missing, os.path.basename(HOST)))
    return LIB


def _compile_lib(force: bool, verbose: bool):
    os.makedirs(OBJ, exist_ok=True)
    extra = ["-Xptxas", "-v"] if verbose else []
    headers = _newest(lambda name: not name.endswith((".cu", ".cpp")))

    def compile_one(src):
        obj = os.path.join(OBJ, src.replace(".cu", ".o"))
        if not (force or verbose) and _fresh(obj, max(headers, os.path.getmtime(os.path.join(CSRC, src)))):
            return obj
        cmd = [NVCC] + FLAGS + extra + ["-c", os.path.join(CSRC, src), "-o", obj]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if verbose or r.returncode:
            sys.stderr.write(r.stdout + r.stderr)
        if r.returncode:
            raise RuntimeError("nvcc failed on %s" % src)
        return obj

    with ThreadPoolExecutor(max_workers=len(SOURCES)) as ex:
        objs = list(ex.map(compile_one, SOURCES))
    tmp = LIB + ".tmp.%d" % os.getpid()
    subprocess.check_call([NVCC, "-shared", "-gencode", "arch=compute_100a,code=sm_100a", "-o", tmp] + objs +
                          ["-cudart", "static"])
    os.replace(tmp, LIB)


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="--verbose" in sys.argv))
