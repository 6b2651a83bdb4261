"""Build the CUDA shared library in-tree with nvcc for sm_100a."""
from __future__ import annotations

import glob
import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libhbmm.so")
BINDING = os.path.join(HERE, "_binding.so")
INCLUDE = os.path.join(os.path.dirname(HERE), "include")

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-O3", "-lineinfo", "-std=c++17",
    "-Xcompiler", "-fPIC",
]


def _nvcc() -> str:
    for cand in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", "nvcc"):
        if cand and (os.path.isabs(cand) and os.path.exists(cand) or not os.path.isabs(cand)):
            return cand
    raise RuntimeError("nvcc not found")


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _older(target: str, deps) -> bool:
    return not os.path.exists(target) or any(os.path.getmtime(d) > os.path.getmtime(target) for d in deps)


def lib_is_stale() -> bool:
    return _older(LIB, sources() + [f for e in ("*.h", "*.cuh") for f in glob.glob(os.path.join(CSRC, e))] + glob.glob(os.path.join(INCLUDE, "*.h")))


def built_for() -> str:
    """What the binding is compiled against; the module carries it as BUILT_FOR."""
    import torch
    return "torch %s, Python %s" % (torch.__version__, sysconfig.get_config_var("SOABI"))


def binding_is_stale() -> bool:
    if _older(BINDING, glob.glob(os.path.join(CSRC, "*.cpp")) + glob.glob(os.path.join(INCLUDE, "*.h"))):
        return True
    with open(BINDING, "rb") as f:
        return built_for().encode() + b"\0" not in f.read()


def build_lib(force: bool = False, verbose: bool = False) -> str:
    """Compile what is out of date: libhbmm.so from every .cu under csrc/ (one object per file, in parallel), and the binding."""
    if force or lib_is_stale():
        _build_cuda(verbose)
    if force or binding_is_stale():
        build_binding()
    return LIB


def _build_cuda(verbose: bool) -> None:
    nvcc = _nvcc()
    objdir = os.path.join(HERE, "_build")
    os.makedirs(objdir, exist_ok=True)
    procs = []
    objs = []
    for src in sources():
        obj = os.path.join(objdir, os.path.basename(src)[:-3] + ".o")
        objs.append(obj)
        cmd = [nvcc] + NVCC_FLAGS + ["-I", INCLUDE, "-c", src, "-o", obj]
        if verbose:
            cmd.insert(1, "-Xptxas=-v")
        procs.append((src, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)))
    for src, p in procs:
        out, _ = p.communicate()
        if verbose or p.returncode != 0:
            sys.stderr.write(out)
        if p.returncode != 0:
            raise RuntimeError("nvcc failed on %s" % src)
    tmp = LIB + ".tmp.%d" % os.getpid()
    subprocess.check_call([nvcc, "-gencode", "arch=compute_100a,code=sm_100a", "-shared", "-o", tmp] + objs)
    os.replace(tmp, LIB)


def build_binding() -> None:
    """The native marshalling of hbmm.py's hot calls (csrc/binding.cpp), against the running torch and Python."""
    import torch
    from torch.utils import cpp_extension as ext
    tmp = BINDING + ".tmp.%d" % os.getpid()
    include = ext.include_paths("cuda") + [sysconfig.get_paths()["include"], INCLUDE]
    cmd = [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-fPIC", "-shared", os.path.join(CSRC, "binding.cpp"), "-o", tmp]
    cmd += ["-D_GLIBCXX_USE_CXX11_ABI=%d" % torch.compiled_with_cxx11_abi(), '-DHBMM_BUILT_FOR="%s"' % built_for()]
    cmd += [a for d in include for a in ("-isystem", d)] + ["-L" + d for d in ext.library_paths("cuda")]
    subprocess.check_call(cmd + ["-ltorch_python", "-ltorch", "-ltorch_cpu", "-lc10", "-lc10_cuda"])
    os.replace(tmp, BINDING)


if __name__ == "__main__":
    print(build_lib(force="--force" in sys.argv, verbose="-v" in sys.argv))
