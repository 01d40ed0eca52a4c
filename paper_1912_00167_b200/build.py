"""Builds libimpact.so (the C-ABI library) in-tree with nvcc for sm_100a, and the binding's native part beside it."""
from __future__ import annotations

import glob
import os
import re
import subprocess
import sys
import sysconfig
import tempfile
from concurrent.futures import ThreadPoolExecutor

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
LIB = os.path.join(PKG, "libimpact.so")


def marshal_name() -> str:
    """The binding's native part, by the Python and the torch that it is built for: it reads torch's objects through headers
    that are compiled in, so one built for another of either is another module, not this one out of date."""
    import torch
    return "_marshal_" + re.sub(r"\W", "_", "%s_torch_%s_%s" % (sysconfig.get_config_var("SOABI"), torch.__version__,
                                                               (torch.version.git_version or "")[:12]))


def marshal_path() -> str:
    return os.path.join(PKG, marshal_name() + ".so")


def _nvcc() -> str:
    return os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")


def sources() -> list[str]:
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def needs_build() -> bool:
    marshal = marshal_path()
    if not (os.path.exists(LIB) and os.path.exists(marshal)):
        return True
    deps = sources() + glob.glob(os.path.join(CSRC, "*.cpp")) + glob.glob(os.path.join(CSRC, "*.h")) + glob.glob(os.path.join(CSRC, "*.cuh"))
    deps += glob.glob(os.path.join(ROOT, "include", "*.h"))
    return any(os.path.getmtime(d) > min(os.path.getmtime(LIB), os.path.getmtime(marshal)) for d in deps)


def build_marshal() -> None:
    """The native part of the Python binding (csrc/marshal.cpp), against the headers and libraries of the installed torch.  By
    nvcc, which knows where CUDA's headers are however it is named."""
    import torch
    root = os.path.dirname(torch.__file__)
    out = marshal_path()
    tmp = out + ".tmp.%d" % os.getpid()
    subprocess.check_call([_nvcc(), "-gencode", "arch=compute_100a,code=sm_100a", "-O2", "-std=c++17", "-shared", "-cudart", "none", "-Xcompiler", "-fPIC,-fno-gnu-unique",
                           "-DNDEBUG", "-DIMPACT_MARSHAL=" + marshal_name(),
                           "-D_GLIBCXX_USE_CXX11_ABI=%d" % torch.compiled_with_cxx11_abi(), "-I", os.path.join(ROOT, "include"),
                           "-I", sysconfig.get_paths()["include"], "-isystem", os.path.join(root, "include"),
                           "-isystem", os.path.join(root, "include", "torch", "csrc", "api", "include"),
                           os.path.join(CSRC, "marshal.cpp"), "-o", tmp,
                           "-L", os.path.join(root, "lib"), "-lc10", "-lc10_cuda", "-ltorch_cpu", "-ltorch_python"])
    os.replace(tmp, out)


def build(force: bool = False, verbose: bool = False) -> str:
    if not force and not needs_build():
        return LIB
    nvcc = _nvcc()
    # (no unique symbols: a process that loads two copies of the library -- two versions, say -- would share what each kernel
    # remembers of its own configuration, and the second copy's launches would fail)
    flags = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17", "-Xfatbin", "-compress-all",
             "-Xcompiler", "-fPIC,-fno-gnu-unique",
             "-I", os.path.join(ROOT, "include"), "-I", CSRC]
    if verbose:
        flags += ["-Xptxas", "-v"]
    tmp = LIB + ".tmp.%d" % os.getpid()
    with tempfile.TemporaryDirectory() as objs:  # the translation units side by side, then one link
        def compile_one(src: str) -> str:
            obj = os.path.join(objs, os.path.basename(src) + ".o")
            subprocess.check_call([nvcc, *flags, "-c", "-o", obj, src])
            return obj
        with ThreadPoolExecutor(max_workers=os.cpu_count() or 1) as pool:
            marshal = pool.submit(build_marshal)
            done = list(pool.map(compile_one, sources()))
            marshal.result()
        subprocess.check_call([nvcc, "-gencode", "arch=compute_100a,code=sm_100a", "-shared", "-o", tmp, *done])
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
