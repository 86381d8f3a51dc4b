"""Build the CUDA library in-tree for sm_103a (GB300) with nvcc.

Each ``csrc/*.cu`` translation unit is compiled in parallel, then linked into
``_build/libfibattn.so`` against the shared CUDA runtime.  The library needs
nothing of PyTorch; ``csrc/marshal.cpp``, the binding's native part, is compiled
with g++ against PyTorch's headers into ``_build/fibattn_marshal.so`` after it.
Rebuilds what is older than a source, a header or this file, and the native part
also when it was made for another PyTorch or Python, or by other commands.
"""
from __future__ import annotations

import glob
import os
import shutil
import subprocess
import sysconfig
from concurrent.futures import ThreadPoolExecutor

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
INCLUDE = os.path.join(os.path.dirname(HERE), "include")
BUILD = os.path.join(HERE, "_build")
LIB = os.path.join(BUILD, "libfibattn.so")
MARSHAL = os.path.join(BUILD, "fibattn_marshal.so")
MARSHAL_SRC = os.path.join(CSRC, "marshal.cpp")
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
NVCC_FLAGS = ["-O3", "-lineinfo", "-std=c++17", "-Xcompiler", "-fPIC", "--expt-relaxed-constexpr",
              "-Xptxas", "-warn-spills"]


def _nvcc() -> str:
    home = os.environ.get("CUDA_HOME") or os.environ.get("CUDA_PATH") or "/usr/local/cuda"
    cand = os.path.join(home, "bin", "nvcc")
    if os.path.exists(cand):
        return cand
    found = shutil.which("nvcc")
    if not found:
        raise RuntimeError("nvcc not found: set CUDA_HOME")
    return found


def _sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _older(target, deps) -> bool:
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    return any(os.path.getmtime(p) > t for p in deps)


def library_is_stale() -> bool:
    return _older(LIB, _sources() + glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(INCLUDE, "*.h")) +
                  [os.path.abspath(__file__)])


def _marshal_abi() -> str:
    """What the native part is bound to: PyTorch's C++ interface and Python's."""
    import torch
    return f"torch {torch.__version__} {sysconfig.get_config_var('SOABI')}"


def _marshal_commands(nvcc, obj, out):
    """The native part's compile and link commands."""
    import torch
    tdir = os.path.dirname(torch.__file__)
    tlib = os.path.join(tdir, "lib")
    cuda = os.path.dirname(os.path.dirname(nvcc))
    inc = [os.path.join(tdir, "include"), os.path.join(tdir, "include", "torch", "csrc", "api", "include"),
           sysconfig.get_paths()["include"], os.path.join(cuda, "include")]
    return (["g++", "-O2", "-std=c++17", "-fPIC", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
             *[f"-I{d}" for d in inc], "-c", MARSHAL_SRC, "-o", obj],
            ["g++", "-shared", "-o", out, obj, f"-L{BUILD}", "-lfibattn", f"-L{tlib}", "-lc10", "-lc10_cuda",
             "-ltorch_cpu", "-ltorch_python", "-Wl,-rpath,$ORIGIN", f"-Wl,-rpath,{tlib}",
             f"-Wl,-rpath,{os.path.join(cuda, 'lib64')}"])


def _marshal_stamp() -> str:
    """Kept beside the native part: its interfaces, then its commands."""
    return "\n".join([_marshal_abi(), *(" ".join(c) for c in _marshal_commands(_nvcc(), "obj", "out"))])


def _built_stamp() -> str:
    try:
        with open(MARSHAL + ".stamp") as f:
            return f.read()
    except OSError:
        return ""


def marshal_is_stale() -> bool:
    return (_older(MARSHAL, [MARSHAL_SRC, os.path.join(INCLUDE, "fibattn.h"), os.path.abspath(__file__)]) or
            _built_stamp() != _marshal_stamp())


def marshal_fits() -> bool:
    """Whether the native part was built for the PyTorch and Python that run."""
    return _built_stamp().split("\n")[0] == _marshal_abi()


def is_stale() -> bool:
    return library_is_stale() or marshal_is_stale()


def _run(cmd, what, verbose=False):
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"{what} failed:\n{r.stderr}")
    if verbose and r.stderr:
        print(r.stderr)


def _pool():
    return ThreadPoolExecutor(max_workers=max(1, min(8, os.cpu_count() or 1)))


def build_library(force: bool = False, verbose: bool = False) -> str:
    """The CUDA library alone."""
    if not force and not library_is_stale():
        return LIB
    os.makedirs(BUILD, exist_ok=True)
    nvcc = _nvcc()
    cuda_lib = os.path.join(os.path.dirname(os.path.dirname(nvcc)), "lib64")

    def compile_one(src):
        obj = os.path.join(BUILD, os.path.basename(src) + ".o")
        _run([nvcc, *ARCH, *NVCC_FLAGS, "-I", INCLUDE, "-c", src, "-o", obj], f"nvcc on {os.path.basename(src)}", verbose)
        return obj

    with _pool() as ex:
        objs = list(ex.map(compile_one, _sources()))
    tmp = LIB + f".tmp{os.getpid()}"
    _run([nvcc, *ARCH, "-shared", "-cudart", "shared", "-o", tmp, *objs, "-Xlinker", f"-rpath={cuda_lib}"], "link")
    os.replace(tmp, LIB)
    return LIB


def build(force: bool = False, verbose: bool = False) -> str:
    """The library, then the binding's native part (compiled alongside; linked
    against the library, which is in place whatever becomes of it)."""
    os.makedirs(BUILD, exist_ok=True)
    obj, tmp = os.path.join(BUILD, "marshal.cpp.o"), MARSHAL + f".tmp{os.getpid()}"

    def compile_marshal():
        if not force and not marshal_is_stale():
            return None
        compile_cmd, link_cmd = _marshal_commands(_nvcc(), obj, tmp)
        _run(compile_cmd, "g++ on marshal.cpp")
        return link_cmd

    with _pool() as ex:
        native = ex.submit(compile_marshal)
        build_library(force, verbose)
        link_cmd = native.result()
    if link_cmd:
        _run(link_cmd, "link of marshal")
        os.replace(tmp, MARSHAL)
        with open(MARSHAL + ".stamp", "w") as f:
            f.write(_marshal_stamp())
    return LIB


if __name__ == "__main__":
    import sys
    make = build_library if "--library" in sys.argv else build
    print(make(force="--force" in sys.argv, verbose=True))
