"""The static shared memory that the dispatch subtracts from the limit of a
block covers what the compiler gives the kernels: a layout that the dispatch
accepts would otherwise be refused at its launch."""
from __future__ import annotations

import ctypes
import os
import re
import subprocess

import pytest

from paper_2606_28560_gb300 import build as b
import paper_2606_28560_gb300 as fa

LIMIT = 227 * 1024
# source file, kernel (one template instance or all), what the dispatch counts
CASES = [("bwd_key_mma.cu", "bwd_key_mma_kernel", "_ZN7fibattn23bwd_key_mma_static_smemEv"),
         ("bwd_mma.cu", "bwd_query_mma_kernel", "_ZN7fibattn19bwd_mma_static_smemEv"),
         ("fwd_mma.cu", r"fwd_mma_kernelILi\dELi1E", "_ZN7fibattn19fwd_mma_static_smemEv"),
         ("fwd_mma.cu", r"fwd_mma_kernelILi\dELi2E", "_ZN7fibattn22fwd_mma_gqa_smem_limitEv")]


@pytest.fixture(scope="module")
def compiled(tmp_path_factory):
    """{file: [(kernel, bytes of static shared memory)]} as the compiler reports them."""
    out = tmp_path_factory.mktemp("smem")
    procs = {}
    for f in sorted({c[0] for c in CASES}):
        cmd = [b._nvcc(), *b.ARCH, *b.NVCC_FLAGS, "-Xptxas", "-v", "-I", b.INCLUDE, "-c", os.path.join(b.CSRC, f),
               "-o", str(out / (f + ".o"))]
        procs[f] = subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)
    found = {}
    for f, p in procs.items():
        text = p.communicate(timeout=600)[0]
        assert p.returncode == 0, text
        found[f] = [(name, int(n)) for name, n in
                    re.findall(r"Compiling entry function '(\w+)'(?:(?!Compiling).)*?(\d+) bytes smem", text, re.S)]
    return found


@pytest.mark.parametrize("file,kernel,symbol", CASES, ids=["key", "query", "forward", "grouped"])
def test_counted_static_shared_memory(compiled, file, kernel, symbol):
    counted = getattr(fa.lib(), symbol)
    counted.restype, counted.argtypes = ctypes.c_size_t, []
    n = counted()
    if symbol.endswith("limitEv"):                # (a limit of the dynamic part)
        n = LIMIT - n
    sizes = [size for name, size in compiled[file] if re.search(kernel, name)]
    assert len(sizes) >= 3 and max(sizes) <= n
