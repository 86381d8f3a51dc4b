"""What the build makes, in which order, and when it makes it again.  The
compilers are stand-ins that only write their output file."""
from __future__ import annotations

import os
import sys
import types

import pytest
import torch

from paper_2606_28560_gb300 import binding, build as b


@pytest.fixture
def fake(monkeypatch, tmp_path):
    """(commands run, set of programs that fail)"""
    ran, broken = [], set()
    binding.lib()                                 # (the real one, before the paths change)

    def run(cmd, **kw):
        ran.append(cmd)
        if os.path.basename(cmd[0]) in broken:
            return types.SimpleNamespace(returncode=1, stderr="no such header", stdout="")
        with open(cmd[cmd.index("-o") + 1], "w") as f:
            f.write("x")
        return types.SimpleNamespace(returncode=0, stderr="", stdout="")

    monkeypatch.setattr(b.subprocess, "run", run)
    monkeypatch.setattr(b, "_nvcc", lambda: "/opt/cuda/bin/nvcc")
    monkeypatch.setattr(b, "BUILD", str(tmp_path))
    monkeypatch.setattr(b, "LIB", str(tmp_path / "libfibattn.so"))
    monkeypatch.setattr(b, "MARSHAL", str(tmp_path / "fibattn_marshal.so"))
    return ran, broken


def test_the_library_is_made_without_the_native_part(fake):
    _, broken = fake
    broken.add("g++")
    with pytest.raises(RuntimeError, match="marshal"):
        b.build()
    assert os.path.exists(b.LIB) and not os.path.exists(b.MARSHAL)


def test_the_library_needs_no_pytorch(fake, monkeypatch):
    monkeypatch.setitem(sys.modules, "torch", None)
    b.build_library()
    assert os.path.exists(b.LIB)


def test_nothing_is_made_twice(fake):
    ran, _ = fake
    b.build()
    assert os.path.exists(b.LIB) and os.path.exists(b.MARSHAL) and not b.is_stale()
    n = len(ran)
    b.build()
    assert len(ran) == n


def test_another_pytorch(fake, monkeypatch):
    """The native part is made again for it, and is not loaded before that."""
    ran, _ = fake
    b.build()
    n = len(ran)
    monkeypatch.setattr(torch, "__version__", "0.0.1+other")
    assert b.is_stale()
    monkeypatch.setattr(binding, "_marshal_module", None)
    with pytest.raises(RuntimeError, match="another PyTorch"):
        binding._marshal()
    b.build()
    assert not b.is_stale() and all(os.path.basename(c[0]) == "g++" for c in ran[n:]) and len(ran) == n + 2


def test_other_commands(fake):
    b.build()
    with open(b.MARSHAL + ".stamp") as f:
        assert "marshal.cpp" in f.read()
    with open(b.MARSHAL + ".stamp", "a") as f:
        f.write(" -DX")
    assert b.is_stale()
