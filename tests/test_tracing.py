"""A traced module computes the attention of the inputs it is called with: the
call is recorded as the autograd Function, with or without gradients.  The
compute calls make their outputs natively, so a trace that bypassed the Function
would hold nothing but the allocation of an output."""
from __future__ import annotations

import ctypes

import numpy as np
import pytest
import torch

import paper_2606_28560_gb300 as fa
from paper_2606_28560_gb300 import autograd as A


def _x(seed, device="cpu"):
    return torch.randn(1, 2, 70, 64, generator=torch.Generator().manual_seed(seed)).to(device)


class _Model(torch.nn.Module):
    """One public entry point of a forward, as a module of one tensor."""
    def __init__(self, entry, learned):
        super().__init__()
        self.entry = entry
        self.layers = torch.nn.ModuleList(fa.FibAttention(W=8, theta=t, learned=learned) for t in (0.3, -0.2))

    def forward(self, x):
        if self.entry == "module":
            return self.layers[0](x, x, x)
        if self.entry == "function":
            return fa.fib_attention(x, x, x, self.layers[0].theta, self.layers[0].offsets, 8)
        return fa.attention_stack(x, list(self.layers))


def _check(device, entry, learned, grad):
    model = _Model(entry, learned)
    with torch.set_grad_enabled(grad):
        traced = torch.jit.trace(model, (_x(1, device),), check_trace=False)
        x = _x(2, device)
        want = model(x)
        torch.full_like(x, float("nan"))          # what a new allocation may be handed
        assert torch.equal(traced(x), want)


@pytest.fixture
def host_calls(monkeypatch):
    """The native forward calls on host tensors: outputs made as they make them,
    filled through their pointers (with q + 1)."""
    def made(q):
        out = torch.empty(q.shape, dtype=q.dtype)
        src = (q.detach().numpy() + np.float32(1)).astype(np.float32)
        ctypes.memmove(out.data_ptr(), src.ctypes.data, src.nbytes)
        return out
    monkeypatch.setattr(A.B, "fwd", lambda q, k, v, *a, **kw: (made(q), torch.empty(q.shape[:3])))
    monkeypatch.setattr(A.B, "fwd_keep", lambda q, k, v, *a, **kw: (made(q), torch.empty(q.shape[:3]), k, None))


modes = pytest.mark.parametrize("entry,learned,grad", [(e, l, g) for e in ("module", "function", "stack")
                                                       for l in (False, True) for g in (False, True)])


@modes
def test_traced_calls_record_the_function(host_calls, entry, learned, grad):
    _check("cpu", entry, learned, grad)


@pytest.mark.gpu
@modes
def test_traced_calls(entry, learned, grad):
    _check("cuda", entry, learned, grad)
