"""The compute calls' native marshalling: what it refuses (no GPU needed), and
that a forward for which no gradient is asked equals the training forward."""
from __future__ import annotations

import numpy as np
import pytest
import torch

import paper_2606_28560_gb300 as fa

F = fa.base("fib", 15)


def _qkv(dtype=torch.bfloat16, device="cpu", H=4, Hkv=2, T=40):
    g = torch.Generator().manual_seed(3)
    return [torch.randn(2, h, T, 64, generator=g).to(device=device, dtype=dtype) for h in (H, Hkv, Hkv)]


def test_refusals():
    q, k, v = _qkv()
    with pytest.raises(ValueError):                               # not on a GPU
        fa.fwd(q, k, v, 0.9, F, 8)
    with pytest.raises(ValueError):
        fa.bwd(q, k, v, torch.zeros(2, 4, 40), q, 0.9, F, 8)
    with pytest.raises(TypeError):
        fa.fwd(q.double(), k.double(), v.double(), 0.9, F, 8)
    with pytest.raises(ValueError):                               # q not [B,H,T,D]
        fa.fwd(q[0], k, v, 0.9, F, 8)
    with pytest.raises(KeyError):
        fa.fwd(q, k, v, 0.9, F, 8, kernel="other")
    with pytest.raises(ValueError):
        fa.fwd(q, k, v, 0.9, F, 8, rotated_k=torch.empty(2, 2, 40, 64))
    with pytest.raises(ValueError):
        fa.fwd(q, k, v, 0.9, F, 8, residuals=torch.empty(16, dtype=torch.uint8))
    with pytest.raises(TypeError):
        fa.fwd(q.numpy(force=True) if q.dtype == torch.float32 else np.zeros(q.shape), k, v, 0.9, F, 8)


@pytest.mark.gpu
def test_refusals_on_the_gpu():
    q, k, v = _qkv(device="cuda")
    with pytest.raises(ValueError):
        fa.fwd(q.transpose(1, 2), k, v, 0.9, F, 8)
    with pytest.raises(ValueError):
        fa.fwd(q, k, v.float(), 0.9, F, 8)
    with pytest.raises(fa.FibattnError) as e:
        fa.fwd(q, k, v, 1.7, F, 8)
    assert e.value.status == 1
    with pytest.raises(fa.FibattnError) as e:
        fa.fwd(q, k, v, 0.9, F, 8, workspace=torch.empty(16, dtype=torch.uint8, device="cuda"))
    assert e.value.status == 1
    layer = fa.FibAttention(W=8, learned=False)
    with torch.no_grad(), pytest.raises(RuntimeError):            # function transforms stay refused
        torch.func.vmap(lambda x: layer(x, x, x))(torch.stack([q, q]))
    with torch.autograd.forward_ad.dual_level(), pytest.raises(RuntimeError):
        layer(torch.autograd.forward_ad.make_dual(q, q), k, v)


@pytest.mark.gpu
@pytest.mark.parametrize("dtype,W,Hkv", [(torch.bfloat16, 8, 4), (torch.bfloat16, 12, 1), (torch.bfloat16, 24, 2),
                                         (torch.float32, 8, 2)], ids=["mma", "grouped", "wide", "f32"])
def test_forward_without_gradients(dtype, W, Hkv):
    q, k, v = _qkv(dtype, "cuda", Hkv=Hkv, T=333)
    layer = fa.FibAttention(W=W, theta=0.3).cuda()
    with torch.no_grad():
        plain = layer(q, k, v)
    out = layer(q.requires_grad_(True), k, v)
    assert out.requires_grad and not plain.requires_grad
    assert torch.equal(out.detach(), plain)
    assert torch.equal(fa.fwd(q.detach(), k, v, layer.alpha, layer.offsets, W)[0], plain)
