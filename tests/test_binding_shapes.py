"""Shapes, types and sizes that would have a kernel read or write past a tensor
are refused on the host, before any launch: the library sees pointers and the
extents of q.  The refusals do not depend on the device of the tensors, so the
same cases run on host tensors here and on the GPU."""
from __future__ import annotations

import pytest
import torch

import paper_2606_28560_gb300 as fa

F = fa.base("fib", 15)
B, H, HKV, T, W = 2, 4, 2, 40, 8


def _args(device, dtype=torch.bfloat16):
    g = torch.Generator().manual_seed(3)
    q, k, v, do = (torch.randn(B, h, T, 64, generator=g).to(device=device, dtype=dtype) for h in (H, HKV, HKV, H))
    return dict(q=q, k=k, v=v, dout=do, lse=torch.zeros(B, H, T, device=device))


def _empty(*shape, dtype=torch.bfloat16):
    return lambda device: torch.empty(shape, dtype=dtype, device=device)


f32, i32 = torch.float32, torch.int32
FWD = {
    "k short": ("k", _empty(B, HKV, T - 1, 64), "k and v must be"), "k batch": ("k", _empty(1, HKV, T, 64), "k and v must be"),
    "v heads": ("v", _empty(B, 1, T, 64), "k and v must be"), "v dim": ("v", _empty(B, HKV, T, 32), "k and v must be"),
    "out short": ("out", _empty(B, H, T - 1, 64), "out must be"), "out type": ("out", _empty(B, H, T, 64, dtype=f32), "out must be"),
    "out strided": ("out", lambda d: torch.empty(B, T, H, 64, dtype=torch.bfloat16, device=d).transpose(1, 2), "out must be"),
    "lse type": ("lse", _empty(B, H, T), "lse must be"), "lse short": ("lse", _empty(B, H, T - 8, dtype=f32), "lse must be"),
    "workspace strided": ("workspace", lambda d: torch.empty(1 << 18, dtype=torch.uint8, device=d)[::2], "workspace must be"),
}
BWD = {
    "k short": FWD["k short"], "v heads": FWD["v heads"], "out short": FWD["out short"], "lse type": FWD["lse type"],
    "dout short": ("dout", _empty(B, H, T - 1, 64), "dout must be"), "lse short": FWD["lse short"],
    "dq short": ("dq", _empty(B, 1, T, 64), "dq must be"), "dq type": ("dq", _empty(B, H, T, 64, dtype=f32), "dq must be"),
    "dk short": ("dk", _empty(B, 1, T, 64), "dk must be"), "dv short": ("dv", _empty(B, HKV, T, 16), "dv must be"),
    "dtheta type": ("dtheta", _empty(1, dtype=torch.float64), "dtheta must be"),
    "dtheta none": ("dtheta", _empty(0, dtype=f32), "dtheta must be"),
    "dd short": ("dd", _empty(14, dtype=f32), "dd must be"), "dd type": ("dd", _empty(15, dtype=i32), "dd must be"),
    "workspace strided": FWD["workspace strided"],
}


def _call(which, device, name, make):
    a = _args(device)
    kw = {name: make(device)}
    a.update({n: kw.pop(n) for n in list(kw) if n in a and (which == "bwd" or n != "lse")})
    if which == "fwd":
        fa.fwd(a["q"], a["k"], a["v"], 0.9, F, W, **kw)
    else:
        fa.bwd(a["q"], a["k"], a["v"], a["lse"], a["dout"], 0.9, F, W, **kw)


@pytest.mark.parametrize("device", ["cpu", pytest.param("cuda", marks=pytest.mark.gpu)])
@pytest.mark.parametrize("which,case", [("fwd", c) for c in FWD] + [("bwd", c) for c in BWD])
def test_refused_on_the_host(which, case, device):
    name, make, msg = (FWD if which == "fwd" else BWD)[case]
    with pytest.raises(ValueError, match=msg):
        _call(which, device, name, make)


@pytest.mark.gpu
def test_buffers_off_the_gpu_are_refused():
    a = _args("cuda")
    for kw in (dict(lse=torch.empty(B, H, T)), dict(out=torch.empty(B, H, T, 64, dtype=torch.bfloat16)),
               dict(workspace=torch.empty(1 << 20, dtype=torch.uint8))):
        with pytest.raises(ValueError):
            fa.fwd(a["q"], a["k"], a["v"], 0.9, F, W, **kw)


@pytest.mark.gpu
def test_larger_and_flat_buffers_are_taken():
    """What holds a call's entries is accepted whatever its shape."""
    a = _args("cuda")
    want, lse = fa.fwd(a["q"], a["k"], a["v"], 0.9, F, W)
    big = torch.empty(B * H * T * 64 + 64, dtype=torch.bfloat16, device="cuda")
    flat = torch.empty(B * H * T + 8, device="cuda")
    out, _ = fa.fwd(a["q"], a["k"], a["v"], 0.9, F, W, out=big, lse=flat)
    assert out is big or out.data_ptr() == big.data_ptr()
    assert torch.equal(big[:want.numel()].view_as(want), want) and torch.equal(flat[:lse.numel()].view_as(lse), lse)
    ref = fa.bwd(a["q"], a["k"], a["v"], lse, a["dout"], 0.9, F, W, out=want)
    got = fa.bwd(a["q"], a["k"], a["v"], flat, a["dout"], 0.9, F, W, out=big, dtheta=torch.empty(4, device="cuda"),
                 dd=torch.empty(32, device="cuda"))
    assert all(torch.equal(x, y) for x, y in zip(ref, got)) and got[3].shape == (1,) and got[4].shape == (15,)
