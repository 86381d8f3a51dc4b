"""Windows longer than the sequence in the row-gather passes: only the slots that
a warp's rows have are walked, and no others are written to or read from the
workspace (which starts as NaN here).  Against the fp64 oracle with the
tolerances of the parity tests: fp32 1e-4; bf16 1e-2 on the output and 3e-2 of the
largest reference entry on gradients (v halved keeps |o| < 4)."""
from __future__ import annotations

import numpy as np
import pytest
import torch

import oracle as O
import paper_2606_28560_gb300 as fa
from paper_2606_28560_gb300 import inputs

pytestmark = pytest.mark.gpu

# (B, H, Hkv, T, W): one chunk of 208 slots or several, blocks whose warps share
# rows or do not, T at 16-row edges and about the chunk
CASES = [(1, 2, 1, 1, 40), (2, 2, 2, 15, 17), (1, 2, 1, 16, 300), (1, 1, 1, 17, 1024), (2, 4, 2, 100, 1024),
         (1, 2, 2, 207, 207), (1, 2, 1, 208, 208), (1, 2, 1, 209, 431), (20, 32, 16, 70, 69), (16, 8, 8, 300, 299),
         (4, 16, 4, 230, 1024), (1, 1, 1, 640, 500)]
F = fa.base("fib", 15)


@pytest.mark.parametrize("dedup", [True, False])
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16], ids=["f32", "bf16"])
@pytest.mark.parametrize("case", CASES, ids=["B%dH%dkv%dT%dW%d" % c for c in CASES])
def test_window_beyond_the_ends(case, dtype, dedup):
    B, H, Hkv, T, W = case
    alpha = 0.77
    q, k, v = inputs.qkv(B, H, T, seed=T + W, dtype=dtype, Hkv=Hkv)
    g = inputs.dout(B, H, T, seed=T + W + 1, dtype=dtype)
    v = (v * 0.5).to(dtype)
    qc, kc, vc, gc = (x.cuda() for x in (q, k, v, g))
    ws = torch.full((fa.bwd_workspace_bytes(B, H, T, W, len(F), dtype, Hkv=Hkv) // 4,), float("nan"), device="cuda")
    out, lse = fa.fwd(qc, kc, vc, alpha, F, W, kernel="gather", dedup=dedup)
    grads = fa.bwd(qc, kc, vc, lse, gc, alpha, F, W, kernel="gather", dedup=dedup, workspace=ws.view(torch.uint8))
    torch.cuda.synchronize()
    n64 = [x.double().numpy() for x in (q, k, v, g)]
    d = O.offsets_fp32(float(np.float32(alpha)), F.astype(np.float64))
    ro, rl = O.forward(*n64[:3], W, d, nthreads=8, dedup=dedup)
    ref = O.backward(*n64, W, d, nthreads=8, dedup=dedup)
    tol, gtol = (1e-4, 1e-4) if dtype == torch.float32 else (1e-2, 3e-2)
    assert np.max(np.abs(out.double().cpu().numpy() - ro)) <= tol
    assert np.max(np.abs(lse.double().cpu().numpy() - rl)) <= tol
    for name, x, r in zip(("dq", "dk", "dv", "dd"), grads[:3] + grads[4:], ref):
        e = np.max(np.abs(x.double().cpu().numpy() - r)) / max(np.max(np.abs(r)), 1e-2)
        assert e <= gtol, (name, e)


def _us(fn, n=20):
    for _ in range(3):
        fn()
    times = []
    for _ in range(5):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        torch.cuda._sleep(2_000_000)              # the host runs ahead of the device
        a.record()
        for _ in range(n):
            fn()
        b.record()
        torch.cuda.synchronize()
        times.append(a.elapsed_time(b) * 1e3 / n)
    return min(times)


def test_a_longer_window_costs_no_more_than_the_sequence():
    """W = 1024 and W = 127 attend the same rows of T = 128; the longer window goes
    through the table in chunks.  It took 6 times as long forward and backward
    while every slot was walked; the bound leaves room for the chunked kernels."""
    B, H, T = 16, 8, 128
    q, k, v, g = (x.cuda() for x in inputs.qkv(B, H, T, seed=1) + (inputs.dout(B, H, T, seed=2),))
    ws = torch.empty(fa.bwd_workspace_bytes(B, H, T, 1024, len(F), torch.float32), dtype=torch.uint8, device="cuda")
    out, lse = fa.fwd(q, k, v, 0.9, F, 127)

    def layer(W):
        fa.fwd(q, k, v, 0.9, F, W, out=out, lse=lse, workspace=ws)
        fa.bwd(q, k, v, lse, g, 0.9, F, W, workspace=ws)
    assert _us(lambda: layer(1024)) <= 3 * _us(lambda: layer(127))


def test_tables_are_made_for_the_sequence():
    """The same at T = 20, where tables of 208 slots left one block an SM: three
    times W = 19's time; now the two take the same kernels and sizes."""
    B, H, T = 64, 16, 20
    q, k, v, g = (x.cuda() for x in inputs.qkv(B, H, T, seed=1) + (inputs.dout(B, H, T, seed=2),))
    ws = torch.empty(fa.bwd_workspace_bytes(B, H, T, 1024, len(F), torch.float32), dtype=torch.uint8, device="cuda")
    out, lse = fa.fwd(q, k, v, 0.9, F, 19)

    def layer(W):
        fa.fwd(q, k, v, 0.9, F, W, out=out, lse=lse, workspace=ws)
        fa.bwd(q, k, v, lse, g, 0.9, F, W, workspace=ws)
    assert _us(lambda: layer(1024)) <= 1.5 * _us(lambda: layer(19))
