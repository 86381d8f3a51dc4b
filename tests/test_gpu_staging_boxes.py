"""The staged rows of the tensor-core kernels at every remainder of an
interval's length: a merged interval is copied as 64-row boxes and, for the
rest, one box of 32 rows (rest <= 32) or 64 (above) that ends with it.  Alphas
whose near interval leaves 0, 8, ..., 56 rows, for both issue forms (W = 8 and
W = 12), with and without residuals, against the fp64 oracle; tolerances are
those of the parity tests (v is halved, so |o| < 4)."""
from __future__ import annotations

import numpy as np
import pytest
import torch

import oracle as O
import paper_2606_28560_gb300 as fa
from paper_2606_28560_gb300 import inputs

F = fa.base("fib", 15)
T = 700
ALPHAS = {0: 0.5274, 8: 0.5411, 16: 0.5548, 24: 0.5822, 32: 0.5959, 40: 0.6233, 48: 0.5, 56: 0.5137}


@pytest.mark.parametrize("W", [8, 12])
@pytest.mark.parametrize("rest", list(ALPHAS))
def test_remainders_are_what_the_cases_stand_for(rest, W):
    for kind in ("query", "key"):
        lens = fa.staging_layout(kind, T, W, ALPHAS[rest], F)["len"]
        assert rest in {int(n) % 64 for n in lens}
        assert min(lens) >= 64                    # a box of the rest never starts before its interval


@pytest.mark.gpu
@pytest.mark.parametrize("Hkv", [2, 1])
@pytest.mark.parametrize("W", [8, 12])
@pytest.mark.parametrize("rest", list(ALPHAS))
def test_forward_and_backward(rest, W, Hkv):
    alpha = ALPHAS[rest]
    q, k, v = inputs.qkv(1, 2, T, seed=100 + rest, dtype=torch.bfloat16, Hkv=Hkv)
    v = (v * 0.5).to(torch.bfloat16)
    g = inputs.dout(1, 2, T, seed=101 + rest, dtype=torch.bfloat16)
    qc, kc, vc, gc = (x.cuda() for x in (q, k, v, g))
    plain, _ = fa.fwd(qc, kc, vc, alpha, F, W, kernel="mma")
    rk, res = fa.rotated_k_like(kc), fa.residuals_like(qc, W, len(F))
    out, lse = fa.fwd(qc, kc, vc, alpha, F, W, rotated_k=rk, residuals=res)
    grads = fa.bwd(qc, kc, vc, lse, gc, alpha, F, W, out=out, rotated_k=rk, residuals=res, kernel="mma")
    torch.cuda.synchronize()
    assert torch.equal(out, plain)
    n64 = [x.double().numpy() for x in (q, k, v, g)]
    d = O.offsets_fp32(float(np.float32(alpha)), F.astype(np.float64))
    ro, _ = O.forward(*n64[:3], W, d, nthreads=8)
    ref = O.backward(*n64, W, d, nthreads=8)
    assert np.max(np.abs(out.double().cpu().numpy() - ro)) <= 1e-2
    for x, r in zip(grads[:3] + grads[4:], ref):
        assert np.max(np.abs(x.double().cpu().numpy() - r)) <= 3e-2 * np.max(np.abs(r))
