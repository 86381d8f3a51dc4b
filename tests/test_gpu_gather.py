"""The row-gather passes at the edges of their blocking, against the fp64
oracle: a warp works on 16 consecutive rows, a block on 16 (its warps share
them) or 64; rows come in batches of 6 (fp32) or 8, rungs singly or in pairs;
a window beyond 208 slots is taken in chunks.

Tolerances are those of the parity tests: fp32 1e-4; bf16 1e-2 on the output
and 3e-2 of the largest reference entry on gradients (v halved keeps |o| < 4).
"""
from __future__ import annotations

import numpy as np
import pytest
import torch

import oracle as O
import paper_2606_28560_gb300 as fa
from paper_2606_28560_gb300 import inputs

pytestmark = pytest.mark.gpu

# (B, H, Hkv, T, W, alpha, base, K): blocks of 16 shared rows up to 608 of
# them, 64-row blocks beyond; T at 16- and 64-row edges; W at batch edges
CASES = [
    (1, 1, 1, 16, 2, 0.9, "fib", 15), (1, 2, 1, 17, 0, 1.3, "pow2", 10), (2, 2, 2, 65, 17, 1.0, "fib", 3),
    (1, 2, 2, 300, 5, 0.77, "fib", 15), (19, 32, 8, 16, 3, 0.6, "fib", 5), (19, 33, 33, 16, 4, 0.6, "fib", 4),
    (20, 32, 16, 63, 8, 1.4, "fib", 15), (20, 32, 32, 65, 20, 0.5, "pow2", 7), (8, 16, 4, 81, 13, 1.5, "fib", 0),
    (1, 1, 1, 500, 207, 1.0, "fib", 15), (1, 2, 1, 450, 208, 0.93, "fib", 15), (1, 1, 1, 700, 431, 1.1, "pow2", 10),
]


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16], ids=["f32", "bf16"])
@pytest.mark.parametrize("case", CASES, ids=[f"B{c[0]}H{c[1]}kv{c[2]}T{c[3]}W{c[4]}{c[6]}{c[7]}" for c in CASES])
def test_forward_and_backward(case, dtype):
    B, H, Hkv, T, W, alpha, base, K = case
    q, k, v = inputs.qkv(B, H, T, seed=7 * T + W, dtype=dtype, Hkv=Hkv)
    g = inputs.dout(B, H, T, seed=7 * T + W + 1, dtype=dtype)
    v = (v * 0.5).to(dtype)
    f = fa.base(base, K)
    qc, kc, vc, gc = (x.cuda() for x in (q, k, v, g))
    out, lse = fa.fwd(qc, kc, vc, alpha, f, W, kernel="gather")
    dq, dk, dv, dth, dd = fa.bwd(qc, kc, vc, lse, gc, alpha, f, W, kernel="gather")
    nq, nk, nv, _, _ = fa.bwd(qc, kc, vc, lse, gc, alpha, f, W, kernel="gather", rung_grads=False)
    torch.cuda.synchronize()
    for x, y in ((dq, nq), (dk, nk), (dv, nv)):
        assert torch.equal(x, y)
    n64 = [x.double().numpy() for x in (q, k, v, g)]
    d = O.offsets_fp32(float(np.float32(alpha)), f.astype(np.float64))
    ro, rl = O.forward(*n64[:3], W, d, nthreads=8)
    rq, rk, rv, rdd = O.backward(*n64, W, d, nthreads=8)
    tol, gtol = (1e-4, 1e-4) if dtype == torch.float32 else (1e-2, 3e-2)
    assert np.max(np.abs(out.double().cpu().numpy() - ro)) <= tol
    assert np.max(np.abs(lse.double().cpu().numpy() - rl)) <= tol
    for name, x, r in (("dq", dq, rq), ("dk", dk, rk), ("dv", dv, rv)) + ((("dd", dd, rdd),) if K else ()):
        e = np.max(np.abs(x.double().cpu().numpy() - r)) / max(np.max(np.abs(r)), 1e-2)
        assert e <= gtol, (name, e)


def test_masked_rows_do_not_reach_a_query():
    """An infinite value row, and a NaN one, change only the queries that
    attend them: with W = 2 and one rung at distance 20, row 0 and row 40 are
    read by queries 0..2 and 20, and 40..42 and 60."""
    T = 100
    q, k, v = (x.cuda() for x in inputs.qkv(1, 1, T, seed=5))
    f = np.array([20.0], dtype=np.float32)
    ref, _ = fa.fwd(q, k, v, 1.0, f, 2)
    v[0, 0, 0] = float("inf")
    v[0, 0, 40] = float("nan")
    out, _ = fa.fwd(q, k, v, 1.0, f, 2)
    hit = torch.zeros(T, dtype=torch.bool)
    hit[[0, 1, 2, 20, 40, 41, 42, 60]] = True
    assert torch.equal(out[0, 0, ~hit], ref[0, 0, ~hit])
    assert not torch.isfinite(out[0, 0, hit]).any()
