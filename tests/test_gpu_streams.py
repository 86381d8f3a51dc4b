"""Calls on a stream other than the current one: what the call allocates stays
the call's while that stream works on it, and what it returns stays the caller's
while the current stream works on it."""
from __future__ import annotations

import pytest
import torch

import paper_2606_28560_gb300 as fa

pytestmark = pytest.mark.gpu
F = fa.base("fib", 15)
HOLD = 20_000_000                                 # cycles that a stream is held back: about 10 ms


def _inputs(dtype, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return [torch.randn(2, 4, 500, 64, generator=g, device="cuda").to(dtype) for _ in range(4)]


def _layer(x, W, stream=None):
    q, k, v, do = x
    out, lse = fa.fwd(q, k, v, 0.9, F, W, stream=stream)
    return (out, lse) + fa.bwd(q, k, v, lse, do, 0.9, F, W, out=out, stream=stream)


@pytest.mark.parametrize("dtype,W", [(torch.bfloat16, 8), (torch.bfloat16, 24), (torch.float32, 8)], ids=["mma", "wide", "f32"])
def test_workspaces_are_the_stream_s(dtype, W):
    x = _inputs(dtype, 1)
    want = _layer(x, W)
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(side):
        torch.cuda._sleep(HOLD)
    got = _layer(x, W, side)
    # the current stream's next allocations, over the sizes the calls used
    junk = [torch.full((n,), float("nan"), device="cuda") for n in [1 << s for s in range(8, 23)] for _ in range(3)]
    torch.cuda.synchronize()
    assert all(torch.equal(a, b) for a, b in zip(want, got))
    del junk


def test_results_are_the_current_stream_s():
    x, y = _inputs(torch.bfloat16, 1), _inputs(torch.bfloat16, 2)
    want = [t.clone() for t in _layer(x, 8)]
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    got = _layer(x, 8, side)
    torch.cuda.current_stream().wait_stream(side)
    torch.cuda._sleep(HOLD)
    copies = [t.clone() for t in got]             # read behind the wait, while
    del got                                       # the caller drops them and
    other = [_layer(y, 8, side) for _ in range(3)]    # the side stream goes on
    torch.cuda.synchronize()
    assert all(torch.equal(a, b) for a, b in zip(want, copies))
    del other


def test_default_stream_by_name():
    """The default stream given explicitly, from under another current stream."""
    x = _inputs(torch.bfloat16, 1)
    want = _layer(x, 8)
    torch.cuda.synchronize()
    with torch.cuda.stream(torch.cuda.Stream()):
        got = _layer(x, 8, torch.cuda.default_stream())
    torch.cuda.synchronize()
    assert all(torch.equal(a, b) for a, b in zip(want, got))
