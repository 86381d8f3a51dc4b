"""Host threads that call at the same time, each on its own stream, with windows
and alphas whose kernels take other amounts of shared memory: the limit of it
belongs to a kernel, and a thread that lowered it had another's launch refused
(seen within some thousand calls of two threads, fp32, W 2 and 100)."""
from __future__ import annotations

import threading

import pytest
import torch

import paper_2606_28560_gb300 as fa

F = fa.base("fib", 15)
CALLS = 1500


def _work(dtype, W, alpha, seed, start, result):
    try:
        g = torch.Generator(device="cuda").manual_seed(seed)
        q, k, v, do = (torch.randn(1, 2, 300, 64, generator=g, device="cuda").to(dtype) for _ in range(4))
        bufs = dict(workspace=torch.empty(1 << 22, dtype=torch.uint8, device="cuda"))
        want = None
        with torch.cuda.stream(torch.cuda.Stream()):
            torch.cuda.synchronize()
            start.wait()
            for _ in range(CALLS):
                out, lse = fa.fwd(q, k, v, alpha, F, W, **bufs)
                if want is None:
                    want = (out,) + fa.bwd(q, k, v, lse, do, alpha, F, W, out=out)
            got = (out,) + fa.bwd(q, k, v, lse, do, alpha, F, W, out=out)
            torch.cuda.current_stream().synchronize()
        assert all(torch.equal(a, b) for a, b in zip(want, got))
    except Exception as e:                        # (handed to the test's thread)
        result.append(e)


@pytest.mark.gpu
@pytest.mark.parametrize("dtype,calls", [(torch.float32, [(2, 1.5), (100, 0.5), (8, 1.0), (200, 1.2)]),
                                         (torch.bfloat16, [(8, 1.5), (7, 0.5), (16, 1.0), (9, 0.6)])],
                         ids=["gather", "mma"])
def test_threads_with_other_windows(dtype, calls):
    start, result = threading.Barrier(len(calls)), []
    threads = [threading.Thread(target=_work, args=(dtype, W, alpha, i, start, result))
               for i, (W, alpha) in enumerate(calls)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not result, result
