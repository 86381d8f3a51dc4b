"""A flag without a truth value is refused before anything is launched, with
the error of the value itself."""
from __future__ import annotations

import pytest
import torch

import paper_2606_28560_gb300 as fa

F = fa.base("fib", 15)


@pytest.mark.parametrize("device", ["cpu", pytest.param("cuda", marks=pytest.mark.gpu)])
@pytest.mark.parametrize("flag", ["dedup", "round_offsets", "rung_grads"])
def test_flag_without_a_truth_value(flag, device):
    q = torch.zeros(1, 2, 40, 64, device=device)
    kw = {flag: torch.tensor([1, 0])}
    with pytest.raises(RuntimeError, match="Boolean value of Tensor"):
        fa.bwd(q, q, q, torch.zeros(1, 2, 40, device=device), q, 0.9, F, 8, **kw)
    if flag != "rung_grads":
        with pytest.raises(RuntimeError, match="Boolean value of Tensor"):
            fa.fwd(q, q, q, 0.9, F, 8, **kw)
