"""Whatever float() takes is a number to the compute calls (alpha, rope_base,
scale): a call with host tensors gets as far as the check of their device."""
from __future__ import annotations

import numpy as np
import pytest
import torch

import paper_2606_28560_gb300 as fa

F = fa.base("fib", 15)


@pytest.mark.parametrize("number", ["0.9", np.float32(0.9), torch.tensor(0.9), np.array(0.9), 1],
                         ids=["text", "numpy", "tensor", "array", "int"])
@pytest.mark.parametrize("name", ["alpha", "rope_base", "scale"])
def test_numbers(name, number):
    q = torch.zeros(1, 2, 40, 64)
    kw = {"alpha": 0.9, name: number}
    alpha = kw.pop("alpha")
    with pytest.raises(ValueError, match="contiguous CUDA"):
        fa.fwd(q, q, q, alpha, F, 8, **kw)
    with pytest.raises(ValueError, match="contiguous CUDA"):
        fa.bwd(q, q, q, torch.zeros(1, 2, 40), q, alpha, F, 8, **kw)


def test_no_number():
    q = torch.zeros(1, 2, 40, 64)
    for bad, error in (("x", ValueError), (None, TypeError), ([0.9], TypeError)):
        with pytest.raises(error, match="float"):
            fa.fwd(q, q, q, bad, F, 8)
