"""ctm_permute where the source is already in destination order (identities, axes of one element
moved): a copy of any size, nothing written beyond it."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,perm", [
    ((1,), (0,)), ((255,), (0,)), ((2**18 - 1,), (0,)), ((2**18,), (0,)), ((2**18 + 1, 1), (1, 0)), ((1000003,), (0,)),
    ((1, 700, 1, 611), (2, 1, 0, 3)), ((33, 1, 129, 77, 1), (4, 0, 2, 1, 3)), ((2,) * 8, tuple(range(8))),
    ((9,) * 7, tuple(range(7))),
])
def test_in_order(dims, perm):
    from paper_2112_13184_gb300 import ctm
    n = int(np.prod(dims))
    x = torch.arange(n, dtype=torch.float64, device="cuda") + 0.5
    out = torch.full((n + 2,), -1.0, dtype=torch.float64, device="cuda")
    ctm.ctm_permute(x, out[1:-1], dims, perm)
    torch.cuda.synchronize()
    assert out[0] == -1.0 and out[-1] == -1.0
    assert torch.equal(out[1:-1], x)
