"""ctm_permute, element by element (below 2^18 of them) and box by box: every element lands where the multi-index says, bit for bit.

The cases put axes across box edges: extents one off a power of two, runs shorter
and longer than a box wants, axes of one element, merged neighbours, eight axes,
arrays of one element and arrays smaller than a box, and three cut axes at once.
"""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctm():
    import paper_2112_13184_gb300.ctm as c

    return c


@pytest.mark.parametrize("dims,perm", [
    ((1,), (0,)), ((1, 1, 1), (2, 0, 1)), ((5,), (0,)), ((4097,), (0,)), ((100001, 1), (1, 0)),
    ((31, 33), (1, 0)), ((33, 31), (1, 0)), ((513, 511), (1, 0)), ((2, 70001), (1, 0)), ((70001, 2), (1, 0)),
    ((3, 3000, 5), (2, 1, 0)), ((3, 3000, 5), (1, 0, 2)), ((65, 3, 65), (2, 1, 0)), ((65, 3, 2, 67), (0, 2, 1, 3)),
    ((17, 19, 23, 29), (3, 1, 0, 2)), ((17, 19, 23, 29), (1, 2, 3, 0)), ((17, 19, 23, 29), (2, 3, 0, 1)),
    ((2,) * 8, (7, 6, 5, 4, 3, 2, 1, 0)), ((2, 3) * 4, (6, 4, 2, 0, 7, 5, 3, 1)),
    ((48, 2, 48, 2, 25), (0, 2, 3, 1, 4)), ((48, 9, 8, 8, 64), (1, 0, 3, 2, 4)), ((1, 40, 1, 50, 60), (4, 0, 3, 2, 1)),
    ((511, 513), (1, 0)), ((512, 512), (1, 0)), ((513, 511), (0, 1)), ((2, 140001), (1, 0)), ((140001, 2), (1, 0)),
    ((3, 30000, 5), (2, 1, 0)), ((3, 30000, 5), (1, 0, 2)), ((67, 65, 69), (2, 1, 0)), ((65, 3, 33, 67), (0, 2, 1, 3)),
    ((17, 37, 23, 29), (3, 1, 0, 2)), ((17, 37, 23, 29), (1, 2, 3, 0)), ((17, 37, 23, 29), (2, 3, 0, 1)),
    ((2, 3, 5, 7, 11, 13, 2, 9), (7, 6, 5, 4, 3, 2, 1, 0)), ((5, 6) * 4, (6, 4, 2, 0, 7, 5, 3, 1)),
    ((48, 5, 48, 5, 25), (0, 2, 3, 1, 4)), ((1, 90, 1, 70, 60), (4, 0, 3, 2, 1)),
    ((600, 7, 600), (2, 1, 0)), ((257, 129, 65), (2, 0, 1)),
])
def test_permute_boxes_exact(ctm, dims, perm):
    n = int(np.prod(dims))
    x = torch.arange(n, dtype=torch.float64, device="cuda") + 0.5
    out = torch.full((n + 2,), -1.0, dtype=torch.float64, device="cuda")
    ctm.ctm_permute(x, out[1:-1], dims, perm)
    torch.cuda.synchronize()
    assert out[0] == -1.0 and out[-1] == -1.0
    want = x.cpu().numpy().reshape(dims).transpose(perm)
    np.testing.assert_array_equal(out[1:-1].cpu().numpy().reshape(want.shape), want)
