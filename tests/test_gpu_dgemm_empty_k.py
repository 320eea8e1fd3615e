"""An FP64 product over an empty K is C = beta C: bit for bit, no read of C where beta = 0."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("tA,tB", [(0, 0), (1, 1)])
@pytest.mark.parametrize("M,N", [(1, 1), (33, 7), (300, 73)])
@pytest.mark.parametrize("beta", [0.0, 1.0, -3.0])
def test_empty_k(M, N, tA, tB, beta):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2112_13184_gb300 import ctm
    C0 = np.random.default_rng(M).integers(-1000, 1001, size=(M, N + 3)).astype(np.float64)
    want = C0.copy()
    want[:, :N] *= beta
    if beta == 0.0:
        C0[:, :N] = np.nan
        want[:, :N] = 0.0
    C = torch.from_numpy(C0).cuda()
    a = torch.zeros(max(M, N), dtype=torch.float64, device="cuda")
    ctm.ctm_dgemm(tA, tB, M, N, 0, 2.0, a, max(M, 1), a, max(N, 1), beta, C, N + 3)
    torch.cuda.synchronize()
    np.testing.assert_array_equal(C.cpu().numpy(), want)
