"""QR of matrices with one entry in each column, in rows 0 to k-1: the reflectors' norm, beta and tau
are then exact in correctly rounded arithmetic (sqrt(fl(y^2)) = |y|, tau = 2), so that R is
diag(|y|) and Q the signed identity bit for bit, over mantissas and exponents (also where y^2 is
close to the ends of the FP64 range)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("N,k", [(1, 1), (64, 64), (500, 8), (1000, 144), (20000, 100)])
def test_diagonal(N, k):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2112_13184_gb300 import ctm
    for seed in range(4):
        rng = np.random.default_rng(1000 * seed + k)
        y = rng.uniform(1.0, 2.0, k) * rng.choice((-1.0, 1.0), k)
        y = np.ldexp(y, rng.integers(-500, 501, k) if seed & 1 else rng.integers(-20, 21, k))
        Y = np.zeros((N, k))
        Y[np.arange(k), np.arange(k)] = y
        Q = torch.empty((N, k), dtype=torch.float64, device="cuda")
        R = torch.empty((k, k), dtype=torch.float64, device="cuda")
        ws = torch.empty(ctm.ctm_qr_workspace_bytes(N, k), dtype=torch.uint8, device="cuda")
        ctm.ctm_qr(torch.from_numpy(Y).cuda(), N, k, Q, R, ws)
        torch.cuda.synchronize()
        np.testing.assert_array_equal(R.cpu().numpy(), np.diag(np.abs(y)))
        np.testing.assert_array_equal(Q.cpu().numpy(), np.sign(Y))
