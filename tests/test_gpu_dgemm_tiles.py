"""FP64 GEMM over the tiles its plan picks: widths from 1 to 73 (every tile
width and its padding), one to five row tiles, K around the 16-wide step,
outputs at a row stride, alpha and beta.  Integer operands: every product
and sum is exact, so the result must equal numpy's bit for bit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def ctm():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2112_13184_gb300 import ctm as m
    return m


SHAPES = [(33, n, 17) for n in (1, 7, 8, 9, 16, 24, 31, 40, 48, 56, 57, 64, 72, 73)]
SHAPES += [(1, 1, 300), (31, 36, 36), (5000, 36, 72), (5000, 72, 36), (129, 144, 144), (20000, 40, 16), (513, 200, 1),
           (16, 1, 70000), (17, 1, 70000), (300, 300, 300)]


@pytest.mark.parametrize("tA,tB", [(0, 0), (1, 0), (0, 1), (1, 1)])
@pytest.mark.parametrize("M,N,K", SHAPES)
def test_exact(ctm, M, N, K, tA, tB):
    rng = np.random.default_rng(M + N + K)
    A = rng.integers(-1000, 1001, size=(K, M) if tA else (M, K)).astype(np.float64)
    B = rng.integers(-1000, 1001, size=(N, K) if tB else (K, N)).astype(np.float64)
    C0 = rng.integers(-1000, 1001, size=(M, N + 3)).astype(np.float64)
    ref = C0.copy()
    ref[:, :N] = 2.0 * ((A.T if tA else A) @ (B.T if tB else B)) - 3.0 * C0[:, :N]
    C = torch.from_numpy(C0).cuda()
    ctm.ctm_dgemm(tA, tB, M, N, K, 2.0, torch.from_numpy(A).cuda(), A.shape[1], torch.from_numpy(B).cuda(), B.shape[1],
                  -3.0, C, N + 3)
    torch.cuda.synchronize()
    np.testing.assert_array_equal(C.cpu().numpy(), ref)
