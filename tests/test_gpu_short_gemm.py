"""Single-chunk (K <= 256) and split emulated products at the edges of their
tiles and output paths: K on either side of one chunk and of a 32-wide
k-block, fewer tiles than epilogue teams, more than two rounds of tiles per
SM, widths that leave a partial 8-column block, outputs whose rows or base
rule out 32- or 16-byte stores, every slice count.  Integer operands of one
leading digit: every kept product and sum is exact, the result must equal
numpy's bit for bit, and what lies outside the output must keep its value."""
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


def run(ctm, M, N, K, slices, ldc, shift, alpha=1.0, beta=0.0):
    rng = np.random.default_rng(M + 3 * N + 7 * K + slices)
    A = rng.integers(-127, 128, size=(M, K)).astype(np.float64)
    B = rng.integers(-127, 128, size=(K, N)).astype(np.float64)
    buf = torch.full((M * ldc + shift + 8,), 5.0, dtype=torch.float64, device="cuda")
    C = buf[shift:]
    ws = torch.zeros(ctm.ctm_gemm_ozaki_workspace_bytes(M, N, K, slices), dtype=torch.uint8, device="cuda")
    ctm.ctm_gemm_ozaki(0, 0, M, N, K, alpha, torch.from_numpy(A).cuda(), K, torch.from_numpy(B).cuda(), N, beta, C, ldc,
                       slices, ws)
    torch.cuda.synchronize()
    assert int(ws[:4].view(torch.int32).item()) == 0
    got = buf.cpu().numpy()
    want = np.full_like(got, 5.0)
    view = want[shift:shift + M * ldc].reshape(M, ldc)
    view[:, :N] = alpha * (A @ B) + beta * 5.0
    np.testing.assert_array_equal(got, want)


@pytest.mark.parametrize("M,N,K", [(1, 1, 1), (130, 7, 31), (128, 16, 32), (300, 17, 33), (129, 80, 255), (200, 81, 256),
                                   (500, 36, 72), (45000, 25, 50), (60000, 64, 64), (2600, 1300, 40), (200, 56, 257),
                                   (512, 40, 512), (100, 9, 4100)])
@pytest.mark.parametrize("pad,shift", [(0, 0), (4, 4), (2, 2), (1, 1), (3, 0)])
def test_exact_outputs(ctm, M, N, K, pad, shift):
    run(ctm, M, N, K, 3, N + pad, shift)


@pytest.mark.parametrize("slices", [2, 3, 4, 5, 6])
@pytest.mark.parametrize("M,N,K", [(700, 72, 72), (700, 72, 700)])
def test_slices_alpha_beta(ctm, M, N, K, slices):
    run(ctm, M, N, K, slices, N, 0)
    run(ctm, M, N, K, slices, N + 1, 0, alpha=-2.0, beta=0.5)
