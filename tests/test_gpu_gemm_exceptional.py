"""Emulated products outside the normal range, in the short (K <= 256), the long and the split form:
rows and columns with an infinity or a NaN give NaN throughout, results beyond FP64 an infinity of
their sign, results below its normal range the subnormal number (rounded once: within one spacing of
2^-1074), zero rows and columns zero -- and none of it touches the other entries.  Integer operands
times powers of two for each row and column: every other result is exact."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("M,N,K", [(300, 21, 40), (300, 64, 256), (16000, 40, 300), (16000, 37, 700), (100, 21, 4100)])
@pytest.mark.parametrize("slices", [3, 5])
def test_exceptional_entries(M, N, K, slices):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2112_13184_gb300 import ctm
    rng = np.random.default_rng(M + N + K)
    A = rng.integers(-127, 128, size=(M, K)).astype(np.float64)
    B = rng.integers(-127, 128, size=(K, N)).astype(np.float64)
    ra, cb = np.zeros(M, dtype=int), np.zeros(N, dtype=int)
    A[2] = 0.0
    B[:, 3] = 0.0
    ra[3::40], ra[4::40], ra[5::40], ra[6::40] = 990, -990, 400, -500
    cb[0], cb[1], cb[4], cb[7] = 100, -70, -90, -400
    with np.errstate(over="ignore", under="ignore", invalid="ignore"):
        want = np.ldexp(A @ B, ra[:, None] + cb[None, :])  # C's ldexp rounds once
    A, B = np.ldexp(A, ra[:, None]), np.ldexp(B, cb[None, :])
    A[0, K // 2], A[1, K - 1], A[M - 1, 0] = np.inf, np.nan, -np.inf
    B[K // 3, 2], B[0, N - 1] = np.nan, np.inf
    for r in (0, 1, M - 1):
        want[r] = np.nan
    for c in (2, N - 1):
        want[:, c] = np.nan
    assert np.isinf(want).any() and ((want != 0) & (np.abs(want) < 2.0**-1022)).any()
    C = torch.full((M, N), 7.0, dtype=torch.float64, device="cuda")
    ws = torch.zeros(ctm.ctm_gemm_ozaki_workspace_bytes(M, N, K, slices), dtype=torch.uint8, device="cuda")
    ctm.ctm_gemm_ozaki(0, 0, M, N, K, 1.0, torch.from_numpy(A).cuda(), K, torch.from_numpy(B).cuda(), N, 0.0, C, N, slices,
                       ws)
    torch.cuda.synchronize()
    assert int(ws[:4].view(torch.int32).item()) == 0
    got = C.cpu().numpy()
    normal = ~(np.abs(want) < 2.0**-1022)  # NaN and infinities among them
    np.testing.assert_array_equal(got[normal], want[normal])
    assert np.max(np.abs(got[~normal] - want[~normal]), initial=0.0) <= 2.0**-1074
