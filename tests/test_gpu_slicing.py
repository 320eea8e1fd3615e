"""Operand slicing of the emulated-FP64 GEMM at the edges of its kernels.

The slicer of an operand is chosen by its layout and K: rows contiguous in
K held in registers (K <= 8192), longer ones by (row, 1024-wide K range); rows
contiguous across K in one launch (K <= 1536, registers up to 512) or in
two passes.  Integer operands that use the leading digits only must give
numpy's product bit for bit whatever the slicer (every kept slice product is
exact), so one pin per kernel and edge needs no tolerance."""
from fractions import Fraction

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


@pytest.mark.parametrize("M,N,K", [(9, 5, 9001), (3, 33, 8193), (33, 65, 8192), (31, 17, 1536), (65, 3, 1537),
                                   (32, 1, 512), (97, 64, 513), (1, 7, 31), (40, 40, 33), (5, 2, 1), (2000, 9, 40)])
@pytest.mark.parametrize("tA,tB", [(0, 0), (1, 0), (0, 1), (1, 1)])
def test_slicers_exact(ctm, M, N, K, tA, tB):
    rng = np.random.default_rng(M + N + K)
    A = rng.integers(-255, 256, size=(K, M) if tA else (M, K)).astype(np.float64)
    B = rng.integers(-65535, 65536, size=(N, K) if tB else (K, N)).astype(np.float64)
    if tB:
        B[:, 0] = 65535.0
    else:
        B[0, :] = 65535.0
    C = torch.empty((M, N), dtype=torch.float64, device="cuda")
    ws = torch.zeros(ctm.ctm_gemm_ozaki_workspace_bytes(M, N, K, 2), dtype=torch.uint8, device="cuda")
    ctm.ctm_gemm_ozaki(tA, tB, M, N, K, 1.0, torch.from_numpy(A).cuda(), A.shape[1], torch.from_numpy(B).cuda(),
                       B.shape[1], 0.0, C, N, 2, ws)
    torch.cuda.synchronize()
    np.testing.assert_array_equal(C.cpu().numpy(), (A.T if tA else A) @ (B.T if tB else B))


def round_away(x, bits):
    """x rounded to a whole number of 2^-bits, halves away from zero (exact rationals: adding 0.5 in
    floating point would itself round 0.5 (1 - 2^-53) up)."""
    y = abs(Fraction(float(x))) * Fraction(2) ** bits
    n = (2 * y.numerator + y.denominator) // (2 * y.denominator)
    return float(n * Fraction(2) ** -bits) * (-1.0 if x < 0 else 1.0)


@pytest.mark.parametrize("slices", [2, 3, 4, 5, 6])
def test_slices_of_every_magnitude(ctm, slices):
    """Rows spanning 2^-1074 .. 1 (denormals, halves, exact powers of two): times the
    identity, every entry comes back rounded to 8 bits per slice below its row's
    power of two, half away from zero in magnitude."""
    rng = np.random.default_rng(slices)
    M = K = 64
    A = rng.standard_normal((M, K)) * np.exp2(rng.integers(-70, 1, size=(M, K)))
    A[1] = np.exp2(-np.arange(K, dtype=np.float64))
    A[2] = -(1.0 - 2.0 ** -53) * np.exp2(-np.arange(K, dtype=np.float64))
    A[3] *= 2.0 ** -1000
    A[4] = np.float64(5e-324) * rng.integers(-1000, 1000, size=K)
    A[5] = 0.0
    mx = np.abs(A).max(axis=1)
    e = np.where(mx == 0, 0, np.maximum(np.frexp(mx)[1], -1022))
    want = np.array([[round_away(A[i, k], 8 * slices - int(e[i])) for k in range(K)] for i in range(M)])
    C = torch.empty((M, K), dtype=torch.float64, device="cuda")
    ws = torch.zeros(ctm.ctm_gemm_ozaki_workspace_bytes(M, K, K, slices), dtype=torch.uint8, device="cuda")
    ctm.ctm_gemm_ozaki(0, 0, M, K, K, 1.0, torch.from_numpy(A).cuda(), K, torch.eye(K, dtype=torch.float64,
                       device="cuda"), K, 0.0, C, K, slices, ws)
    torch.cuda.synchronize()
    # up to 5 slices the levels >= 2 fit one FP32 accumulator's 24 bits and the product keeps
    # round(2^28 F) below the level-1 unit, 2^-44 of the row's power of two; with 6 their FP32
    # rounding shows (the documented 2^-36)
    tol = 2.0 ** -43 if slices < 6 else 2.0 ** -36
    assert np.all(np.abs(C.cpu().numpy() - want) <= np.ldexp(tol, e)[:, None])


@pytest.mark.parametrize("M,N,K", [(33, 2, 1537), (1, 1, 4096), (65, 3, 4097), (31, 1, 8191), (48, 5, 1200), (640, 1, 511),
                                   (2, 1, 300), (5000, 1, 1536), (40000, 1, 530), (9000, 1, 4090), (1300, 1, 8192)])
def test_column_slicer_clusters(ctm, M, N, K):
    """A read along its rows' contiguous direction: clusters of 2 to 16, one CTA and the long form.  The
    only large entry of a row sits at its last k, so that a CTA without the cluster's maximum goes wrong."""
    rng = np.random.default_rng(M + K)
    A = rng.integers(-1, 2, size=(K, M)).astype(np.float64)
    A[K - 1, :] = 60000.0
    B = rng.integers(-255, 256, size=(K, N)).astype(np.float64)
    C = torch.empty((M, N), dtype=torch.float64, device="cuda")
    ws = torch.zeros(ctm.ctm_gemm_ozaki_workspace_bytes(M, N, K, 2), dtype=torch.uint8, device="cuda")
    ctm.ctm_gemm_ozaki(1, 0, M, N, K, 1.0, torch.from_numpy(A).cuda(), M, torch.from_numpy(B).cuda(), N, 0.0, C, N, 2, ws)
    torch.cuda.synchronize()
    np.testing.assert_array_equal(C.cpu().numpy(), A.T @ B)
