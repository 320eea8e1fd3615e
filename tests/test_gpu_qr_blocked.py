"""Blocked Householder QR (ctm_qr) at the edges of its panels and forms.

Shapes: k around multiples of the 8-column panel, one column, square
matrices, row counts on either side of the cluster / grid rule and of whole
rows per CTA, more than 512 columns (two column passes), columns that are
zero or repeated (their reflector is the identity or rounding noise: Q stays
orthonormal all the same).  The bars are those of test_gpu_kernels.test_qr:
orthogonality 1e-13 N, reconstruction 1e-14 max|Y| N, with N >= 16 in them so
that one-row cases keep a few units of rounding."""
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


def qr(ctm, Y):
    N, k = Y.shape
    Q = torch.full((N, k), float("nan"), dtype=torch.float64, device="cuda")
    R = torch.full((k, k), float("nan"), dtype=torch.float64, device="cuda")
    ws = torch.full((ctm.ctm_qr_workspace_bytes(N, k),), 0xFF, dtype=torch.uint8, device="cuda")
    ctm.ctm_qr(torch.from_numpy(Y).cuda(), N, k, Q, R, ws)
    torch.cuda.synchronize()
    assert int(ws[:4].view(torch.int32).item()) == 0
    return Q.cpu().numpy(), R.cpu().numpy()


def check(Y, Q, R):
    N, k = Y.shape
    n = max(N, 16)
    assert np.max(np.abs(Q.T @ Q - np.eye(k))) < 1e-13 * n
    assert np.max(np.abs(np.tril(R, -1)), initial=0.0) == 0.0
    assert np.all(np.diag(R) >= 0)
    assert np.max(np.abs(Q @ R - Y)) <= 1e-14 * np.abs(Y).max() * n


@pytest.mark.parametrize("N,k", [(1, 1), (2, 1), (5, 5), (8, 8), (9, 9), (33, 1), (32, 32), (31, 7), (130, 8),
                                 (129, 17), (255, 144), (512, 40), (1024, 36), (1024, 72), (1031, 81), (2592, 81),
                                 (600, 520), (8192, 144), (9001, 130), (40000, 8), (200000, 3)])
def test_qr_shapes(ctm, N, k):
    rng = np.random.default_rng(N + 3 * k)
    Y = rng.standard_normal((N, k)) * np.logspace(0, -12, k)[None, :]
    Q, R = qr(ctm, Y)
    check(Y, Q, R)
    Q2, R2 = qr(ctm, Y)  # fixed summation order: a rerun gives the same bits
    np.testing.assert_array_equal(Q, Q2)
    np.testing.assert_array_equal(R, R2)


@pytest.mark.parametrize("N,k", [(40, 20), (700, 33), (3000, 48)])
def test_qr_zero_and_repeated_columns(ctm, N, k):
    rng = np.random.default_rng(k)
    Y = rng.standard_normal((N, k))
    Y[:, 0] = 0.0
    Y[:, 9] = 0.0
    Y[:, 12] = Y[:, 3]
    Y[:, k - 1] = 0.0
    Q, R = qr(ctm, Y)
    check(Y, Q, R)
    check(np.zeros((N, k)), *qr(ctm, np.zeros((N, k))))
