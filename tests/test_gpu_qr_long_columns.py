"""QR of up to eight very long columns, on either side of the panel widths 8, 4, 2 and 1 that let the
row slabs fit in shared memory, and beyond (a column at a time): no wide step in time between the
last two of them.  Bars: orthogonality and column residual sqrt(N) 2^-52, twice the rounding
of sums of N terms of random sign."""
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


def setup(ctm, Y):
    N, k = Y.shape
    f64 = dict(dtype=torch.float64, device="cuda")
    Q, R = torch.full((N, k), float("nan"), **f64), torch.full((k, k), float("nan"), **f64)
    ws = torch.empty(ctm.ctm_qr_workspace_bytes(N, k), dtype=torch.uint8, device="cuda")
    return Q, R, ws


@pytest.mark.parametrize("N,k", [(400000, 1), (420000, 1), (1900000, 1), (2200000, 1), (900000, 2), (1200000, 2),
                                 (300000, 3), (640000, 3), (950000, 3), (300000, 4), (480000, 4), (700000, 4), (380000, 5),
                                 (315000, 6), (270000, 7), (231000, 8), (236000, 8), (360000, 8), (440000, 8), (500000, 8)])
def test_shapes(ctm, N, k):
    Y = np.random.default_rng(N + k).standard_normal((N, k)) * np.logspace(0, -6, k)
    Q, R, ws = setup(ctm, Y)
    ctm.ctm_qr(torch.from_numpy(Y).cuda(), N, k, Q, R, ws)
    torch.cuda.synchronize()
    q, r = Q.cpu().numpy(), R.cpu().numpy()
    bar = np.sqrt(N) * 2.0**-52
    assert np.max(np.abs(q.T @ q - np.eye(k))) < bar
    assert np.max(np.abs(np.tril(r, -1)), initial=0.0) == 0.0
    assert np.all(np.diag(r) >= 0)
    assert np.max(np.linalg.norm(q @ r - Y, axis=0) / np.linalg.norm(Y, axis=0)) < bar


@pytest.mark.parametrize("k,N", [(1, 1900000), (4, 480000), (8, 236000)])
def test_time_grows_with_the_rows(ctm, k, N):
    def us(n):
        Y = torch.randn((n, k), dtype=torch.float64, device="cuda")
        Q, R, ws = setup(ctm, Y)
        best = 1e9
        for _ in range(8):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            torch.cuda.synchronize()
            a.record()
            for _ in range(5):
                ctm.ctm_qr(Y, n, k, Q, R, ws)
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b) / 5 * 1e3)
        return best

    whole, third = us(N), us(N // 3)
    print(f"{N} x {k}: {whole:.0f} us, a third of the rows: {third:.0f} us")
    assert whole < 10 * third
