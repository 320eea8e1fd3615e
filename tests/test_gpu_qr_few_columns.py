"""QR of few columns: 1 to 8 columns, and tails of 1 to 8 columns behind whole panels, on either
side of a CTA's row groups (512 threads over the columns); and one column takes no longer than four
(a serial sum over its 512 row groups once took longer than everything else).  Bars as in
test_gpu_qr_blocked: orthogonality 1e-13 N, reconstruction 1e-14 max|Y| N, N >= 16 in them."""
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


@pytest.mark.parametrize("k", [1, 2, 3, 4, 5, 6, 7, 8, 9, 11, 15, 20])
@pytest.mark.parametrize("N", [20, 511, 512, 8200, 100003])
def test_shapes(ctm, N, k):
    Y = np.random.default_rng(N + k).standard_normal((N, k)) * np.logspace(0, -6, k)
    f64 = dict(dtype=torch.float64, device="cuda")
    Q, R = torch.full((N, k), float("nan"), **f64), torch.full((k, k), float("nan"), **f64)
    ws = torch.empty(ctm.ctm_qr_workspace_bytes(N, k), dtype=torch.uint8, device="cuda")
    ctm.ctm_qr(torch.from_numpy(Y).cuda(), N, k, Q, R, ws)
    torch.cuda.synchronize()
    assert int(ws[:4].view(torch.int32).item()) == 0
    q, r = Q.cpu().numpy(), R.cpu().numpy()
    assert np.max(np.abs(q.T @ q - np.eye(k))) < 1e-13 * N
    assert np.max(np.abs(np.tril(r, -1)), initial=0.0) == 0.0
    assert np.all(np.diag(r) >= 0)
    assert np.max(np.abs(q @ r - Y)) <= 1e-14 * np.abs(Y).max() * N


def test_one_column_is_no_slower_than_four(ctm):
    def us(N, k):
        f64 = dict(dtype=torch.float64, device="cuda")
        Y, Q, R = torch.randn((N, k), **f64), torch.empty((N, k), **f64), torch.empty((k, k), **f64)
        ws = torch.empty(ctm.ctm_qr_workspace_bytes(N, k), dtype=torch.uint8, device="cuda")
        s = torch.cuda.Stream()
        ctm.ctm_qr(Y, N, k, Q, R, ws, stream=s)
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            for _ in range(20):
                ctm.ctm_qr(Y, N, k, Q, R, ws, stream=s)
        best = 1e9
        for _ in range(10):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            torch.cuda.synchronize()
            a.record()
            g.replay()
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b) / 20 * 1e3)
        return best

    one, four = us(1000, 1), us(1000, 4)
    print(f"1000 x 1: {one:.1f} us, 1000 x 4: {four:.1f} us")
    assert one < four
