"""Jacobi SVD (ctm_svd) over the sizes of its two-kernel form: one pair, odd
and even k, whole and partial 16-entry lanes, every cluster size, the last k
it takes (256) and the first beyond (257).  Bars as in test_gpu_kernels:
reconstruction 1e-14 k max, V 1e-13 k, U 1e-12 k of orthonormal; singular
values against LAPACK to 1e-12 relative plus 1e-14 k s_0."""
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


def svd(ctm, G, shift=0):
    k = G.shape[0]
    U = torch.empty((k, k), dtype=torch.float64, device="cuda")
    V = torch.empty((k, k), dtype=torch.float64, device="cuda")
    S = torch.empty(k, dtype=torch.float64, device="cuda")
    ws = torch.full((ctm.ctm_svd_workspace_bytes(k) + shift,), 0xFF, dtype=torch.uint8, device="cuda")[shift:]
    ctm.ctm_svd(torch.from_numpy(np.ascontiguousarray(G)).cuda(), k, U, S, V, ws)
    torch.cuda.synchronize()
    return U.cpu().numpy(), S.cpu().numpy(), V.cpu().numpy(), int(ws[:4].view(torch.int32).item())


def check(G, U, S, V):
    k = G.shape[0]
    n = max(k, 4)
    sref = np.linalg.svd(G, compute_uv=False)
    assert np.all(np.diff(S) <= 0)
    assert np.all(np.abs(S - sref) < 1e-12 * sref + 1e-14 * n * sref[0])
    assert np.max(np.abs((U * S) @ V.T - G)) < 1e-14 * n * sref[0]
    assert np.max(np.abs(V.T @ V - np.eye(k))) < 1e-13 * n
    assert np.max(np.abs(U.T @ U - np.eye(k))) < 1e-12 * n


@pytest.mark.parametrize("k", [1, 2, 3, 4, 7, 16, 17, 31, 32, 33, 48, 63, 81, 128, 143, 160, 193, 255, 256, 257])
def test_svd_sizes(ctm, k):
    rng = np.random.default_rng(k)
    G = rng.standard_normal((k, k)) * np.logspace(0, -12, k)[None, :]
    U, S, V, st = svd(ctm, G)
    assert st == 0
    check(G, U, S, V)


@pytest.mark.parametrize("k", [20, 81, 144])
def test_svd_scales_exactly(ctm, k):
    """G and 2^e G take the same rotations: U and V equal bit for bit, S
    scaled exactly; a workspace at an 8-byte boundary gives the same."""
    rng = np.random.default_rng(1000 + k)
    G = np.tril(rng.standard_normal((k, k))) * np.logspace(0, -9, k)[:, None]
    U, S, V, _ = svd(ctm, G)
    check(G, U, S, V)
    for e in (-300, 300):
        U2, S2, V2, _ = svd(ctm, np.ldexp(G, e), shift=8)
        np.testing.assert_array_equal(U2, U)
        np.testing.assert_array_equal(V2, V)
        np.testing.assert_array_equal(S2, np.ldexp(S, e))


def test_svd_zero_columns_and_ties(ctm):
    """Zero columns stay unrotated (U zero there), equal norms rotate by 45 degrees."""
    k = 24
    G = np.zeros((k, k))
    U, S, V, st = svd(ctm, G)
    assert st == 0 and np.all(S == 0) and np.all(U == 0)
    np.testing.assert_array_equal(np.sort(V, axis=None), np.sort(np.eye(k), axis=None))
    G = np.eye(k) + np.ones((k, k)) / 8
    U, S, V, st = svd(ctm, G)
    assert st == 0
    check(G, U, S, V)
