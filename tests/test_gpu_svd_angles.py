"""Rotation angles of the Jacobi SVD to the precision of its dot products.

Columns of norms 1 to 1e-3 in disjoint pairs with a cosine of 1.5e-8, all others orthogonal: one
sweep rotates each pair once, and the next finds nothing above its tolerance (3.1e-15).  An angle
with FP32's relative error leaves cosines of 5.6e-16 in root mean square, below the tolerance and
thus in U for good.  Bar for the pairs: 2^-52.  With exact angles what is left is the rounding of the
dot product (48 terms of ~1/48, 2^-53 each, random in sign: below 2^-53 / sqrt(48) per addition, a
dozen additions) and of the entries (2^-53 / sqrt(48) for each of three operations): below 0.6e-16,
a quarter of the bar."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("seed", range(4))
def test_cosines_of_u(seed):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2112_13184_gb300 import ctm
    k = 48
    rng = np.random.default_rng(seed)
    q = np.linalg.qr(rng.standard_normal((k, k)))[0]
    i = np.arange(0, k, 2)
    e = np.zeros((k, k))
    e[i, i + 1] = 1.5e-8 * rng.choice((-1.0, 1.0), k // 2)
    G = (q + q @ e) * np.logspace(0, -3, k)
    f64 = dict(dtype=torch.float64, device="cuda")
    U, S, V = torch.empty((k, k), **f64), torch.empty(k, **f64), torch.empty((k, k), **f64)
    ws = torch.empty(ctm.ctm_svd_workspace_bytes(k), dtype=torch.uint8, device="cuda")
    ctm.ctm_svd(torch.from_numpy(np.ascontiguousarray(G)).cuda(), k, U, S, V, ws)
    torch.cuda.synchronize()
    u = U.cpu().numpy().astype(np.longdouble)  # descending norms: the columns in their order
    u /= np.sqrt((u * u).sum(axis=0))
    c = (u[:, i] * u[:, i + 1]).sum(axis=0).astype(np.float64)
    assert np.sqrt(np.mean(c * c)) < 2.0**-52
