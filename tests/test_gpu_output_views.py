"""Emulated products written through a column view: row-major, columns split over two axes, and
views whose offsets the epilogue cannot hold (in reverse, 2^32 elements apart), which are refused
without a launch -- short and long K, tiles that end inside an 8-column block, alpha and beta; the
split products (few tiles, K > 256) take them in 64 bits.  The library's internal entry points are called by
name: the public calls write row-major outputs only.  Integer operands: the result is exact, what
lies outside the output keeps its value."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


class OzView(ctypes.Structure):
    _fields_ = [("n", ctypes.c_int), ("dim", ctypes.c_int * 4), ("stride", ctypes.c_longlong * 4)]


def view(*axes):  # (extent, stride), innermost last
    pad = 4 - len(axes)
    return OzView(len(axes), (ctypes.c_int * 4)(*[a[0] for a in axes], *[1] * pad),
                  (ctypes.c_longlong * 4)(*[a[1] for a in axes], *[0] * pad))


@pytest.mark.parametrize("M,N,K", [(130, 24, 40), (300, 21, 40), (16000, 24, 300), (130, 90, 300), (64, 32, 4100)])
@pytest.mark.parametrize("alpha,beta", [(1.0, 0.0), (-2.0, 0.5)])
@pytest.mark.parametrize("kind", ["plain", "reversed", "far apart", "two axes"])
def test_column_views(M, N, K, alpha, beta, kind):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2112_13184_gb300 import ctm
    if kind == "two axes" and N % 3:
        pytest.skip("needs N in threes")
    lib = ctypes.CDLL(ctm._lib._name)
    split = getattr(lib, "_ZN3ctm13oz_split_viewEPKdiiRKNS_6OzViewES4_iPvP11CUstream_st")
    gemm = getattr(lib, "_ZN3ctm12oz_gemm_viewEiiiiPKvS1_ddPdRKNS_6OzViewES5_PvmPiP11CUstream_sti")
    P, s = ctypes.c_void_p, 3
    rng = np.random.default_rng(M + N + K)
    A = rng.integers(-127, 128, size=(M, K)).astype(np.float64)
    B = rng.integers(-127, 128, size=(N, K)).astype(np.float64)
    dA, dB = torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda()
    whole = ctm.ctm_gemm_ozaki_workspace_bytes(M, N, K, s)
    sa, sb, ws = (torch.zeros(whole, dtype=torch.uint8, device="cuda") for _ in range(3))
    err = torch.zeros(1, dtype=torch.int32, device="cuda")
    buf = torch.full((M * N + 16,), 5.0, dtype=torch.float64, device="cuda")
    base = buf.data_ptr() + 8 * 8
    n = np.arange(N)
    if kind == "plain":
        cols, off = view((N, 1)), n
    elif kind == "reversed":
        cols, off, base = view((N, -1)), -n, base + 8 * (N - 1)
    elif kind == "far apart":
        cols, off = view((N // 2, 2**31), (2, 1)), None
    else:  # column (a, b) of 3 x N/3 at b 3 + a
        cols, off = view((3, 1), (N // 3, 3)), n // (N // 3) + 3 * (n % (N // 3))
    for X, R, out in ((dA, M, sa), (dB, N, sb)):
        assert split(P(X.data_ptr()), R, K, ctypes.byref(view((R, K))), ctypes.byref(view((K, 1))), s, P(out.data_ptr()),
                     P(0)) == 0
    split_k = K > 256 and M < 1000  # few tiles and more than one chunk of K
    if off is None and split_k:
        pytest.skip("not held by the buffer")
    st = gemm(M, N, K, s, P(sa.data_ptr()), P(sb.data_ptr()), ctypes.c_double(alpha), ctypes.c_double(beta), P(base),
              ctypes.byref(view((M, N))), ctypes.byref(cols), P(ws.data_ptr()), ctypes.c_size_t(whole), P(err.data_ptr()),
              P(0), 0)
    if kind in ("reversed", "far apart") and not split_k:
        assert st == 1  # cudaErrorInvalidValue
        torch.cuda.synchronize()
        assert bool((buf == 5.0).all())
        return
    assert st == 0
    torch.cuda.synchronize()
    assert int(err.item()) == 0
    want = np.full(M * N + 16, 5.0)
    first = (base - buf.data_ptr()) // 8
    at = first + N * np.arange(M)[:, None] + off[None, :]
    want[at] = alpha * (A @ B.T) + beta * 5.0
    np.testing.assert_array_equal(buf.cpu().numpy(), want)
