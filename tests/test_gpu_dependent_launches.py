"""Chains of kernels without a synchronisation in between, on a stream and in a graph, give
the bits of the same calls synchronised one by one: each kernel reads what the one before
wrote, and overwrites what the one before that read."""
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def ctm():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2112_13184_gb300 import ctm as m
    return m


def chain(ctm, x, n, steps, sync, stream=None):
    """x (n x n) through transposes, FP64 and emulated products and back into x."""
    y, z = torch.empty_like(x), torch.empty_like(x)
    ws = torch.zeros(ctm.ctm_gemm_ozaki_workspace_bytes(n, n, n, 5), dtype=torch.uint8, device="cuda")
    s = stream
    after = torch.cuda.synchronize if sync else (lambda: None)
    calls = [lambda: ctm.ctm_permute(x, y, (n, n), (1, 0), stream=s),
             lambda: ctm.ctm_dgemm(0, 1, n, n, n, 1.0 / n, x, n, y, n, 0.0, z, n, stream=s),
             lambda: ctm.ctm_gemm_ozaki(1, 0, n, n, n, 1.0 / n, z, n, y, n, 0.0, x, n, 5, ws, stream=s),
             lambda: ctm.ctm_permute(x, z, (n, n), (1, 0), stream=s),
             lambda: ctm.ctm_gemm_ozaki(0, 1, n, n, n, 1.0 / n, z, n, y, n, 0.5, x, n, 5, ws, stream=s)]

    def run():
        for _ in range(steps):
            for c in calls:
                c()
                after()
    return run, (y, z, ws)


@pytest.mark.parametrize("n,steps", [(7, 40), (64, 40), (200, 20), (520, 10), (1536, 3)])
def test_chain_bits(ctm, n, steps):
    g = torch.Generator(device="cuda").manual_seed(n)
    x0 = torch.randn(n, n, dtype=torch.float64, device="cuda", generator=g)
    x = x0.clone()
    run, _ = chain(ctm, x, n, steps, sync=True)
    run()
    torch.cuda.synchronize()
    want = x.clone()
    for _ in range(3):
        x = x0.clone()
        run, _keep = chain(ctm, x, n, steps, sync=False)
        torch.cuda.synchronize()
        run()
        torch.cuda.synchronize()
        assert torch.equal(x, want)


@pytest.mark.parametrize("n", [64, 520])
def test_chain_bits_in_a_graph(ctm, n):
    g = torch.Generator(device="cuda").manual_seed(n)
    x0 = torch.randn(n, n, dtype=torch.float64, device="cuda", generator=g)
    x = x0.clone()
    run, _ = chain(ctm, x, n, 4, sync=True)
    run()
    torch.cuda.synchronize()
    want = x.clone()
    x.copy_(x0)
    s = torch.cuda.Stream()
    run, _keep = chain(ctm, x, n, 4, sync=False, stream=s)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=s):
        run()
    torch.cuda.synchronize()
    for _ in range(2):
        x.copy_(x0)
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(x, want)
