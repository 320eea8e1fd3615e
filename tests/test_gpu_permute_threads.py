"""ctm_permute from several host threads at once, each with boxes of another size (49.2 to 52.4 KB of
shared memory): every call is accepted and every element lands where the multi-index says."""
import threading

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

CASES = [((44, 18, 31, 31), (0, 1, 3, 2)), ((142, 66, 124), (2, 0, 1)), ((128, 51, 112), (0, 2, 1)),
         ((89, 70, 134), (2, 0, 1)), ((1024, 700), (1, 0)), ((72, 91, 6, 27), (2, 1, 0, 3))]


def test_threads_with_other_boxes():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2112_13184_gb300 import ctm
    jobs = []
    for dims, perm in CASES:
        x = torch.arange(int(np.prod(dims)), dtype=torch.float64, device="cuda") + 0.5
        jobs.append((dims, perm, x, torch.empty_like(x), torch.cuda.Stream()))
    torch.cuda.synchronize()
    failed = []
    start = threading.Barrier(len(jobs))

    def work(dims, perm, x, y, stream):
        start.wait()
        for _ in range(3000):
            try:
                ctm.ctm_permute(x, y, dims, perm, stream=stream)
            except Exception as e:  # a refused launch: the context stays usable
                failed.append((dims, str(e)))
                return

    threads = [threading.Thread(target=work, args=j) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not failed, failed
    for dims, perm, x, y, _ in jobs:
        want = x.cpu().numpy().reshape(dims).transpose(perm)
        np.testing.assert_array_equal(y.cpu().numpy().reshape(want.shape), want)
