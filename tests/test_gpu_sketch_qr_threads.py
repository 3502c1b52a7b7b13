"""Randomized Gram-Schmidt from two host threads at once, one with the largest
sketch, one with a smaller sketch that also needs more than 48 KB of shared
memory: each result is that of the call alone, bit for bit."""
import threading

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_two_sizes_from_two_threads():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2508_05400_gb300 import build as B
    B.build()
    from paper_2508_05400_gb300 import rks
    K = torch.from_numpy(np.random.RandomState(5).standard_normal((12, 4000))).cuda()
    sizes = [8192, 6200]
    want = {d: rks.sketch_qr(K, d, 8, 3, method="rgs") for d in sizes}
    errors = []

    def run(d):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                for _ in range(60):
                    Q, R, S = rks.sketch_qr(K, d, 8, 3, method="rgs")
                    assert torch.equal(Q, want[d][0]) and np.array_equal(R, want[d][1]) and np.array_equal(S, want[d][2])
        except BaseException as e:
            errors.append(f"d = {d}: {e!r}")
    threads = [threading.Thread(target=run, args=(d,)) for d in sizes]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
