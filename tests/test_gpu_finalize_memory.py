"""Device memory of the solvers' final step: the FP64 path keeps the Ritz
vectors only (min(m + 1, 2 k + 2) columns); the others also the converted
kept columns (as many)."""
import pytest

from paper_2508_05400_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2508_05400_gb300 import build as B
    B.build()
    return torch


@pytest.mark.parametrize("prec,blocks", [("fp64", 1), ("df", 2)])
def test_memory_taken_by_the_final_step(gpu, prec, blocks):
    from paper_2508_05400_gb300 import rks
    A = I.toeplitz_tridiag(500_000)
    k, p = 20, 30
    with rks.Solver.from_csr(A, k, p, 2 * (k + p), which="LR", prec=prec, max_restarts=1) as s:
        s.solve()                                   # kernels loaded, pools grown
    with rks.Solver.from_csr(A, k, p, 2 * (k + p), which="LR", prec=prec, max_restarts=1) as s:
        before = gpu.cuda.mem_get_info()[0]
        s.solve()
        taken = before - gpu.cuda.mem_get_info()[0]
    block = 500_000 * 8 * (2 * k + 2)
    assert (blocks - 0.2) * block < taken < (blocks + 0.5) * block
