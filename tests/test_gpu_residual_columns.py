"""FP64 residuals and Rayleigh quotients of one to nine Ritz vectors (the kernel
takes four real ones at a time, the last one to three by kernels of that many;
before convergence some are conjugate pairs) on symmetric matrices with rows of every length: short ones, ones on either side
of the limit of a long row, all of them long, one far longer than its
neighbours, and several such beside each other.  Compared with the oracle's
sums of the same vectors: FP64 sums of at most 3000 products per row in another
order.
"""
import numpy as np
import pytest
import scipy.sparse as sp

from oracle import rks as R
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


def _matrix(kind, n=3001):
    rng = np.random.RandomState(len(kind))
    w = {"short": 2, "at_limit": 31, "all_long": 60}.get(kind, 3)
    A = sp.diags([rng.standard_normal(n - o) for o in range(w + 1)], range(w + 1), shape=(n, n), format="lil")
    if kind in ("one_far_longer", "several"):
        for i in ([1500] if kind == "one_far_longer" else [64, 65, 66, 70, 95, 96, 3000]):
            A[i, :] = rng.standard_normal(n)
    A = sp.csr_matrix(A)
    A = sp.csr_matrix(sp.triu(A) + sp.triu(A, 1).T + sp.diags(np.linspace(0, 200, n)))
    A.sort_indices()
    return I.CSR(n, A.indptr.astype(np.int32), A.indices.astype(np.int32), A.data)


@pytest.mark.parametrize("prec", ["df", "fp64"])
@pytest.mark.parametrize("k", [1, 2, 3, 4, 5, 7, 9])
@pytest.mark.parametrize("kind", ["short", "at_limit", "all_long", "one_far_longer", "several"])
def test_residuals_of_real_columns(kind, k, prec):
    from paper_2508_05400_gb300 import rks
    A = _matrix(kind)
    with rks.Solver.from_csr(A, k, 12, 4 * (k + 12), which="LR", tol=1e-10, u1=I.start_vector(A.n, 1), prec=prec,
                             max_restarts=3) as s:
        s.solve()
        lam, X, res = s.eigpairs()
        rq = s.rayleigh()
    res_o, rq_o = R.true_residuals(A.to_scipy(), rks.unpack_eigvecs(lam, X), lam)
    # rounding of a row's products and of the sums over n rows, on ||A||_1 ||x||
    assert np.all(np.abs(res - res_o) <= 1e-13 + 1e-10 * res_o)
    assert np.all(np.abs(rq - rq_o) <= 1e-12 * I.norm1(A))
