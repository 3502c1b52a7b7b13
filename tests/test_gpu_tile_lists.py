"""The sketch's tile lists where their copies into shared memory change form:
tiles that start at any even row, so that the entries of a zeta that is no
multiple of 4 are 4-byte aligned only; sketch sizes that are no multiple of 4;
every number of lanes per sketch row; ragged last tiles; storage by diagonals,
ELLPACK and row pointers; both directions of the update's tile order.

The first expansion of Algorithm 2 is compared column by column with the FP64
oracle, at the tolerance of the other expansion tests.
"""
import numpy as np
import pytest
import scipy.sparse as sp

from oracle import rks as R
from oracle import sketch as SK
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


def _matrix(kind):
    if kind == "conv2d":
        return I.convdiff_2d(140, 143, 1.0, 20.0, 10.0)
    if kind == "conv3d":
        return I.convdiff_3d(71, 71, 71, I.lognormal_field((71, 71, 71)), (10.0, 5.0, 2.0), dtype=np.float32)
    n = 20_011                                                    # 3 to 9 random columns a row
    rng = np.random.RandomState(n)
    rows = [np.unique(np.append(rng.randint(0, n, rng.randint(2, 9)), i)) for i in range(n)]
    ptr = np.concatenate([[0], np.cumsum([r.size for r in rows])])
    return I.CSR(n, ptr.astype(np.int32), np.concatenate(rows).astype(np.int32), rng.standard_normal(ptr[-1]))


@pytest.mark.parametrize("kind,d,zeta", [
    ("conv2d", 50, 6), ("conv2d", 71, 3), ("conv2d", 130, 5), ("conv2d", 515, 1), ("random", 61, 7),
    ("random", 258, 16), ("conv3d", 96, 8)])
def test_first_expansion_per_column(kind, d, zeta):
    from paper_2508_05400_gb300 import rks
    A = _matrix(kind)
    u1 = I.start_vector(A.n, 1)
    with rks.Solver.from_csr(A, 4, 12, d, which="LM", tol=1e-12, zeta=zeta, u1=u1, max_restarts=-1) as s:
        s.solve()
        U, S, H = s.krylov()
    st = R.start(sp.csr_matrix(A.to_scipy()), SK.omega_matrix(A.n, d, zeta, 0), u1)
    R.extend(st, 16)
    for got, want in ((H, st.Ba), (S, st.Sa), (U, st.Ua)):
        err = np.linalg.norm(got - want, axis=0) / np.maximum(np.linalg.norm(want, axis=0), 1e-300)
        assert err.max() <= 1e-10
