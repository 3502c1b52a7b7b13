"""The one-launch expansion of small problems gives the bits of the separate
kernels (which run when the kernel classes are timed), at the edges of its
ranges: one CTA to sixteen, one and two tiles per CTA, S and M or the basis in
shared memory or not, storage by diagonals and CSR, ragged rows and sketch
sizes that are no multiple of anything.
"""
import numpy as np
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


def _matrix(kind, n):
    if kind == "tridiag":
        return I.paper_tridiag(n, "exponential")
    if kind == "conv2d":
        return I.convdiff_2d(n, n + 3, 1.0, 20.0, 10.0)
    if kind == "conv3d":                                   # FP32 values
        return I.convdiff_3d(n, n, n, I.lognormal_field((n, n, n)), (10.0, 5.0, 2.0), dtype=np.float32)
    rng = np.random.RandomState(n)                         # CSR: 3 to 9 random columns a row
    rows = [np.unique(np.append(rng.randint(0, n, rng.randint(2, 9)), i)) for i in range(n)]
    ptr = np.concatenate([[0], np.cumsum([r.size for r in rows])])
    return I.CSR(n, ptr.astype(np.int32), np.concatenate(rows).astype(np.int32), rng.standard_normal(ptr[-1]))


@pytest.mark.parametrize("kind,size,k,p,d,zeta,fused", [
    ("tridiag", 60, 3, 7, 24, 4, True), ("tridiag", 127, 4, 12, 33, 5, True), ("tridiag", 2000, 10, 30, 80, 4, True),
    ("conv2d", 31, 6, 18, 72, 8, True), ("conv2d", 120, 16, 40, 200, 8, True), ("conv3d", 25, 8, 24, 96, 8, True),
    ("random", 1025, 5, 15, 50, 8, True), ("random", 16_384, 6, 18, 64, 16, True),
    # too many rows, too large sketches: the separate kernels
    ("conv2d", 179, 20, 60, 320, 8, False), ("conv3d", 25, 8, 24, 500, 16, False),
    ("random", 20_011, 8, 24, 1024, 8, False)])
def test_same_bits_as_the_separate_kernels(kind, size, k, p, d, zeta, fused):
    from paper_2508_05400_gb300 import rks
    A = _matrix(kind, size)
    u1 = I.start_vector(A.n, 3)
    got = []
    for profile in (False, True):
        with rks.Solver.from_csr(A, k, p, d, which="LR", tol=1e-10, zeta=zeta, u1=u1, keep=k, max_restarts=3,
                                 profile=profile) as s:
            s.solve()
            got.append((s.eigpairs(), s.krylov(), s.stats()["launches_total"]))
    (e0, k0, l0), (e1, k1, l1) = got
    for a, b in zip(e0 + k0, e1 + k1):
        assert np.array_equal(a, b)
    assert (l0 < l1) == fused
