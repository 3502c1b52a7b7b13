"""rks_basis_product_df at the edges of its tiles: one row, ragged rows and
columns (the last K-step's columns are clamped), every width class of the
output (one or two MMAs per digit, one or two CTAs per SM), columns of very
different size, zero and subnormal rows, in place.

Bound: 2^-44 of (row maximum x column sum of |Q|), the accuracy the product
has had: seven 7-bit digits per operand leave 2^-47 of the row and column
scales per term, the dropped digit pairs and the light groups less than that.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2508_05400_gb300 import build as B
    B.build()
    return torch


@pytest.mark.parametrize("n,nin,nout,kind,inplace", [
    (1, 1, 1, "normal", False), (127, 3, 2, "normal", False), (129, 17, 16, "normal", True),
    (40_001, 80, 21, "graded", True), (5000, 33, 33, "normal", False), (300, 100, 50, "graded", True),
    (4097, 150, 51, "normal", True), (1000, 192, 64, "normal", False), (500, 24, 8, "empty", False)])
def test_product_within_the_digit_bound(gpu, n, nin, nout, kind, inplace):
    from paper_2508_05400_gb300 import rks
    rng = np.random.RandomState(n + nin)
    U = rng.standard_normal((nin, n))
    if kind == "graded":
        U *= 10.0 ** rng.uniform(-9, 9, (nin, 1))
    if kind == "empty":
        U[:, ::3] = 0.0
        U[:, 1::3] *= 1e-310
    Q = rng.standard_normal((nin, nout))
    ldu = (n + 31) // 32 * 32 + 32
    Ud = gpu.zeros(max(nin, nout), ldu, dtype=gpu.float64, device="cuda")
    Ud[:nin, :n] = gpu.from_numpy(U).cuda()
    out = Ud if inplace else gpu.full((nout, ldu), 7.0, dtype=gpu.float64, device="cuda")
    rks.basis_product_df(Ud, ldu, n, nin, Q, out)
    got = out[:nout, :n].cpu().numpy()
    want = (Q.T.astype(np.longdouble) @ U.astype(np.longdouble)).astype(np.longdouble)
    tol = 2.0**-44 * np.abs(Q).sum(axis=0)[:, None] * np.abs(U).max(axis=0)[None, :] + 1e-300
    assert np.all(np.abs(got - want) <= tol)
    if not inplace:
        assert np.all(out[:, n:].cpu().numpy() == 7.0)      # nothing past the rows is written
