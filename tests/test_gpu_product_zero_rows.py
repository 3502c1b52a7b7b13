"""rks_basis_product_df on rows of zeros, of subnormal numbers, and of zeros
beside values so small that the row's scale reaches below the normal numbers.

A zero row gives exact zeros; subnormal inputs count as zeros.  Elsewhere the
bound is that of the product, 2^-44 of (row maximum x column sum of |Q|), and
one unit of the subnormal result.
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


@pytest.mark.parametrize("n,nin,nout", [(1, 1, 1), (500, 4, 1), (500, 24, 8), (1000, 192, 64)])
@pytest.mark.parametrize("fill", [0.0, -0.0, 1e-310, -5e-324])
@pytest.mark.parametrize("small", [1e-290, 4e-308])
def test_zero_rows_and_zeros_beside_tiny_values(gpu, n, nin, nout, fill, small):
    from paper_2508_05400_gb300 import rks
    rng = np.random.RandomState(n + nin)
    U = np.full((nin, n), fill)
    full = np.zeros(n, bool)
    full[2::3] = True                                   # an ordinary row
    U[:, full] = rng.standard_normal((nin, full.sum()))
    one = np.zeros(n, bool)
    one[1::3] = True                                    # one tiny value, the rest of the row is the fill
    U[0, one] = small * rng.uniform(1, 2, one.sum())
    Q = rng.standard_normal((nin, nout))
    out = gpu.full((nout, n), 7.0, dtype=gpu.float64, device="cuda")
    rks.basis_product_df(gpu.from_numpy(U).cuda(), n, n, nin, Q, out)
    got = out.cpu().numpy()
    U[np.abs(U) < 2.0**-1022] = 0.0
    want = Q.T.astype(np.longdouble) @ U.astype(np.longdouble)
    assert np.all(got[:, ~full & ~one] == 0.0)
    tol = 2.0**-44 * np.abs(Q).sum(axis=0)[:, None] * np.abs(U).max(axis=0)[None, :].astype(np.longdouble)
    assert np.all(np.abs(got - want) <= tol + np.longdouble(2.0**-1074) * (np.abs(want) > 0))
