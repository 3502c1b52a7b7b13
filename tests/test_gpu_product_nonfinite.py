"""Rows with an infinity or a NaN in the tensor-core products: every output of
such a row is no number, and the other rows are those of the finite input."""
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


@pytest.mark.parametrize("nin,nout", [(3, 2), (24, 21), (100, 50)])
@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan])
def test_rows_with_no_numbers(gpu, nin, nout, bad):
    from paper_2508_05400_gb300 import rks
    n = 1000
    rng = np.random.RandomState(nin)
    U = rng.standard_normal((nin, n))
    Q = rng.standard_normal((nin, nout))
    Q[nin - 1, 0] = 0.0
    out = [gpu.zeros(nout, n, dtype=gpu.float64, device="cuda") for _ in range(2)]
    rks.basis_product_df(gpu.from_numpy(U).cuda(), n, n, nin, Q, out[0])
    rows = np.array([0, 127, 128, 500, n - 1])
    U[nin - 1, rows] = bad
    U[0, rows[2]] = 1e300
    rks.basis_product_df(gpu.from_numpy(U).cuda(), n, n, nin, Q, out[1])
    a, b = out[0].cpu().numpy(), out[1].cpu().numpy()
    assert not np.isfinite(b[:, rows]).any()
    assert np.array_equal(np.delete(b, rows, axis=1), np.delete(a, rows, axis=1))
