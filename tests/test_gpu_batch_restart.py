"""The persistent batch at every width class of its restart product (an exact
width, a guarded one, the widest) and with the tile lists in shared memory or
read from global memory (zeta = 16: no room beside two CTAs per SM).

Checked after three restarts: the Krylov relation still holds, so that a Ritz
pair's residual is its estimate |b^T y| up to the sketch's distortion of two
norms (each within a factor of 2 for these d / m; a wrong product is off by
orders), for estimates above the double-float rounding of the basis; and the
results are the same bits with one CTA per problem and with four.
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


@pytest.mark.parametrize("k,p,keep,d,zeta", [
    (4, 8, 4, 64, 16), (4, 10, 5, 64, 8), (7, 13, 7, 80, 8), (9, 15, 9, 96, 8), (8, 24, 12, 128, 8),
    (14, 18, 14, 128, 8), (16, 24, 18, 120, 4)])
def test_restarted_pairs(k, p, keep, d, zeta):
    from paper_2508_05400_gb300 import rks
    mats = [I.convdiff_2d(70, 75, 1.0, 5.0, 3.0), I.convdiff_2d(41, 53, 1.0, 2.0, 1.0)]
    got = []
    for ctas in (1, 4):
        with rks.DevBatch(mats, k, p, d, which="LM", tol=1e-14, seed=0, zeta=zeta, maxit=3, conv="norm1", verify=0.0,
                          keep=keep, ctas=ctas) as b:
            b.solve(allow_noconv=True)
            got.append([b.eigpairs(i) for i in range(len(mats))])
    for one, four in zip(*got):
        for x, y in zip(one, four):
            assert np.array_equal(x, y)
        lam, X, res, rq, est = one
        sel = est > 1e-11
        assert lam.size >= k and np.any(sel)
        assert np.all(res[sel] <= 4.0 * est[sel]) and np.all(res[sel] >= 0.25 * est[sel])
