"""rks_basis_product_f32 at the edges of its tiles and pipeline: one row, ragged
rows, one K-step (fewer than the stages) to sixteen, ragged columns, every
group of output columns, several tiles per CTA, in place.

Bound: 2^-23 (6 nk + 8) sum_l |u_l| |q_l| for nk K-steps of 16 columns: each of
the 6 nk products added to the FP32 accumulator may lose a unit of its last
place, and so may the few additions inside one; the splits themselves leave
less than 2^-31.
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


@pytest.mark.parametrize("n,nin,nout,inplace", [
    (1, 1, 1, False), (127, 8, 7, False), (129, 9, 8, True), (128, 32, 17, False), (5000, 33, 33, True),
    (150_001, 48, 16, False), (300, 150, 51, True), (120_000, 17, 64, False), (1000, 256, 64, True)])
def test_product_within_the_split_bound(gpu, n, nin, nout, inplace):
    from paper_2508_05400_gb300 import rks
    rng = np.random.RandomState(n + nin)
    U = (rng.standard_normal((nin, n)) * 10.0 ** rng.uniform(-6, 6, (nin, 1))).astype(np.float32)
    Q = rng.standard_normal((nin, nout))
    ldu = (n + 31) // 32 * 32 + 32
    Ud = gpu.zeros(max(nin, nout), ldu, dtype=gpu.float32, device="cuda")
    Ud[:nin, :n] = gpu.from_numpy(U).cuda()
    out = Ud if inplace else gpu.full((nout, ldu), 7.0, dtype=gpu.float32, device="cuda")
    rks.basis_product_f32(Ud, ldu, n, nin, Q, out)
    got = out[:nout, :n].cpu().numpy().astype(np.float64)
    nk = 2 * ((nin + 31) // 32)
    tol = 2.0**-23 * (6 * nk + 8) * (np.abs(Q).T @ np.abs(U.astype(np.float64)))
    assert np.all(np.abs(got - Q.T @ U.astype(np.float64)) <= tol)
    if not inplace:
        assert np.all(out[:, n:].cpu().numpy() == 7.0)      # nothing past the rows is written
