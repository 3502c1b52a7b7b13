"""rks_basis_product_df with a result that shares memory with its input: in the
same rows (in place, or from another column on), in other rows (shifted by
less than a tile, by a tile and by more than a column), and interleaved in the
padding of the columns.  The values are those of a result in its own memory.
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


@pytest.mark.parametrize("n,ldu,nin,nout,shift", [
    (40_001, 40_032, 24, 8, 0), (40_001, 40_032, 24, 8, 3 * 40_032), (40_001, 40_032, 24, 8, 1),
    (40_001, 40_032, 24, 8, 128), (40_001, 40_032, 24, 21, 2 * 40_032 + 20_000), (40_001, 40_032, 24, 8, -5),
    (5000, 10_000, 16, 5, 5000), (5000, 10_000, 16, 5, 4999), (5000, 5000, 3, 3, 5000 * 3)])
def test_result_over_the_input(gpu, n, ldu, nin, nout, shift):
    from paper_2508_05400_gb300 import rks
    rng = np.random.RandomState(n + nin)
    base = 64
    buf = gpu.from_numpy(rng.standard_normal(ldu * (nin + nout + 4) + 2 * base)).cuda()
    U = buf[base:]
    Q = rng.standard_normal((nin, nout))
    own = gpu.zeros(nout * ldu, dtype=gpu.float64, device="cuda")
    rks.basis_product_df(U, ldu, n, nin, Q, own)
    before = buf.clone()
    out = buf[base + shift:]
    rks.basis_product_df(U, ldu, n, nin, Q, out)
    written = gpu.zeros_like(buf, dtype=gpu.bool)
    for o in range(nout):
        assert gpu.equal(out[o * ldu:o * ldu + n], own[o * ldu:o * ldu + n])
        written[base + shift + o * ldu:base + shift + o * ldu + n] = True
    assert gpu.equal(buf[~written], before[~written])          # nothing else is written
