"""rks_sketch_apply bin by bin: a bin's error is bounded by the values that fall
into that bin, whatever the others are.  Inputs of a wide range: one entry far
above the rest (at the start, at the end, in a tile of its own), values that
shrink or grow from tile to tile, exponents spread over the whole range of
FP64, subnormal numbers beside ordinary ones.

Bound per bin: FP64 accumulation, one rounding per addend, and two per partial
sum of at most 304 CTAs: (addends + 608) 2^-53 sum |x| over the bin, and half
a subnormal unit for each rounding there.
"""
import numpy as np
import pytest

from oracle import sketch as SK

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2508_05400_gb300 import build as B
    B.build()
    return torch


def _case(kind, n):
    rng = np.random.RandomState(n)
    x = rng.standard_normal(n)
    if kind == "spike9":
        x[n // 3] = -1e9
    elif kind.startswith("spike"):
        x[{"spike0": 0, "spike_end": n - 1, "spike_mid": n // 2}[kind]] = 1e20
    elif kind == "shrinking":
        x *= np.logspace(30, -30, n)
    elif kind == "growing":
        x *= np.logspace(-30, 30, n)
    elif kind == "range":
        x = np.ldexp(x, rng.randint(-1000, 1000, n))
    elif kind == "subnormal":
        x[::3] *= 5e-310
    return x


@pytest.mark.parametrize("n,d,zeta,kind", [
    (1000, 200, 2, "spike0"), (20_000, 600, 8, "spike_end"), (311_297, 600, 8, "spike_mid"),
    (311_297, 3072, 4, "spike9"), (200_000, 96, 16, "shrinking"), (200_000, 96, 8, "growing"),
    (100_000, 3000, 8, "range"), (100_000, 600, 8, "range"), (5000, 700, 1, "subnormal"),
    (50_000, 3073, 8, "spike_mid"), (400_000, 600, 8, "normal")])
def test_every_bin_as_accurate_as_its_own_values(gpu, n, d, zeta, kind):
    from paper_2508_05400_gb300 import rks
    x = _case(kind, n)
    z = rks.sketch_apply(gpu.from_numpy(x).cuda(), d, zeta, 7).cpu().numpy()
    rows, signs = SK.rows_signs(n, d, zeta, 7)
    ref, mag, cnt = np.zeros(d, np.longdouble), np.zeros(d, np.longdouble), np.zeros(d)
    np.add.at(ref, rows, signs * x[:, None].astype(np.longdouble))
    np.add.at(mag, rows, np.abs(x)[:, None].astype(np.longdouble))
    np.add.at(cnt, rows, 1.0)
    ref /= np.sqrt(np.longdouble(zeta))
    tol = (cnt + 608) * (2.0**-53 * mag + 2.0**-1075)
    assert np.all(np.abs(z - ref) <= tol)
