"""The fixed-point sums of rks_sketch_apply at the edges of its tiles and of its
number range, against the oracle's Omega summed in extended precision.

Bound per bin, from the kernel's arithmetic: every addend is rounded to within
2^-57 of the largest |x| (59-bit integers, at most two spare bits), and at
most 456 partial sums are scaled and added in FP64 (two roundings each).
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
    x = np.random.RandomState(n).standard_normal(n)
    if kind == "growing":
        x *= np.logspace(-30, 30, n)          # the power of two is raised many times
    elif kind == "wide":
        x *= 10.0 ** np.random.RandomState(1).uniform(-12, 12, n)
    elif kind == "zero":
        x[:] = 0.0
    return x


@pytest.mark.parametrize("n,d,zeta,kind", [
    (1, 16, 8, "normal"), (511, 16, 8, "normal"), (513, 33, 16, "normal"), (77_825, 64, 4, "wide"),
    (311_296, 600, 8, "normal"), (311_297, 96, 8, "growing"), (400_000, 3072, 8, "wide"), (50_000, 3073, 8, "normal"),
    (3000, 80, 5, "zero")])
def test_sums_within_the_derived_bound(gpu, n, d, zeta, kind):
    from paper_2508_05400_gb300 import rks
    x = _case(kind, n)
    z = rks.sketch_apply(gpu.from_numpy(x).cuda(), d, zeta, 7).cpu().numpy()
    rows, signs = SK.rows_signs(n, d, zeta, 7)
    ref, mag, cnt = np.zeros(d, np.longdouble), np.zeros(d), np.zeros(d)
    np.add.at(ref, rows, signs * x[:, None].astype(np.longdouble))
    np.add.at(mag, rows, np.abs(x)[:, None])
    np.add.at(cnt, rows, 1.0)
    ref /= np.sqrt(np.longdouble(zeta))
    # d > 3072 adds in FP64 bins: one rounding per addend and per partial sum instead
    tol = 2 * 456 * 2.0**-53 * mag + cnt * 2.0**-57 * np.abs(x).max() if d <= 3072 else (cnt + 912) * 2.0**-53 * mag
    assert np.all(np.abs(z - ref) <= tol)


def test_infinities_and_nans_stay_in_their_bins(gpu):
    from paper_2508_05400_gb300 import rks
    n, d, zeta = 70_001, 64, 4
    x = _case("normal", n)
    x[60_000], x[123] = np.inf, np.nan
    z = rks.sketch_apply(gpu.from_numpy(x).cuda(), d, zeta, 7).cpu().numpy()
    rows, signs = SK.rows_signs(n, d, zeta, 7)
    assert np.array_equal(np.flatnonzero(np.isnan(z)), np.unique(rows[123]))
    only_inf = np.setdiff1d(rows[60_000], rows[123])
    assert np.all(np.isinf(z[only_inf])) and np.isfinite(np.delete(z, np.r_[rows[123], rows[60_000]])).all()
