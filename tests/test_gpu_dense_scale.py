"""The device dense step on matrices far from unit size (rks_dev_ordered_schur):
the reflectors' vectors are quadratic in the matrix and squared again, so the
squares leave the range of FP64 long before the matrix does.  Scaling by a
power of two changes no digit of the problem: orthogonality, similarity and
eigenvalues have the bounds of the unit-sized matrix."""
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


@pytest.mark.parametrize("m", [3, 8, 32, 64])
@pytest.mark.parametrize("p", [-330, -270, -266, -90, 200, 330])
def test_dense_step_of_a_scaled_matrix(m, p):
    from paper_2508_05400_gb300 import rks
    B = np.random.default_rng(m).standard_normal((m, m))
    T, Q, lam, _ = rks.dev_ordered_schur(np.ldexp(B, p), "LR", min(m - 1, 13))
    T, lam = np.ldexp(T, -p), np.ldexp(lam.real, -p) + 1j * np.ldexp(lam.imag, -p)
    nb = np.linalg.norm(B)
    assert np.linalg.norm(Q.T @ Q - np.eye(m)) <= 1e-13 * m
    assert np.linalg.norm(B - Q @ T @ Q.T) <= 1e-13 * nb
    assert np.all(np.tril(T, -2) == 0.0)
    assert np.allclose(np.sort_complex(lam), np.sort_complex(np.linalg.eigvals(B)), atol=1e-11 * nb)
