"""rks_sketch_qr at the edges of its panels (8 columns), of its 4 x 4 Gram
blocks and of its row tiles, all four methods, against the uniqueness of the
factorisation: K = Q R with R upper triangular and positive diagonal, and
(Omega Q)^T (Omega Q) = I or Q^T Q = I.

Bounds: a double-float pair carries 2^-48; K = Q R to s such roundings of the
largest product (s * 2^-46 relative to ||K||), orthonormality to the same times
the condition of these well-conditioned blocks (below 1e2): 1e-11.
"""
import numpy as np
import pytest

from oracle import sketch as SK

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("method", ["rgs", "whiten", "rcholqr", "rhqr"])
@pytest.mark.parametrize("n,s,d,zeta", [(2051, 1, 40, 4), (1025, 7, 64, 8), (3000, 8, 64, 8), (20_011, 17, 96, 8),
                                        (5001, 33, 800, 8)])
def test_factorisation_at_panel_edges(method, n, s, d, zeta):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2508_05400_gb300 import build as B
    B.build()
    from paper_2508_05400_gb300 import rks
    K = np.random.RandomState(n).standard_normal((s, n))
    K[1:] += 0.5 * K[:-1]
    Q, R, S = rks.sketch_qr(torch.from_numpy(K).cuda(), d, zeta, 3, method=method)
    Q = Q.cpu().numpy()
    assert np.array_equal(R, np.triu(R)) and np.all(np.diag(R) > 0)
    assert np.linalg.norm(R.T @ Q - K) <= s * 2.0**-46 * np.linalg.norm(K)
    if method == "rhqr":
        T = SK.omega_matrix(n - s, d, zeta, 3) @ Q[:, s:].T
        G = T.T @ T + Q[:, :s] @ Q[:, :s].T
    else:
        T = SK.omega_matrix(n, d, zeta, 3) @ Q.T
        G = Q @ Q.T if method == "rcholqr" else T.T @ T
    assert np.linalg.norm(G - np.eye(s)) <= 1e-11
    assert np.linalg.norm(S - T) <= 1e-11 * np.linalg.norm(T)
