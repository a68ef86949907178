"""The cluster tridiagonalisation at the edges of its size classes: 3 rows, the
register classes (128, 256, 512 rows in one cluster), the hand-over from several
clusters (513 .. 1024 rows) and from the grid-wide kernel (1025).  Bounds of the
other Gram eigensolver tests: 3e-5 s_1, isometry 1e-4, weight 1e-5; the result is
the same on every run."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [3, 4, 5, 31, 32, 33, 127, 128, 129, 255, 256, 257, 511, 512, 513, 514, 640, 1023, 1024, 1025])
def test_cluster_tridiagonalisation(n):
    from paper_2207_05612_gb300 import binding
    rng = np.random.default_rng(n)
    g = (rng.normal(size=(n, n + 3)) + 1j * rng.normal(size=(n, n + 3))) / np.sqrt(2 * n)
    want = np.linalg.svd(g, compute_uv=False)
    chi = max(1, n // 2)
    s, k, u = binding.dmrgc_test_svd_gram(2, g, chi, 2e-5)
    assert k == chi
    assert np.abs(s[:k + 1] - want[:k + 1]).max() <= 3e-5 * want[0]
    assert np.abs(u.conj().T @ u - np.eye(k)).max() < 1e-4
    f_opt = float(np.sum(want[:k] ** 2))
    assert abs(float(np.sum(np.abs(u.conj().T @ g) ** 2)) - f_opt) <= 1e-5 * f_opt
    s2, k2, u2 = binding.dmrgc_test_svd_gram(2, g, chi, 2e-5)
    assert k2 == k and np.array_equal(s, s2) and np.array_equal(u, u2)


@pytest.mark.parametrize("n", [130, 600])
def test_cluster_tridiagonalisation_of_a_block_diagonal_gram(n):
    """Columns that need no reflector (already tridiagonal) and zero rows."""
    from paper_2207_05612_gb300 import binding
    g = np.diag(np.linspace(1.0, 0.2, n)).astype(complex)
    g[n - 5:, :] = 0
    s, k, u = binding.dmrgc_test_svd_gram(2, g, n // 3, 2e-5)
    assert k == n // 3
    assert np.abs(s[:k] - np.linspace(1.0, 0.2, n)[:k]).max() < 3e-5
    assert np.abs(u.conj().T @ u - np.eye(k)).max() < 1e-4
