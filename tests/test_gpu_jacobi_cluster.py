"""The cluster-resident Jacobi kernel at the edges of its size classes.

complex64: up to 512 rows (register classes 64, 128, 256, 512) and 256 columns
(128 above 256 rows); FP64: up to 512 rows and 64 columns.  Sizes one past an
edge take the next class or the grid-wide kernels.  Against LAPACK, with the
tolerances of the other Jacobi tests: complex64 3e-5 s_1 (numerical-zero level
1e-5 |G|_F), FP64 1e-12 s_1.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SIZES = [(1, 2), (2, 2), (3, 5), (7, 3), (16, 8), (17, 9), (32, 33), (33, 32), (63, 64), (64, 65), (65, 64), (100, 17),
         (127, 128), (128, 129), (129, 127), (256, 256), (257, 128), (255, 257), (511, 128), (512, 129), (513, 31),
         (400, 24), (24, 200)]


@pytest.mark.parametrize("prec,tol", [(3, 3e-5), (0, 1e-12)])
@pytest.mark.parametrize("m,n", SIZES)
def test_cluster_jacobi_against_lapack(prec, tol, m, n):
    from paper_2207_05612_gb300 import binding
    rng = np.random.default_rng(1000 * m + n)
    g = (rng.normal(size=(m, n)) + 1j * rng.normal(size=(m, n))) / np.sqrt(2 * max(m, n))
    want = np.linalg.svd(g, compute_uv=False)
    r = min(m, n)
    chi = max(1, r // 2)
    s, k, u = binding.dmrgc_test_svd(prec, g, chi, 1e-12 if prec == 0 else 2e-5)
    zero = (1e-13 if prec == 0 else 1e-5) * np.linalg.norm(g)
    big = want > 3 * zero
    assert np.abs(s[:r] - want)[big].max() <= tol * want[0]
    assert k == chi
    assert np.abs(u.conj().T @ u - np.eye(k)).max() < (1e-11 if prec == 0 else 1e-4)
    f_opt = float(np.sum(want[:k] ** 2))
    assert abs(float(np.sum(np.abs(u.conj().T @ g) ** 2)) - f_opt) <= (1e-11 if prec == 0 else 1e-5) * f_opt


@pytest.mark.parametrize("scale", [1e-60, 1e60])
def test_fp64_rotation_parameters_at_extreme_scales(scale):
    """The FP64 rotation takes its angle from FP32 arithmetic on scaled values:
    the scale of the matrix must not matter."""
    from paper_2207_05612_gb300 import binding
    rng = np.random.default_rng(9)
    g = scale * (rng.normal(size=(48, 40)) + 1j * rng.normal(size=(48, 40)))
    want = np.linalg.svd(g, compute_uv=False)
    s, k, u = binding.dmrgc_test_svd(0, g, 20, 1e-12)
    assert k == 20 and np.abs(s - want).max() <= 1e-12 * want[0]
    assert np.abs(u.conj().T @ u - np.eye(k)).max() < 1e-11


@pytest.mark.parametrize("prec,tol", [(3, 3e-5), (0, 1e-12)])
def test_equal_and_parallel_columns(prec, tol):
    """Columns of equal norm (the 45 degree rotation), parallel and zero ones."""
    from paper_2207_05612_gb300 import binding
    rng = np.random.default_rng(4)
    a = rng.normal(size=(40, 10)) + 1j * rng.normal(size=(40, 10))
    g = np.concatenate([a, 1j * a, np.zeros((40, 6)), a[:, :5] * np.exp(0.7j)], axis=1)
    want = np.linalg.svd(g, compute_uv=False)
    s, k, u = binding.dmrgc_test_svd(prec, g, 31, 1e-12 if prec == 0 else 2e-5)
    assert k == 10
    assert np.abs(s[:10] - want[:10]).max() <= tol * want[0]
    assert np.abs(u.conj().T @ u - np.eye(10)).max() < (1e-11 if prec == 0 else 1e-4)
