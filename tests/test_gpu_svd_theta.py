"""The truncated SVD of one update by the route the sweep takes, against LAPACK:
the staged Gram eigensolver in every complex64 mode and both directions, and the
LQ reduction of wide matrices before the Jacobi SVD.

Bounds.  Isometry: the Jacobi SVD stops when every pair of columns is orthogonal to
8 eps sqrt(m); every route is held to twice that.  Rank: the values above the
larger of rel_cut s_1 and the numerical zero (complex64: 1e-5 |G|_F), where values
within 5% of it may fall on either side.  Weight: a direction at the cut carries at
most 4e-10 s_1^2, and a few lie that close, so the span may miss 1e-9 of the optimum
of its rank.  LQ: a backward error of n eps s_1, so values to 2 n eps s_1 and the
off-diagonal of U^+ G G^+ U, which any other orthonormal U would fill, to
4 n eps s_1^2 (eps of the type, and 8 eps sqrt(m) s_1^2 from the stopping rule)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

EPS32, EPS64 = 2.0 ** -24, 2.0 ** -53

SPECTRA = {
    "graded3": lambda q: 10.0 ** (-3 * np.arange(q) / q),
    "graded5": lambda q: 10.0 ** (-5 * np.arange(q) / q),
    "graded8": lambda q: 10.0 ** (-8 * np.arange(q) / q),
    "step": lambda q: np.where(np.arange(q) < q // 3, 1.0, 1e-3) * np.linspace(1, 0.5, q),
    "half": lambda q: np.where(np.arange(q) < q // 2, 1.0, 0.0) * np.linspace(1, 0.3, q),
}


def _matrix(m, n, spectrum, seed):
    rng = np.random.default_rng(seed)
    q = min(m, n)
    s = SPECTRA[spectrum](q)
    s = s / np.linalg.norm(s)
    u, v = (np.linalg.qr(rng.normal(size=(k, q)) + 1j * rng.normal(size=(k, q)))[0] for k in (m, n))
    return (u * s) @ v.conj().T, s


def _missed(g, s, u):
    q = np.linalg.qr(u)[0]
    best = np.sum(s[:u.shape[1]] ** 2)
    return (best - np.sum(np.abs(q.conj().T @ g) ** 2)) / best


@pytest.mark.parametrize("right", [False, True])
@pytest.mark.parametrize("prec", [1, 2, 3])
@pytest.mark.parametrize("m,n,chi,spectrum,parts", [
    (257, 300, 512, "graded3", 2), (300, 300, 512, "graded5", 3), (301, 401, 150, "graded8", 2), (400, 400, 500, "half", 1),
    (512, 700, 256, "step", 2), (600, 512, 600, "graded8", 3), (1024, 520, 512, "graded5", 3), (1024, 1024, 512, "step", 2)])
def test_stages(m, n, chi, spectrum, parts, prec, right):
    from paper_2207_05612_gb300 import binding
    g, s = _matrix(m, n, spectrum, m + n)
    k, u, got = binding.dmrgc_test_svd_theta(prec, g, chi, 2e-5, right=right)
    iso = np.abs(u.conj().T @ u - np.eye(k)).max()
    missed = _missed(g, s, u)
    print(f"{m} x {n} {spectrum} mode {prec}: k {k}, parts {got}, isometry {iso:.1e}, weight missed {missed:.1e}")
    assert got == parts
    cut = max(2e-5 * s[0], 1e-5)
    assert min(chi, np.sum(s > 1.05 * cut)) <= k <= min(chi, np.sum(s > cut / 1.05))
    assert iso < 2 * 8 * EPS32 * np.sqrt(m)
    assert missed < 1e-9


# the register classes of the reduction (64, 128, 256, 512 columns) at their edges,
# the fewest and the most rows of each type
@pytest.mark.parametrize("prec", [0, 3])
@pytest.mark.parametrize("m,n,spectrum", [
    (2, 3, "step"), (2, 512, "graded3"), (5, 64, "graded3"), (17, 65, "step"), (63, 64, "graded5"), (64, 128, "step"),
    (65, 129, "graded3"), (100, 255, "half"), (127, 256, "graded3"), (128, 257, "graded5"), (128, 511, "step"),
    (128, 512, "graded3"), (200, 256, "step"), (256, 512, "graded3")])
def test_wide_matrices(m, n, spectrum, prec):
    from paper_2207_05612_gb300 import binding
    g, s = _matrix(m, n, spectrum, m * n)
    eps, zero, cut = (EPS64, 1e-13, 1e-12) if prec == 0 else (EPS32, 1e-5, 2e-5)
    for case in ("as it is", "parallel and zero rows"):
        if case != "as it is":
            g = g.copy()
            g[m - 1] = 0
            g[m // 2] = (0.6 + 0.8j) * g[0]
            s = np.linalg.svd(g, compute_uv=False)
        k, u, parts = binding.dmrgc_test_svd_theta(prec, g, m, cut, svd_path=1)
        assert parts == 0
        level = max(cut * s[0], zero * np.linalg.norm(s))
        assert k <= np.sum(s > level / 1.05)
        if prec == 0:   # a column below the numerical zero is left as it is: in complex64 it can hold part of a value above
            assert k >= np.sum(s > 1.05 * level)
        stop = 8 * eps * np.sqrt(m)
        assert np.abs(u.conj().T @ u - np.eye(k)).max() < 2 * stop
        w = u.conj().T @ g
        assert np.abs(np.sqrt(np.sum(np.abs(w) ** 2, axis=1)) - s[:k]).max() < (2 * n * eps + stop) * s[0]
        h = w @ w.conj().T
        assert np.abs(h - np.diag(np.diag(h))).max() < (4 * n * eps + stop) * s[0] ** 2
