"""The LQ reduction of wide theta matrices inside the sweep.

A left-to-right update left of the centre orthogonalises a theta with up to four
times more columns than rows; the Jacobi path replaces it by the L of its LQ
factorisation.  FP32 (CUDA cores, Jacobi path) against the FP64 mode on the same
loaded state and layer: the partial fidelities of FP32 products and an SVD exact
to ~1e-6 agree to 2e-5; FP64 keeps a right-to-left / left-to-right invariant.
"""
import numpy as np
import pytest

from synthetic import circuits as sc

pytestmark = pytest.mark.gpu


def _state(n, chi, rng):
    bond = [min(2 ** i, 2 ** (n - i), chi) for i in range(n + 1)]
    mps = []
    for i in range(n):
        z = rng.normal(size=(2 * bond[i + 1], bond[i])) + 1j * rng.normal(size=(2 * bond[i + 1], bond[i]))
        q = np.linalg.qr(z)[0] if i else z / np.linalg.norm(z)
        mps.append(q.conj().T.reshape(bond[i], 2, bond[i + 1]))
    return mps


# theta widths up to 2 chi columns: 64 .. 512, the register classes of the
# reduction, with odd bonds
@pytest.mark.parametrize("rows,cols,chi_in,chi", [(2, 4, 9, 16), (3, 4, 24, 40), (3, 5, 40, 77), (4, 4, 64, 130)])
def test_wide_updates_fp32_against_fp64(rows, cols, chi_in, chi):
    from paper_2207_05612_gb300 import DMRGC_FP32, DMRGC_FP64, Context
    mps = _state(rows * cols, chi_in, np.random.default_rng(chi))
    layer = sc.random_circuit(rows, cols, 2, seed=chi).layers[0]
    hist = {}
    for prec in (DMRGC_FP64, DMRGC_FP32):
        ctx = Context(rows, cols, chi, precision=prec, svd_path=1, sweep_rel_cutoff=2e-5, zip_rel_cutoff=4e-3)
        ctx.set_mps(mps)
        ctx.apply_layer(layer)
        ctx.sweep(2)
        hist[prec] = np.array(ctx.history())
        new, centre = ctx.get_mps()
        for i, a in enumerate(new):
            al, _, ar = a.shape
            if i < centre:
                q = a.reshape(al * 2, ar)
                assert np.abs(q.conj().T @ q - np.eye(ar)).max() < (1e-11 if prec == DMRGC_FP64 else 1e-4)
        ctx.close()
    assert np.abs(hist[DMRGC_FP32] / hist[DMRGC_FP64] - 1).max() < 2e-5
