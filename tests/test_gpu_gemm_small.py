"""The 16 x 16 tile products (FP64 and FP32 CUDA cores) at the edges of their
tiles and K splits: one element, one past a tile, K below, at and past a block
and a split (2, 4 and 8 CTAs per tile), every operand op.  Bounds as for the
other GEMM tests: 1e-12 (FP64), 2e-5 (FP32) times sqrt(K)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

OPS = {0: lambda x: x, 1: lambda x: x.T, 2: lambda x: x.conj().T, 3: lambda x: x.conj()}


@pytest.mark.parametrize("prec,tol", [(0, 1e-12), (3, 2e-5)])
@pytest.mark.parametrize("m,n,k", [(1, 1, 1), (1, 40, 3), (16, 16, 16), (17, 15, 17), (33, 31, 32), (20, 50, 64), (16, 48, 130),
                                   (9, 200, 257), (64, 64, 511), (300, 20, 33)])
def test_small_tile_products(prec, tol, m, n, k):
    from paper_2207_05612_gb300 import binding
    rng = np.random.default_rng(m + 31 * n + 977 * k)
    for op_a in range(4):
        for op_b in range(4):
            a = rng.normal(size=(m, k) if op_a in (0, 3) else (k, m)) + 1j
            b = rng.normal(size=(k, n) if op_b in (0, 3) else (n, k)) - 0.5j
            want = OPS[op_a](a) @ OPS[op_b](b)
            got = binding.dmrgc_test_gemm(prec, a, b, op_a, op_b, m, n, k)
            assert np.abs(got - want).max() <= tol * np.abs(want).max() * np.sqrt(k), (op_a, op_b)
            again = binding.dmrgc_test_gemm(prec, a, b, op_a, op_b, m, n, k)
            assert np.array_equal(got, again)
