"""Amplitudes on the tensor cores, where the strings are grouped by their bit at
each site (groups of whole 128-row tiles), against the FP64 read-out, which
multiplies both halves of a site tensor and picks one (as do fewer than 128
strings on the tensor cores).

A product of K terms with operands rounded to 2 x 11 bits and FP32 sums is off by
at most about 2^-21 of sum |v||a|, for a random state sqrt(K) times the value:
over 12 sites of up to 24 columns 12 x 5 x 2^-21 = 2.9e-5 of a typical amplitude;
the bound is 8 times that, 2.3e-4 of the rms over 256 random strings.  A string taken from the
wrong row is off by about 1.  16386 and
20000 strings need a second chunk."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bits_one", [0.5, 0.0, 1.0, 0.01])
@pytest.mark.parametrize("count", [1, 2, 127, 128, 129, 255, 257, 1025, 16386, 20000])
def test_grouped_rows_against_fp64(count, bits_one):
    from paper_2207_05612_gb300 import DMRGC_FP64, DMRGC_TF32X3, Context
    rng = np.random.default_rng(count)
    n, chi = 12, 24
    bond = [min(2 ** i, 2 ** (n - i), chi) for i in range(n + 1)]
    mps = [(rng.normal(size=(l, 2, r)) + 1j * rng.normal(size=(l, 2, r))) / np.sqrt(2 * l)
           for l, r in zip(bond[:-1], bond[1:])]
    bits = (rng.random((count, n)) < bits_one).astype(np.uint8)
    some = rng.integers(0, 2, (256, n)).astype(np.uint8)
    amps = []
    for precision in (DMRGC_FP64, DMRGC_TF32X3):
        ctx = Context(3, 4, chi, precision=precision)
        ctx.set_mps(mps)
        amps.append(ctx.amplitude(bits))
        if precision == DMRGC_FP64:
            rms = np.sqrt(np.mean(np.abs(ctx.amplitude(some)) ** 2))
        ctx.close()
    off = np.abs(amps[1] - amps[0]).max()
    print("largest difference / rms", off / rms)
    assert off < 2.3e-4 * rms
