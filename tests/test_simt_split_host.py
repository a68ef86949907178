"""Which CUDA-core kernel a product takes, without a GPU: gemm_simt.cu's rule built
into a host program (tests/host/simt_split.cu).  0: 64 x 64 tiles; else 16 x 16
tiles with K split over that many CTAs."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def split(tmp_path_factory):
    from paper_2207_05612_gb300 import build
    try:
        nvcc = build.nvcc()
    except RuntimeError:
        pytest.skip("needs nvcc")
    exe = str(tmp_path_factory.mktemp("host") / "simt_split")
    r = subprocess.run([nvcc, *build.ARCH, "-std=c++17", "--expt-relaxed-constexpr", "-I" + os.path.join(ROOT, "include"),
                        "-I" + build.CSRC, os.path.join(ROOT, "tests", "host", "simt_split.cu"), "-o", exe],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr

    def run(fp64, sizes):
        args = [str(x) for s in sizes for x in s]
        return [int(x) for x in subprocess.run([exe, str(int(fp64)), *args], capture_output=True, text=True,
                                               check=True).stdout.split()]
    return run


def test_fp32_products_that_fill_the_chip_keep_the_large_tiles(split):
    """The 16 x 16 kernel reaches half of the other's FP32 rate, so it is for grids that
    leave the chip idle: with two waves of large tiles and more (1024 x 1024 x 512:
    139 us against 207) the large tiles stay, below one wave of them the small ones."""
    large = [(1024, 1024, 512, 1), (1100, 1100, 300, 1), (1024, 1280, 1024, 1), (1152, 1152, 512, 1),
             (2048, 1024, 512, 1), (2048, 2048, 256, 1), (64, 64, 64, 305), (64, 256, 32, 128)]
    assert split(False, large) == [0] * len(large)
    small = [(1, 1, 1, 1), (16, 16, 16, 1), (64, 64, 512, 1), (200, 200, 200, 1), (256, 256, 1024, 1), (512, 512, 512, 1),
             (32, 1024, 512, 1), (4, 8, 4, 512), (1000, 300, 40, 1)]
    assert all(split(False, small))


def test_fp64_products_weigh_a_large_tile_as_sixteen(split):
    """At two FMAs a clock and SM both kernels run at the FMA rate: 1024 x 1024 x 512
    takes 4.2 ms on large tiles and 3.6 on small ones."""
    assert split(True, [(1024, 1024, 512, 1), (64, 64, 512, 1), (128, 128, 128, 1), (768, 768, 512, 1),
                        (2048, 2048, 256, 1)]) == [1, 8, 2, 0, 0]
