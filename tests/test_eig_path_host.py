"""Host logic of the truncated SVD's eigensolver path, without a GPU: api.cu built by
the host compiler with stand-ins for the CUDA runtime and the kernel families it
calls (tests/host/eig_path.cpp), so that a failing launch is an error code."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA = os.environ.get("CUDA_HOME", "/usr/local/cuda")


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    gxx = shutil.which("g++")
    if not gxx or not os.path.exists(os.path.join(CUDA, "include", "cuda_runtime.h")):
        pytest.skip("needs g++ and the CUDA headers")
    exe = str(tmp_path_factory.mktemp("host") / "eig_path")
    # what no scenario reaches stays unresolved
    r = subprocess.run([gxx, "-std=c++17", "-O0", "-no-pie", "-I" + os.path.join(ROOT, "include"),
                        "-I" + os.path.join(CUDA, "include"), "-I" + os.path.join(ROOT, "paper_2207_05612_gb300", "csrc"),
                        os.path.join(ROOT, "tests", "host", "eig_path.cpp"), "-o", exe,
                        "-Wl,--unresolved-symbols=ignore-in-object-files", "-ldl", "-lpthread"],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr

    def run(scenario):
        r = subprocess.run([exe, scenario], capture_output=True, text=True)
        assert r.returncode == 0, (r.returncode, r.stdout, r.stderr)
        return r.stdout.splitlines()
    return run


def test_failed_reduction_is_an_error(host):
    """A reduction that fails with an error of the call (out of memory 2, out of
    launch resources 701) returns DMRGC_ECUDA (3), in the first stage and in a
    later one; one that does not take the launch shape (9) is declined and the
    Jacobi SVD decides."""
    got = host("failed_reduction")
    want = []
    for rows, calls in ((250, (1,)), (400, (1, 2))):
        for call in calls:
            for error in (2, 701, 9):
                want.append(f"reduce rows={rows} call={call} error={error}: status={0 if error == 9 else 3} done=0 "
                            f"declined={1 if error == 9 else 0}")
    assert got == want


def test_bond_visits(host):
    """Which updates of one bond try the eigensolver.  A matrix that it does not take
    says nothing of the bond's other direction; a declined spectrum sends to the
    Jacobi SVD what resolves no more than the form that declined it."""
    assert host("visits") == [
        "tall then wide 600 x 250 left to right: not tried",
        "tall then wide 600 x 250 right to left: taken",
        "tall then wide 600 x 250 left to right: not tried",
        "grown bond 250 x 400 left to right: declined",
        "grown bond 250 x 400 left to right: skipped",
        "grown bond 300 x 400 left to right: taken",
        "grown bond 250 x 400 left to right: skipped",
        "one Gram matrix 250 x 400 left to right: declined",
        "one Gram matrix 250 x 400 left to right: skipped",
        "one Gram matrix 400 x 400 right to left: taken",
        "stages 400 x 400 left to right: declined",
        "stages 400 x 400 right to left: skipped",
        "stages 250 x 400 left to right: skipped",
        "low rank 250 x 150 left to right: not tried",
        "low rank 250 x 200 left to right: taken",
        "low rank, wide cut 250 x 150 left to right: taken",
        "records 400 x 400 left to right: declined",
        "records 400 x 400 right to left: taken",
    ]
