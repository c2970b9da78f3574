"""The grouped GEMM's tiles on the host (the library's make_tiles, called by a small program): every output once, in order,
also where a block has more than 2^31 outputs, a block or triangle of one row, and K split evenly over several CTAs."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def driver(tmp_path_factory):
    import __graft_entry__
    lib = os.path.join(ROOT, "paper_1103_5391_gb300", "libtdmrg.so")
    if not os.path.exists(lib):
        __graft_entry__.build()
    cuda = os.path.dirname(os.path.dirname(shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"))
    exe = str(tmp_path_factory.mktemp("tiles") / "tiles")
    csrc = os.path.join(ROOT, "paper_1103_5391_gb300", "csrc")
    r = subprocess.run(["g++", "-std=c++17", "-O2", os.path.join(ROOT, "tests", "tiles_driver.cpp"), "-o", exe, "-I", csrc,
                        "-I", os.path.join(ROOT, "include"), "-I", os.path.join(cuda, "include"), lib,
                        "-Wl,-rpath," + os.path.dirname(lib), "-Wl,--unresolved-symbols=ignore-all"], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return exe


@pytest.mark.parametrize("m,n,k,herm", [(1, 1, 1, 0), (1, 700, 5, 0), (700, 1, 5, 0), (37, 41, 9, 0), (37, 41, 3000, 0), (1, 1, 4, 1),
                                        (23, 23, 9, 1), (300, 300, 5, 1), (61, 61, 3072, 1), (46400, 46400, 4, 0), (65600, 65600, 4, 1)])
def test_tiles_cover_the_outputs(driver, m, n, k, herm):
    r = subprocess.run([driver, str(m), str(n), str(k), str(herm)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
