"""The plan that a factorization uses: build_fronts on the host, its rows on the GPU.

tests/host/fronts_check.cpp compares build_fronts with build_skel (which
test_symbolic_host.py checks against the geometry) on the CPU; tests/host/rows_check.cu
compares the device's row lists with build_skel's and filter_rows' on the GPU.  Grids
with C = 2 cells per dimension at the last level, where on the periodic grid both
neighbours of a cell are the same cell, are among them.
"""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = os.path.join(ROOT, "paper_1607_00346_gb300", "csrc")
HOST = os.path.join(ROOT, "tests", "host")

GRIDS = [(8, 4, ""), (12, 3, ""), (20, 5, ""), (24, 3, ""), (32, 4, ""), (14, 7, ""),
         (8, 4, "p"), (12, 3, "p"), (20, 5, "p"), (32, 4, "p"), (14, 7, "p")]


def _run(exe, n, m, bc):
    p = subprocess.run([exe, str(n), str(m)] + ([bc] if bc else []), stdout=subprocess.PIPE, text=True)
    assert p.returncode == 0, p.stdout
    assert p.stdout.strip().endswith("OK") and int(p.stdout.split()[0]) > 0


@pytest.fixture(scope="module")
def fronts(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no C++ compiler")
    exe = str(tmp_path_factory.mktemp("fronts") / "check")
    subprocess.run([cxx, "-O2", "-std=c++17", "-pthread", "-I", SRC, os.path.join(HOST, "fronts_check.cpp"),
                    os.path.join(SRC, "symbolic.cpp"), "-o", exe], check=True)
    return exe


@pytest.mark.parametrize("n,m,bc", GRIDS)
def test_fronts_are_those_of_the_checked_plan(fronts, n, m, bc):
    _run(fronts, n, m, bc)


@pytest.fixture(scope="module")
def rows(tmp_path_factory):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_1607_00346_gb300 import build
    lib = build.build_library()
    exe = str(tmp_path_factory.mktemp("rows") / "check")
    subprocess.run([build._nvcc(), *build.ARCH, "-O2", "-std=c++17", "-I", build.INCLUDE, "-I", SRC,
                    os.path.join(HOST, "rows_check.cu"), lib, "-Xlinker", "-rpath=" + os.path.dirname(lib),
                    "-o", exe], check=True)
    return exe


@pytest.mark.gpu
@pytest.mark.parametrize("n,m,bc", GRIDS)
def test_row_lists_on_the_gpu_are_those_of_the_checked_plan(rows, n, m, bc):
    _run(rows, n, m, bc)
