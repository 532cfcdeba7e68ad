"""Entries of the sliced FP64 products against sums in extended precision.

tests/host/f64_products_check.cu derives the bound and has the sizes: one entry to
several tiles and more slices than the work space holds, ragged in every dimension,
transposed, triangular, A A^T, with the scales in k that a factorization's products have.
"""
import os
import subprocess

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_every_entry_is_within_the_bound_of_the_split(tmp_path):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_1607_00346_gb300 import build
    lib = build.build_library()
    exe = str(tmp_path / "check")
    subprocess.run([build._nvcc(), *build.ARCH, "-O2", "-std=c++17", "-Xcompiler", "-ffp-contract=off",
                    "-I", build.INCLUDE, "-I", build.CSRC,
                    os.path.join(ROOT, "tests", "host", "f64_products_check.cu"), lib,
                    "-Xlinker", "-rpath=" + os.path.dirname(lib), "-o", exe], check=True)
    p = subprocess.run([exe], stdout=subprocess.PIPE, text=True)
    assert p.returncode == 0 and p.stdout.strip().endswith("OK"), p.stdout
