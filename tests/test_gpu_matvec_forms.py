"""The fine and the coarse form of the mat-vecs give the same bits.

Which form runs depends on how many thread blocks a list has (gemv.cu); the coarse one
carries the large applies.  tests/host/matvec_check.cu compares them on the same
operations, and the second test applies a whole factor large enough for it.
"""
import os
import subprocess

import pytest

from paper_1607_00346_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def H():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_1607_00346_gb300 import hif
    hif.load()
    return hif


def test_fine_and_coarse_lists_give_the_same_bits(H, tmp_path):
    from paper_1607_00346_gb300 import build
    lib = build.build_library()
    exe = str(tmp_path / "check")
    subprocess.run([build._nvcc(), *build.ARCH, "-O2", "-std=c++17", "-I", build.INCLUDE, "-I", build.CSRC,
                    os.path.join(ROOT, "tests", "host", "matvec_check.cu"), lib,
                    "-Xlinker", "-rpath=" + os.path.dirname(lib), "-o", exe], check=True)
    p = subprocess.run([exe], stdout=subprocess.PIPE, text=True)
    assert p.returncode == 0 and p.stdout.strip().endswith("OK"), p.stdout


@pytest.mark.parametrize("prec", [0, 1])
def test_every_block_of_a_large_apply_is_bitwise_the_single_column(H, prec):
    a = torch.from_numpy(inputs.coeff_log_uniform(64, -1.0, 1.0, 4500)).cuda()
    f = torch.from_numpy(inputs.normal_rhs(64, 16, 4501)).cuda()
    with H.factor(64, 4, a, b_const=0.1, eps=1e-4, precision=prec) as h:
        one = torch.zeros_like(f)
        for c in range(f.shape[0]):
            h.apply(f[c:c + 1], one[c:c + 1])
        for nrhs in (2, 3, 4, 5, 8, 11, 16):
            u = torch.full_like(f[:nrhs], float("nan"))
            h.apply(f[:nrhs], u)
            assert torch.equal(u, one[:nrhs]), nrhs
