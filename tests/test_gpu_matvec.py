"""The apply's mat-vecs over every block size of right-hand sides.

Each column of an apply has to get the bits of its own one-column apply in any
block (16, 8, 4, 2, 1 columns, full or partly masked), in a grouped apply too,
and a column that is not finite must leave the others alone.  Leaf sizes 3 to 5
give matrices of 8 to several hundred rows and columns with every remainder of
the 64-row tiles and 32-column groups; eps = 0 has the largest triangles.
"""
import numpy as np
import pytest

from paper_1607_00346_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def H():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_1607_00346_gb300 import hif
    hif.load()
    return hif


@pytest.mark.parametrize("n,m,eps", [(12, 3, 0.0), (24, 3, 1e-4), (20, 5, 0.0), (32, 4, 1e-6)])
@pytest.mark.parametrize("prec", [0, 1])
def test_every_block_of_columns_is_bitwise_the_single_column(H, n, m, eps, prec):
    a = torch.from_numpy(inputs.coeff_log_uniform(n, -1.0, 1.0, 4100 + n)).cuda()
    f = torch.from_numpy(inputs.normal_rhs(n, 33, 4200 + n)).cuda()
    with H.factor(n, m, a, b_const=0.1, eps=eps, precision=prec) as h:
        one = torch.zeros_like(f)
        for c in range(f.shape[0]):
            h.apply(f[c:c + 1], one[c:c + 1])
        for nrhs in (2, 3, 4, 5, 7, 8, 9, 15, 16, 17, 19, 33):
            u = torch.full_like(f[:nrhs], float("nan"))
            h.apply(f[:nrhs], u)
            assert torch.equal(u, one[:nrhs]), nrhs
            g = torch.full_like(u, float("nan"))
            H.apply_batch([h], [f[:nrhs]], [g])
            assert torch.equal(g, u), nrhs


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("bad", [np.inf, np.nan])
def test_a_column_that_is_not_finite_leaves_the_others_alone(H, prec, bad):
    n = 24
    a = torch.from_numpy(inputs.coeff_log_uniform(n, -1.0, 1.0, 4300)).cuda()
    f = torch.from_numpy(inputs.normal_rhs(n, 13, 4301)).cuda()
    with H.factor(n, 3, a, b_const=0.1, eps=1e-4, precision=prec) as h:
        u = torch.zeros_like(f)
        h.apply(f, u)
        f[5, 17] = bad
        v = torch.zeros_like(f)
        h.apply(f, v)
    keep = [c for c in range(13) if c != 5]
    assert torch.equal(u[keep], v[keep])
    assert not bool(torch.isfinite(v[5]).all())
