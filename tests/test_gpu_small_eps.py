"""FP32 factors with tolerances near and below what their ID can resolve.

Below eps 1e-7 the pivots of the Gram form are noise; such factors take the row
reduction and the pivoted QR.  The solve error with tensor cores is 7 to 11 times that
of the FMA form (the 3xTF32 products), 12 times allowed, whatever the eps; the solve
converges.  eps = 1e-7 is the least that takes the Gram form.
"""
import numpy as np
import pytest

from oracle import stencil
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


@pytest.mark.parametrize("n,m,span,eps", [(48, 3, 2.0, 1e-7), (48, 3, 2.0, 9.9e-8), (64, 4, 1.0, 1e-10),
                                          (48, 3, 2.0, 1e-12), (64, 4, 2.0, 1e-12)])
def test_fp32_factor_with_a_small_eps(H, n, m, span, eps):
    a = inputs.coeff_log_uniform(n, -span, span, 31)
    A = stencil.assemble(a, 0.1, n)
    x = inputs.normal_rhs(n, 1, 32)[0]
    ax = torch.from_numpy(A @ x).cuda()
    f = torch.from_numpy(inputs.normal_rhs(n, 2, 33)).cuda()
    es = {}
    for tc in (True, False):
        u, v = torch.empty_like(ax), torch.zeros_like(f)
        with H.factor(n, m, torch.from_numpy(a).cuda(), b_const=0.1, eps=eps, precision=1, tensor_cores=tc) as h:
            h.apply(ax, u)
            its, rel = h.solve(f, v)
        es[tc] = np.linalg.norm(u.cpu().numpy() - x) / np.linalg.norm(x)
        assert max(rel) <= 1e-10
    assert es[True] <= 12.0 * es[False], es
