"""Leading-block Cholesky at the edges of its 16- and 64-column steps.

One level of cells of side m: every cell eliminates (m-1)^3 interior points or a
few more at the boundary (1 to 512), the root the separators, so p runs over 1, the
edges of the 16-column steps inside a 64 x 64 diagonal block, one block, several
blocks with a remainder, and more than 256.  eps = 0 makes F^{-1} A x = x up to
rounding.  With b = 1e4 the operator's condition number is below 3, so the
bounds are 200 roundings of each precision (FP32: 3xTF32 products, 22 bits).
"""
import numpy as np
import pytest

from oracle import stencil
from paper_1607_00346_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m", [2, 3, 4, 5, 6, 7, 9])
@pytest.mark.parametrize("prec,tc,bound", [(0, True, 200 * 2.0 ** -53), (0, False, 200 * 2.0 ** -53),
                                           (1, True, 200 * 2.0 ** -22), (1, False, 200 * 2.0 ** -24)])
def test_exact_elimination_to_rounding(m, prec, tc, bound):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_1607_00346_gb300 import hif
    n = 2 * m
    a = inputs.coeff_log_uniform(n, -0.3, 0.3, 6100 + n)
    A = stencil.assemble(a, 1e4, n)
    x = inputs.normal_rhs(n, 1, 6200 + n)[0]
    f = torch.from_numpy(A @ x).cuda()
    u = torch.zeros_like(f)
    with hif.factor(n, m, torch.from_numpy(a).cuda(), b_const=1e4, eps=0.0, precision=prec,
                    tensor_cores=tc) as h:
        h.apply(f, u)
    assert np.linalg.norm(u.cpu().numpy() - x) <= bound * np.linalg.norm(x)
