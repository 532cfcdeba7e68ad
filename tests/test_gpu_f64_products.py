"""FP64 products on the tensor cores (8-bit slices, exact sums) against the FMA form.

eps = 0 (exact elimination) makes F^{-1} A x = x up to rounding, so the solve
error measures the arithmetic alone.  The sliced products round once per entry,
the FMA form once per multiply-add; the rest of the factorization is the same,
so the sliced error may not exceed the FMA form's by more than the spread of
two runs of rounding (a factor 2), and stays within the FP64 tolerance of the
exact mode (1e-10; coefficients over up to six decades).  The sizes give
products from 1 x 1 x 1 to several 128 x 64 tiles, ragged in every dimension,
with each of the triangular operands.
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


def _error(H, n, m, a, x, ax, eps, **kw):
    u = torch.zeros(n ** 3, dtype=torch.float64, device="cuda")
    with H.factor(n, m, torch.from_numpy(a).cuda(), b_const=0.1, eps=eps, **kw) as h:
        h.apply(torch.from_numpy(ax).cuda(), u)
    return np.linalg.norm(u.cpu().numpy() - x) / np.linalg.norm(x)


@pytest.mark.parametrize("n,m", [(8, 4), (14, 7), (18, 9), (20, 5), (24, 3), (28, 7)])
@pytest.mark.parametrize("span", [0.5, 2.0, 3.0])
def test_sliced_products_err_no_more_than_fma(H, n, m, span):
    a = inputs.coeff_log_uniform(n, -span, span, 5100 + n)
    A = stencil.assemble(a, 0.1, n)
    x = inputs.normal_rhs(n, 1, 5200 + n)[0]
    ax = A @ x
    err = {tc: _error(H, n, m, a, x, ax, 0.0, tensor_cores=tc) for tc in (True, False)}
    assert err[False] < 1e-10 and err[True] < 1e-10, err
    assert err[True] <= 2.0 * err[False] + 1e-15, err


def test_sliced_products_in_the_skeletonized_factor(H):
    # eps > 0: row reduction and skeleton products as well; the error is eps's
    n = 32
    a = inputs.coeff_log_uniform(n, -1.0, 1.0, 5300)
    A = stencil.assemble(a, 0.1, n)
    x = inputs.normal_rhs(n, 1, 5301)[0]
    ax = A @ x
    err = {tc: _error(H, n, 4, a, x, ax, 1e-6, tensor_cores=tc) for tc in (True, False)}
    assert abs(err[True] - err[False]) <= 1e-3 * err[False], err


@pytest.mark.parametrize("n,m,eps", [(32, 4, 1e-6), (48, 3, 1e-4)])
def test_sliced_and_fma_factors_are_the_same_operator(H, n, m, eps):
    # the row reduction's reflectors shrink by ten decades and more; rounding of
    # either form moves F^{-1} f by the condition number (1e5) times 2^-53
    a = torch.from_numpy(inputs.coeff_log_uniform(n, -1.0, 1.0, 5400 + n)).cuda()
    f = torch.from_numpy(inputs.normal_rhs(n, 1, 5500 + n)).cuda()
    u = {}
    for tc in (True, False):
        u[tc] = torch.zeros_like(f)
        with H.factor(n, m, a, b_const=0.1, eps=eps, tensor_cores=tc) as h:
            h.apply(f, u[tc])
    assert float(torch.linalg.norm(u[True] - u[False]) / torch.linalg.norm(u[False])) <= 1e-11
