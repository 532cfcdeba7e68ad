"""Edges of the conjugate-gradient kernels: finished columns, limits, sizes.

The kernels' sums run over blocks of 1024 points, so the sizes have one partial
block (8^3), a ragged last block (9 = 9 * 1: n = 18, 20) and several.  Solutions are
checked with the oracle's operator: the iteration stops at ||r|| <= 1e-10 ||f||,
and the recursively updated residual differs from the true one by rounding
(condition number below 1e4 here), so the true one is held to 2e-10.
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


def _system(H, n, m, prec, **kw):
    a = inputs.coeff_log_uniform(n, -0.5, 0.5, 7100 + n)
    h = H.factor(n, m, torch.from_numpy(a).cuda(), b_const=1.0, eps=1e-4, precision=prec, **kw)
    return h, stencil.assemble(a, 1.0, n)


@pytest.mark.parametrize("n,m", [(8, 4), (18, 9), (20, 5), (24, 3)])
@pytest.mark.parametrize("prec", [0, 1])
def test_zero_and_easy_columns_finish_alone(H, n, m, prec):
    h, A = _system(H, n, m, prec)
    f = inputs.normal_rhs(n, 5, 7200 + n)
    f[1] = 0.0
    f[3] *= 1e-200                       # squares of its entries underflow: norm 0
    f[4] = A @ np.ones(n ** 3)
    fd = torch.from_numpy(f).cuda()
    u = torch.full_like(fd, float("nan"))
    its, rel = h.solve(fd, u)
    uc = u.cpu().numpy()
    assert its[1] == 0 and rel[1] == 0.0 and not uc[1].any()
    assert its[3] == 0 and rel[3] == 0.0 and not uc[3].any()
    for c in (0, 2, 4):
        assert its[c] >= 1 and rel[c] <= 1e-10
        assert np.linalg.norm(f[c] - A @ uc[c]) <= 2e-10 * np.linalg.norm(f[c])
    # each column is the one it gets alone
    for c in (0, 2, 4):
        one = torch.zeros_like(fd[c:c + 1])
        i1, _ = h.solve(fd[c:c + 1].clone(), one)
        assert i1[0] == its[c] and torch.equal(one[0], u[c])
    h.close()


@pytest.mark.parametrize("limit", [0, 1])
def test_iteration_limit(H, limit):
    n = 16
    h, A = _system(H, n, 4, 1, max_iter=limit)
    f = inputs.normal_rhs(n, 2, 7300)
    fd = torch.from_numpy(f).cuda()
    u = torch.full_like(fd, float("nan"))
    with pytest.raises(H.HifError) as e:
        h.solve(fd, u)
    assert e.value.status == 4           # HIF_ERR_NO_CONVERGENCE
    its, rel = h.solve(fd, u, check=False)
    assert its == [limit, limit]
    uc = u.cpu().numpy()
    for c in range(2):
        true = np.linalg.norm(f[c] - A @ uc[c]) / np.linalg.norm(f[c])
        assert abs(true - rel[c]) <= 1e-12 + 1e-6 * rel[c]
    # an all-zero system converges without an iteration
    z = torch.zeros_like(fd)
    its, rel = h.solve(z, u)
    assert its == [0, 0] and rel == [0.0, 0.0] and not bool(u.any())
    h.close()
