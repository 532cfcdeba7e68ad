"""The Gram-matrix ID of FP32 faces against the QR forms.

n = 32 has faces of about 240 DOFs (one CTA of 256 columns), n = 48 and 64 up to some
620 (clusters of 2 and 3, a ragged last CTA), with ranks from a few (eps = 0.3) over
several blocks of 64 pivots to every column (eps = 1e-9, below FP32 resolution).
The Gram form is at least as exact as FP32 QR, so its factor's solve error may
exceed the FP32 QR form's only by the products' own difference (3xTF32 against FMA,
22 against 24 bits: a factor 16 covers it), or reach the FP64 factor's.
"""
import numpy as np
import pytest

from oracle import stencil
from paper_1607_00346_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,m", [(32, 4), (48, 3), (64, 4)])
@pytest.mark.parametrize("eps", [0.3, 1e-3, 1e-6, 1e-9])
def test_gram_and_qr_skeletons(n, m, eps):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_1607_00346_gb300 import hif
    a = inputs.coeff_log_uniform(n, -1.0, 1.0, 8100 + n)
    A = stencil.assemble(a, 0.1, n)
    x = inputs.normal_rhs(n, 1, 8200 + n)[0]
    ax = torch.from_numpy(A @ x).cuda()
    ad = torch.from_numpy(a).cuda()
    err, kept = {}, {}
    for prec, tc in ((1, True), (1, False), (0, True)):
        u = torch.zeros_like(ax)
        with hif.factor(n, m, ad, b_const=0.1, eps=eps, precision=prec, tensor_cores=tc) as h:
            h.apply(ax, u)
            kept[prec, tc] = h.stats()["active_after"]
            if prec == 1 and tc:
                z = torch.zeros_like(ax)
                its, rel = h.solve(ax, z)
                assert rel[0] <= 1e-10
                true = np.linalg.norm(A @ z.cpu().numpy() - A @ x) / np.linalg.norm(A @ x)
                assert true <= 2e-10
        err[prec, tc] = np.linalg.norm(u.cpu().numpy() - x) / np.linalg.norm(x)
    assert err[1, True] <= max(16.0 * err[1, False], 2.0 * err[0, True]), (err, kept)
    if eps >= 1e-6:   # at 1e-9 FP32 noise decides what is kept
        for l, k in enumerate(kept[0, True]):
            assert abs(kept[1, True][l] - k) <= 0.01 * k, kept


def test_fronts_wider_than_1024_columns():
    # 96^3: the faces of the last level have up to 1141 DOFs, clusters of 256-column
    # CTAs (the levels below: 128-column CTAs); the bounds are those above
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_1607_00346_gb300 import hif
    n = 96
    a = inputs.coeff_log_uniform(n, -2.0, 2.0, 8300)
    A = stencil.assemble(a, 0.1, n)
    x = inputs.normal_rhs(n, 1, 8301)[0]
    ax = torch.from_numpy(A @ x).cuda()
    err, kept = {}, {}
    for tc in (True, False):
        u = torch.zeros_like(ax)
        with hif.factor(n, 3, torch.from_numpy(a).cuda(), b_const=0.1, eps=1e-6, precision=1,
                        tensor_cores=tc) as h:
            h.apply(ax, u)
            kept[tc] = h.stats()["active_after"]
        err[tc] = np.linalg.norm(u.cpu().numpy() - x) / np.linalg.norm(x)
    assert err[True] <= 16.0 * err[False], (err, kept)
    for k, q in zip(kept[True], kept[False]):
        assert abs(k - q) <= 0.01 * q, kept
