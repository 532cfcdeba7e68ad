"""Device memory of a factorization: the counted peak and the predicted one.

stats()["peak_bytes"] counts the work space of the products and of the Gram form too, so
it is at least what the stream-ordered pool held at its fullest (its lists of fronts
and products, a few tens of bytes each, are not counted: 1% and 1 MiB are allowed for
them).  hif_predict_bytes is an upper estimate of it: for the admission of a
factorization an estimate below the peak is wrong at any margin.
"""
import ctypes

import pytest

from paper_1607_00346_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

USED_MEM_HIGH = 8   # cudaMemPoolAttrUsedMemHigh


@pytest.fixture(scope="module")
def H():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_1607_00346_gb300 import hif
    hif.load()
    return hif


class _Pool:
    def __init__(self):
        torch.zeros(1, device="cuda")
        try:
            self.rt = ctypes.CDLL("libcudart.so.%s" % torch.version.cuda.split(".")[0])
        except OSError:
            pytest.skip("no CUDA runtime library to ask")
        self.pool = ctypes.c_void_p()
        assert self.rt.cudaDeviceGetDefaultMemPool(ctypes.byref(self.pool), 0) == 0

    def reset(self):
        torch.cuda.synchronize()
        v = ctypes.c_uint64(0)
        assert self.rt.cudaMemPoolSetAttribute(self.pool, USED_MEM_HIGH, ctypes.byref(v)) == 0

    def high(self):
        v = ctypes.c_uint64()
        assert self.rt.cudaMemPoolGetAttribute(self.pool, USED_MEM_HIGH, ctypes.byref(v)) == 0
        return v.value


@pytest.mark.parametrize("n,m,prec,eps,periodic", [
    (16, 4, 0, 1e-6, True), (20, 5, 0, 0.0, True), (24, 3, 1, 1e-3, True),
    (32, 4, 1, 1e-4, False), (32, 4, 0, 1e-3, False),
    (48, 3, 1, 1e-6, False), (48, 3, 1, 1e-3, False), (48, 12, 0, 1e-6, False),
    (64, 4, 1, 1e-6, False), (64, 4, 1, 1e-4, False), (64, 4, 0, 1e-4, False),
    (64, 8, 0, 0.0, False), (96, 3, 1, 1e-6, False), (96, 3, 1, 1e-4, False),
])
def test_peak_counts_the_work_space_and_is_predicted(H, n, m, prec, eps, periodic):
    pool = _Pool()
    a = torch.from_numpy(inputs.coeff_log_uniform(n, -1.0, 1.0, 9100 + n)).cuda()
    pool.reset()
    with H.factor(n, m, a, b_const=0.1 * (n * n if periodic else 1), eps=eps, precision=prec,
                  periodic=periodic) as h:
        peak = h.stats()["peak_bytes"]
    assert peak >= 0.99 * pool.high() - (1 << 20)
    assert peak <= H.predict_bytes(n, m, periodic=periodic, eps=eps, precision=prec)
