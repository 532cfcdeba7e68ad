"""Arrays shared between the systems of a batch.

hif_apply_batch reads every right-hand side before it writes any solution, and
hif_solve_batch reads a right-hand side before a later system clears its solution,
so a solution may go to another system's right-hand side; results are bitwise those
of separate arrays.  The systems differ in size of the factor (leaf cells, tolerance)
so that their streams run at different speeds, the widest last and first.
"""
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


# 24^3 throughout; (leaf cell, tolerance) of the three operators
KINDS = [(3, 1e-2), (6, 1e-6), (12, 1e-4)]


def _factors(H, prec):
    hs = []
    for k, (m, eps) in enumerate(KINDS):
        a = torch.from_numpy(inputs.coeff_log_uniform(24, -1.0, 1.0, 8100 + k)).cuda()
        hs.append(H.factor(24, m, a, b_const=0.1, eps=eps, precision=prec))
    return hs


def _rhs(nrhs):
    return [torch.from_numpy(inputs.normal_rhs(24, nrhs, 8200 + k)).cuda() for k in range(3)]


# (right-hand side of each system, solution of each system) as buffer numbers; buffers
# 0-2 hold the right-hand sides
@pytest.mark.parametrize("fi,ui", [
    ([0, 1, 2], [1, 2, 0]),    # a ring
    ([0, 1, 2], [2, 0, 1]),    # and the other way round
    ([0, 1, 2], [1, 0, 2]),    # two exchanged, one in place
    ([0, 0, 0], [0, 1, 2]),    # a shared right-hand side, in place in the first system
    ([0, 0, 0], [3, 4, 0]),    # and in the last
])
@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("nrhs", [1, 9])
def test_apply_batch_reads_before_it_writes(H, fi, ui, prec, nrhs):
    hs, f = _factors(H, prec), _rhs(nrhs)
    want = [torch.empty_like(f[0]) for _ in hs]
    for h, i, w in zip(hs, fi, want):
        h.apply(f[i], w)
    for _ in range(3):
        buf = [x.clone() for x in f] + [torch.empty_like(f[0]) for _ in range(2)]
        H.apply_batch(hs, [buf[i] for i in fi], [buf[i] for i in ui])
        for i, w in zip(ui, want):
            assert torch.equal(buf[i], w)


@pytest.mark.parametrize("fi,ui", [
    ([0, 1, 2], [3, 0, 1]),    # each solution over the right-hand side before it
    ([0, 1, 2], [3, 4, 0]),
    ([0, 0, 2], [3, 4, 0]),
])
@pytest.mark.parametrize("prec", [0, 1])
def test_solve_batch_reads_before_a_later_system_writes(H, fi, ui, prec):
    hs, f = _factors(H, prec), _rhs(5)
    want, its = [torch.empty_like(f[0]) for _ in hs], []
    for h, i, w in zip(hs, fi, want):
        its.append(h.solve(f[i], w)[0])
    for _ in range(3):
        buf = [x.clone() for x in f] + [torch.empty_like(f[0]) for _ in range(2)]
        got = H.solve_batch(hs, [buf[i] for i in fi], [buf[i] for i in ui])
        for i, w, a, b in zip(ui, want, its, got):
            assert torch.equal(buf[i], w)
            assert list(a) == list(b[0])
