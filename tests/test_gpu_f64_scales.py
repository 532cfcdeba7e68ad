"""FP64 products as slices where the coefficients have structure: blocks, layers, a ramp.

A slice holds an entry in fixed point below the largest entry of its row, so a soft
region's entries must not share a scale with a stiff one's.  eps = 0 makes the factor
exact up to rounding; the right-hand side A x with x of O(1) everywhere shows the
rounding of every region at its own scale.  The reference is the same system solved in
extended precision: the GPU's own operator (read off its residual), and the FMA
factor's solution refined with residuals in extended precision until it stands still.

Both forms round at 2^-53 of the same quantities, so the sliced form may err by no more
than twice the FMA form's error (the spread of two runs of rounding, as in
test_gpu_f64_products), with a floor of 1e-15.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

LD = np.longdouble


@pytest.fixture(scope="module")
def H():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_1607_00346_gb300 import hif
    hif.load()
    return hif


def _field(kind, n, decades, seed):
    rng = np.random.default_rng(seed)
    i = np.arange(n ** 3)
    x, y, z = i % n, i // n % n, i // (n * n)
    half = 0.5 * decades
    if kind == "ramp":
        return 10.0 ** (half * (2.0 * x / (n - 1) - 1.0)) * rng.uniform(0.9, 1.1, n ** 3)
    if kind == "iid":
        return 10.0 ** rng.uniform(-half, half, n ** 3)
    stiff = {"blocks": (x // 10 + y // 10 + z // 10) % 2 == 0,
             "layers": z // 5 % 2 == 0,
             "holes": ~((x % 7 < 3) & (y % 7 < 3) & (z % 7 < 3))}[kind]
    return np.where(stiff, 10.0 ** half, 10.0 ** -half) * rng.uniform(0.9, 1.1, n ** 3)


def _operator(h, n):
    """The diagonal and the couplings to +x, +y, +z, from residuals of seven colours
    (a point and its six neighbours all differ)."""
    N = n ** 3
    i = np.arange(N)
    x, y, z = i % n, i // n % n, i // (n * n)
    colour = (x + 2 * y + 3 * z) % 7
    f = torch.zeros(1, N, dtype=torch.float64, device="cuda")
    r = torch.empty_like(f)
    R = np.empty((7, N))
    for c in range(7):
        h.residual(f, torch.from_numpy((colour == c).astype(np.float64)).cuda().reshape(1, N), r)
        R[c] = r.cpu().numpy()[0]
    up = []
    for d, p in ((1, x), (2, y), (3, z)):
        v = R[(colour + d) % 7, i].copy()
        v[p == n - 1] = 0.0
        up.append(v.astype(LD))
    return -R[colour, i].astype(LD), up


def _matvec(op, n, u):
    diag, up = op
    s = diag * u
    for c, st in zip(up, (1, n, n * n)):
        s[:-st] -= c[:-st] * u[st:]
        s[st:] -= c[:-st] * u[:-st]
    return s


def _errors(H, kind, n, m, decades, seed):
    """Errors of the FMA and of the sliced factor's solution, in 2-norm and max-norm."""
    N = n ** 3
    a = torch.from_numpy(_field(kind, n, decades, seed)).cuda()
    x = np.random.default_rng(seed + 1).uniform(0.5, 1.5, N) * np.random.default_rng(seed + 2).choice([-1, 1], N)
    u = torch.empty(1, N, dtype=torch.float64, device="cuda")
    got = []
    with H.factor(n, m, a, b_const=0.1, eps=0.0, tensor_cores=False) as h:
        op = _operator(h, n)
        f = _matvec(op, n, x.astype(LD)).astype(np.float64)

        def apply(h, v):
            h.apply(torch.from_numpy(v.astype(np.float64)).cuda().reshape(1, N), u)
            return u.cpu().numpy()[0].astype(LD)

        got.append(apply(h, f))
        ref = got[0].copy()
        for _ in range(6):
            step = apply(h, f.astype(LD) - _matvec(op, n, ref))
            ref += step
        assert float(np.linalg.norm(step.astype(np.float64))) <= 1e-18 * float(np.linalg.norm(ref.astype(np.float64)))
    with H.factor(n, m, a, b_const=0.1, eps=0.0, tensor_cores=True) as h:
        got.append(apply(h, f))
    ref64 = ref.astype(np.float64)
    return [(np.linalg.norm(e) / np.linalg.norm(ref64), np.abs(e).max() / np.abs(ref64).max())
            for e in ((g - ref).astype(np.float64) for g in got)]


@pytest.mark.parametrize("kind", ["blocks", "layers", "holes", "ramp", "iid"])
@pytest.mark.parametrize("decades", [2, 3.5, 4, 6])
@pytest.mark.parametrize("n,m", [(20, 5), (28, 7), (32, 4)])
def test_sliced_products_keep_the_scales_of_soft_and_stiff_regions(H, kind, n, m, decades):
    fma, sliced = _errors(H, kind, n, m, decades, 7000 + n)
    for e0, e1 in zip(fma, sliced):
        assert e1 <= 2.0 * e0 + 1e-15, (fma, sliced)
