"""The work that users of the library have it do, as cases that can be timed.

Every case goes through the Python binding of the C ABI
(``paper_1607_00346_gb300.hif``) with device arrays: a factorization followed
by the preconditioned solve, a solve with a resident factor, the solve of
several resident operators together, an apply, a residual.  Grid sizes, leaf
sizes, tolerances, right-hand-side counts and coefficient laws are those of
the workloads of ``inputs.py``, of the serving loop and of the tests.

Solves stop at a relative residual of 1e-12, the tolerance at which the
paper's own solver stops.
"""
import numpy as np
import torch

from paper_1607_00346_gb300 import hif

TOL = 1e-12

# (n, m): n = m 2^L points per dimension with a leaf cell of side m
GRIDS = [(16, 4), (20, 5), (24, 3), (32, 4), (40, 5), (48, 3), (64, 4), (80, 5), (96, 3)]


def _case(name, kind, n, m, precision, eps, nrhs, span, b, periodic=False):
    """a = 10^U(-span, span) per grid point, b constant, N(0,1) right-hand sides."""
    return {"name": name, "kind": kind, "n": n, "m": m, "precision": precision, "eps": eps,
            "nrhs": nrhs, "span": span, "b": b, "periodic": periodic}


def _batch(name, systems, eps, span):
    """systems: "n/m/nrhs" of each resident operator, separated by blanks."""
    return {"name": name, "kind": "batch", "systems": systems, "precision": "fp32", "eps": eps,
            "span": span, "b": 0.0, "periodic": False}


def listed():
    return [
        # the smallest problem of the workloads: plain double, the Laplacian;
        # latency and launches count
        _case("factor_solve_16_fp64", "factor_solve", 16, 4, "fp64", 1e-6, 1, 0.0, 0.0),
        # the paper's Example 1 on its own periodic grid (b = 0.1 against the
        # stencil without its 1/h^2)
        _case("factor_solve_32_periodic", "factor_solve", 32, 4, "fp64", 1e-3, 1, 0.0,
              0.1 * 32 * 32, True),
        # the double-precision workload of medium size, eight right-hand sides
        _case("factor_solve_64_fp64", "factor_solve", 64, 4, "fp64", 1e-4, 8, 1.0, 0.0),
        # two requests of the serving mix whose operators are not resident
        # (leaf cells of side 3, odd numbers of right-hand sides)
        _case("factor_solve_48_fp32", "factor_solve", 48, 3, "fp32", 1e-6, 5, 2.0, 0.0),
        _case("factor_solve_96_fp32", "factor_solve", 96, 3, "fp32", 1e-6, 11, 2.0, 0.0),
        # the benchmark workload: a large operator factored and solved once
        _case("factor_solve_128_fp32", "factor_solve", 128, 4, "fp32", 1e-6, 1, 1.0, 0.1),
        # a resident operator asked for one solution: the smallest of the
        # serving mix, and the largest with as many columns as a request has
        _case("solve_32_fp32", "solve", 32, 4, "fp32", 1e-6, 1, 2.0, 0.0),
        _case("solve_128_fp32", "solve", 128, 4, "fp32", 1e-6, 16, 1.0, 0.1),
        # waiting requests of four resident operators solved together
        _batch("solve_batch", "32/4/1 48/3/5 64/4/16 96/3/3", 1e-6, 2.0),
        # F^{-1} used inside a caller's own iteration, in double
        _case("apply_64_fp64", "apply", 64, 4, "fp64", 1e-6, 8, 1.0, 0.0),
        # the residual in double that such an iteration asks for
        _case("residual_128", "residual", 128, 4, "fp32", 1e-3, 3, 1.0, 0.1),
    ]


def draw(rng):
    kind = rng.choice(["factor_solve", "factor_solve", "factor_solve", "factor_solve", "solve",
                       "solve", "batch", "apply", "residual"])
    eps = rng.choice([1e-3, 1e-4, 1e-6])
    span = rng.choice([1.0, 1.5, 2.0])
    if kind == "batch":
        systems = " ".join("%d/%d/%d" % (*rng.choice(GRIDS[2:]), rng.randint(1, 16))
                           for _ in range(rng.randint(2, 5)))
        c = _batch("", systems, min(eps, 1e-4), span)
        del c["name"]
        return c
    precision = rng.choice(["fp64", "fp32"]) if kind != "apply" else "fp64"
    most = 64 if precision == "fp64" else 96
    n, m = rng.choice([g for g in GRIDS if g[0] <= most])
    periodic = kind == "factor_solve" and n <= 24 and rng.random() < 0.5
    b = rng.choice([0.0, 0.1, 1.0, rng.uniform(0.0, 10.0)])
    if periodic:
        b = 0.1 * n * n
    nrhs = rng.choice([1, rng.randint(1, 16)])
    c = _case("", kind, n, m, precision, eps, nrhs, span, b, periodic)
    del c["name"]
    return c


# ---- inputs -------------------------------------------------------------------


def _systems(case):
    """The (n, m, nrhs) of every operator of the case."""
    if case["kind"] == "batch":
        return [tuple(int(v) for v in s.split("/")) for s in case["systems"].split()]
    return [(case["n"], case["m"], case["nrhs"])]


def _inputs(case, seed, k):
    """Coefficient, right-hand sides and (for the residual) an iterate of operator k."""
    n, _, nrhs = _systems(case)[k]
    g = torch.Generator(device="cuda")
    g.manual_seed(1000003 * (seed + 1) + k)
    kw = dict(generator=g, device="cuda", dtype=torch.float64)
    a = torch.pow(10.0, (2.0 * torch.rand(n ** 3, **kw) - 1.0) * case["span"])
    f = torch.randn(nrhs, n ** 3, **kw)
    u = torch.randn(nrhs, n ** 3, **kw) if case["kind"] == "residual" else torch.zeros_like(f)
    return a, f, u


def _options(case):
    return dict(b_const=case["b"], eps=case["eps"],
                precision=hif.PREC_FP64 if case["precision"] == "fp64" else hif.PREC_FP32,
                pcg_tol=TOL, periodic=case["periodic"])


def prepare(case, seed):
    """Inputs on the device; for every kind but factor_solve the resident factors too."""
    state = {"kind": case["kind"], "a": [], "f": [], "u": [], "grid": _systems(case),
             "options": _options(case), "h": []}
    for k, (n, m, _) in enumerate(state["grid"]):
        a, f, u = _inputs(case, seed, k)
        state["a"].append(a)
        state["f"].append(f)
        state["u"].append(u)
        if case["kind"] != "factor_solve":
            state["h"].append(hif.factor(n, m, a, **state["options"]))
    if case["kind"] == "residual":
        state["r"] = torch.empty_like(state["f"][0])
    return state


def run(state):
    kind, f, u = state["kind"], state["f"], state["u"]
    if kind == "factor_solve":
        n, m, _ = state["grid"][0]
        with hif.factor(n, m, state["a"][0], **state["options"]) as h:
            h.solve(f[0], u[0])
        return u[0]
    if kind == "solve":
        state["h"][0].solve(f[0], u[0])
        return u[0]
    if kind == "batch":
        hif.solve_batch(state["h"], f, u)
        return u
    if kind == "apply":
        return state["h"][0].apply(f[0], u[0])
    return state["h"][0].residual(f[0], u[0], state["r"])


# ---- counts --------------------------------------------------------------------


def work(case):
    """Fits to the library's own counts of a factorization's flops and of the
    factor's entries (within about 25% for m = 3 to 5; a looser tolerance needs
    less, the periodic grid's larger fronts more).  A solve reads the factor
    twice per iteration, an apply twice."""
    double = case["precision"] == "fp64"
    size = 8 if double else 4
    less = {1e-6: 1.0, 1e-4: 0.6, 1e-3: 0.45}[case["eps"]]
    iters = {1e-6: 3 if double else 5, 1e-4: 5, 1e-3: 6}[case["eps"]]
    total_bytes = total_flops = 0.0
    for n, _, nrhs in _systems(case):
        N = float(n) ** 3
        entries = 250.0 * N * (n / 16.0) ** 0.8 * less ** 0.5 * (3.0 if case["periodic"] else 1.0)
        factor = 2.15e8 * (n / 16.0) ** 5.25 * less * (9.0 if case["periodic"] else 1.0)
        vectors = 8.0 * N * nrhs
        if case["kind"] == "residual":
            total_bytes += 8.0 * N * 4 + 3.0 * vectors
            total_flops += 14.0 * N * nrhs
        elif case["kind"] == "apply":
            total_bytes += 2.0 * size * entries + 2.0 * vectors
            total_flops += 4.0 * entries * nrhs
        elif case["kind"] == "factor_solve":
            total_bytes += 8.0 * N + size * entries + 2.0 * vectors
            total_flops += factor + iters * (4.0 * entries + 24.0 * N) * nrhs
        else:
            total_bytes += iters * 2.0 * size * entries + 8.0 * N * 4 + 2.0 * vectors
            total_flops += iters * (4.0 * entries + 24.0 * N) * nrhs
    return {"bytes": total_bytes, "flops": total_flops}


# ---- the same results in plain 64-bit arithmetic -----------------------------------


class _Operator:
    """The seven-point operator on an n^3 grid (last axis fastest)."""

    def __init__(self, a, b, n, periodic):
        a = a.reshape(n, n, n)
        inv_h2 = float(n if periodic else n + 1) ** 2
        self.periodic, self.c, self.diag = periodic, [], torch.full_like(a, b)
        for d in (2, 1, 0):
            nxt = torch.roll(a, -1, d)
            up = 2.0 * a * nxt / (a + nxt)
            if not periodic:
                last = up.narrow(d, n - 1, 1)
                last.copy_(a.narrow(d, n - 1, 1))
            down = torch.roll(up, 1, d)
            if not periodic:
                down.narrow(d, 0, 1).copy_(a.narrow(d, 0, 1))
            self.diag += (up + down) * inv_h2
            up = up * inv_h2
            if not periodic:
                up.narrow(d, n - 1, 1).zero_()
            self.c.append((d + 1, up, torch.roll(up, 1, d)))

    def __call__(self, u):
        v = self.diag * u
        for d, up, down in self.c:   # a zero coupling takes the wrapped value out
            v -= up * torch.roll(u, -1, d)
            v -= down * torch.roll(u, 1, d)
        return v

    def solve(self, f):
        """Conjugate gradients with the diagonal, restarted from the true residual."""
        u = torch.zeros_like(f)
        dot = lambda x, y: (x * y).sum(dim=(1, 2, 3), keepdim=True)  # noqa: E731
        norm = dot(f, f)
        for _ in range(3):
            r = f - self(u)
            z = r / self.diag
            p, rz = z.clone(), dot(r, z)
            for k in range(1, 4001):
                q = self(p)
                al = rz / dot(p, q)
                u += al * p
                r -= al * q
                if k % 50 == 0 and bool((dot(r, r) <= 1e-30 * norm).all()):
                    break
                z = r / self.diag
                new = dot(r, z)
                p = z + (new / rz) * p
                rz = new
        return u


def exact(case, seed):
    """A^{-1} f for the solves and the applies (an apply is as far from it as the
    tolerance of its factor lets it be), f - A u for the residual."""
    outs = []
    for k, (n, _, nrhs) in enumerate(_systems(case)):
        a, f, u = _inputs(case, seed, k)
        A = _Operator(a, case["b"], n, case["periodic"])
        f3 = f.reshape(nrhs, n, n, n)
        if case["kind"] == "residual":
            out = f3 - A(u.reshape(nrhs, n, n, n))
        else:
            out = A.solve(f3)
        outs.append(out.reshape(nrhs, n ** 3).cpu().numpy().astype(np.float64))
    return outs if case["kind"] == "batch" else outs[0]
