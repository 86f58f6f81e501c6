"""The solves that a user of this framework runs, as timed cases.

A case is one call (or one short sequence of calls) of the public binding
``paper_1612_04846_gb300.bura`` on a plan that the program keeps:

* ``solve``: ``bura_solve`` of one right-hand side on the device, on a 2-D or 3-D grid with constant or block
  log-uniform coefficients, in mixed precision (the default), with double-float refinement or in FP64;
* ``csr``: ``bura_solve`` with an assembled P1 finite-element matrix (a half-cube coefficient jump);
* ``sum``: ``bura_solve_sum`` of a sinc quadrature whose nodes are spread over several ``bura_setup_shifts`` plans;
* ``batch``: many 2-D problems captured as one graph, ``BuraBatch.run`` + ``wait``;
* ``serve``: what a request of a serving loop costs: ``bura_retarget`` of a resident plan and ``bura_solve_host``.

``exact`` gives the same values in 64 bits: the sine eigenbasis where the operator is constant, else a conjugate
gradient method of its own for every shifted system.  The weights and shifts of the best uniform rational
approximation are read from the committed high-precision table, so alpha takes the table's values.
"""
import json
import math

import numpy as np
import torch

from paper_1612_04846_gb300 import bura

ALPHAS = (0.1, 0.25, 0.5, 0.75, 0.9)  # the powers the committed coefficient table holds
DEV = "cuda"


def listed():
    return [
        # the smallest solve of a batch or a server: nothing but launches and latency
        dict(name="solve_63x63", kind="solve", nx=63, ny=63, nz=0, var=False, prec="mixed", alpha=0.5, k=5, tol=1e-6),
        # a serving loop's request on a small grid, host arrays in and out, alpha changing from request to request
        dict(name="serve_127x127", kind="serve", nx=127, ny=127, nz=0, var=False, prec="mixed", alpha=0.25, k=6, tol=1e-6),
        # an ordinary 2-D solve on a grid that is neither square nor a multiple of any tile
        dict(name="solve_383x255", kind="solve", nx=383, ny=255, nz=0, var=False, prec="mixed", alpha=0.25, k=8, tol=1e-6),
        # the headline workload of bench.py
        dict(name="solve_1023x1023", kind="solve", nx=1023, ny=1023, nz=0, var=False, prec="mixed", alpha=0.5, k=7, tol=1e-6),
        # the quadrature comparison (plans of caller-given shifts summed), at the tolerance of bench.py's comparison
        dict(name="sum_511x511", kind="sum", nx=511, ny=511, nz=0, var=False, prec="mixed", alpha=0.5, kprime=0.7, tol=1e-8),
        # 2-D with a variable coefficient field, as the serving mix has it
        dict(name="solve_var_511x511", kind="solve", nx=511, ny=511, nz=0, var=True, prec="mixed", alpha=0.75, k=6, tol=1e-6),
        # the FP64 path (no mixed precision), for users who ask for it
        dict(name="fp64_511x511", kind="solve", nx=511, ny=511, nz=0, var=False, prec="fp64", alpha=0.5, k=7, tol=1e-6),
        # 3-D, constant coefficients, ragged axes
        dict(name="solve_127x95x63", kind="solve", nx=127, ny=95, nz=63, var=False, prec="mixed", alpha=0.5, k=8, tol=1e-6),
        # 3-D with a variable field at a serving size
        dict(name="solve_var_63x63x63", kind="solve", nx=63, ny=63, nz=63, var=True, prec="mixed", alpha=0.25, k=5, tol=1e-6),
        # the largest single solve: 16.6 million unknowns, 10 shifted systems, variable coefficients
        dict(name="solve_var_255x255x255", kind="solve", nx=255, ny=255, nz=255, var=True, prec="mixed", alpha=0.5, k=9, tol=1e-6),
        # an assembled sparse matrix
        dict(name="csr_63x63x63", kind="csr", nx=63, ny=63, nz=63, var=True, prec="mixed", alpha=0.5, k=7, tol=1e-6),
        # many independent problems of mixed sizes, powers and degrees in one graph launch
        dict(name="batch_32", kind="batch", count=32, nmax=511, tol=1e-6),
    ]


def _axis(rng, lo, hi):
    """An axis length q * 2^p - 1 in [lo, hi], spread over the logarithm: odd, and coarsenable p times."""
    while True:
        n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
        p = rng.randint(3, 8)
        q = max(1, int(round((n + 1) / 2.0 ** p)))
        n = q * 2 ** p - 1
        if lo <= n <= hi and q <= 8:
            return n


def draw(rng):
    kind = rng.choice(("solve2", "solve2", "solve2", "var2", "var2", "fp64", "solve3", "var3", "var3", "csr", "sum", "batch", "serve"))
    c = dict(kind="solve", nx=0, ny=0, nz=0, var=False, prec="mixed", alpha=rng.choice(ALPHAS), k=rng.randint(5, 9), tol=1e-6)
    if kind in ("solve2", "var2", "fp64", "sum"):
        top = 1023 if kind in ("solve2", "var2") else 511
        c["nx"] = _axis(rng, 31, top)
        c["ny"] = c["nx"] if rng.random() < 0.4 else _axis(rng, max(31, c["nx"] // 4), min(top, 4 * c["nx"]))
        c["var"] = kind == "var2"
        if kind == "fp64":
            c["prec"] = "fp64"
        elif kind == "solve2" and rng.random() < 0.2:
            c["prec"] = "df"
        elif kind == "sum":
            c.update(kind="sum", kprime=rng.choice((0.6, 0.7, 0.8)), tol=1e-8, alpha=rng.choice(ALPHAS[1:4]))
            del c["k"]
    elif kind in ("solve3", "var3"):
        c["nx"] = _axis(rng, 15, 191)
        for a in ("ny", "nz"):
            c[a] = c["nx"] if rng.random() < 0.4 else _axis(rng, max(15, c["nx"] // 3), min(191, 3 * c["nx"]))
        c["var"] = kind == "var3"
    elif kind == "csr":
        n = rng.choice((15, 23, 31, 40, 47, 55, 63))
        c.update(kind="csr", nx=n, ny=n, nz=n, var=True)
    elif kind == "batch":
        c = dict(kind="batch", count=rng.randint(8, 48), nmax=rng.choice((127, 255, 511)), tol=1e-6)
    else:
        c.update(kind="serve", nx=_axis(rng, 31, 511))
        c["ny"] = c["nx"]
    return c


# ---------------------------------------------------------------------- inputs
def _gen(seed, salt):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 1000003 + salt)
    return g


def _rhs(n, seed, salt=0):
    """f i.i.d. uniform on [-1, 1]."""
    return torch.rand(n, generator=_gen(seed, salt), dtype=torch.float64, device=DEV) * 2 - 1


def _shape(case):
    return (case["nx"], case["ny"]) if not case["nz"] else (case["nx"], case["ny"], case["nz"])


def _faces(shape, seed):
    """Face coefficients (device arrays, x fastest) of a field that is log-uniform on [1e-2, 1] per block of 8^d blocks."""
    d = len(shape)
    lo = math.log(1e-2)
    field = torch.exp(lo * torch.rand((8,) * d, generator=_gen(seed, 77), dtype=torch.float64, device=DEV))
    out = []
    for axis in range(d):  # 0: x-faces, ...
        a = field
        for dim in range(d):  # dimension `dim` of the array is axis d - 1 - dim
            ax = d - 1 - dim
            n = shape[ax]
            x = torch.arange(n + 1, device=DEV, dtype=torch.float64) + 0.5 if ax == axis else torch.arange(n, device=DEV, dtype=torch.float64) + 1
            a = a.index_select(dim, (8 * x / (n + 1)).long().clamp(max=7))
        out.append(a.contiguous())
    return out


def _p1(n, mu=1e-3):
    """CSR arrays of the P1 stiffness matrix on the n^3 interior vertices of the uniform Kuhn mesh of the cube, with the
    coefficient mu in the half x < 1/2 and 1 in the other: an axis edge carries h/6 times the coefficients of its six
    tetrahedra (2, 1, 1, 2 of them in the four cubes around it)."""
    m = n + 1
    cells = np.broadcast_to(np.where((np.arange(m) + 0.5) / m < 0.5, mu, 1.0), (m, m, m))  # [z, y, x] per cube
    v = np.arange(1, m)
    h6 = 1.0 / (6.0 * m)
    sl = lambda s: slice(1, None) if s else slice(0, -1)  # the cube above / below a vertex along an axis
    ex = h6 * sum((2 if s == t else 1) * cells[sl(s), sl(t), :] for s in (0, 1) for t in (0, 1))
    ey = h6 * sum((2 if s == t else 1) * cells[sl(s), :, sl(t)] for s in (0, 1) for t in (0, 1))
    ez = h6 * sum((2 if s == t else 1) * cells[:, sl(s), sl(t)] for s in (0, 1) for t in (0, 1))
    z, y, x = np.meshgrid(v - 1, v - 1, v - 1, indexing="ij")
    row = (z * n + y) * n + x
    w = [ez[:-1], ey[:, :-1], ex[:, :, :-1], None, ex[:, :, 1:], ey[:, 1:], ez[1:]]
    w[3] = -sum(a for a in w if a is not None)
    step = [-n * n, -n, -1, 0, 1, n, n * n]
    ok = [z > 0, y > 0, x > 0, x >= 0, x < n - 1, y < n - 1, z < n - 1]
    keep = np.stack([a.ravel() for a in ok], axis=1)
    val = np.stack([-a.ravel() for a in w], axis=1)
    col = np.stack([(row + s).ravel() for s in step], axis=1)
    ptr = np.concatenate([[0], np.cumsum(keep.sum(axis=1))])
    return ptr.astype(np.int32), col[keep].astype(np.int32), np.ascontiguousarray(val[keep])


def _quadrature(alpha, kprime, lam):
    """Weights and shifts of the sinc quadrature of A^-alpha for the operator scaled by lam."""
    m = math.ceil(math.pi ** 2 / (4 * alpha * kprime ** 2))
    M = math.ceil(math.pi ** 2 / (4 * (1 - alpha) * kprime ** 2))
    el = np.arange(-m, M + 1)
    c = 2 * kprime * math.sin(math.pi * alpha) / math.pi * lam ** (alpha - 1) * np.exp(2 * (alpha - 1) * el * kprime)
    return c, -np.exp(-2 * el * kprime) / lam


def _problems(case):
    """The batch's problems: grids of the sizes up to nmax, powers and degrees in turn."""
    sizes = [n for n in (63, 127, 255, 511) if n <= case["nmax"]]
    return [(sizes[(5 * i + i // 3) % len(sizes)], ALPHAS[(3 * i + i // 5) % 5], 5 + (2 * i + i // 4) % 5) for i in range(case["count"])]


# ---------------------------------------------------------------------- plans and passes
def _options(case):
    o = bura.bura_default_options()
    if case.get("prec") == "fp64":
        o.precision = bura.BURA_PREC_FP64
    elif case.get("prec") == "df":
        o.refine = bura.BURA_REFINE_DF
    return o


class _State:
    """Plans and buffers of a case; the plans are freed with it."""

    def __init__(self):
        self.plans, self.batch = [], None

    def __del__(self):
        if self.batch is not None:
            self.batch.close()
        for p in self.plans:
            bura.bura_destroy(p)


def prepare(case, seed):
    s = _State()
    s.case, kind = case, case["kind"]
    if kind == "batch":
        s.f = [_rhs(n * n, seed, 10 + i) for i, (n, _, _) in enumerate(_problems(case))]
        s.u = [torch.empty_like(f) for f in s.f]
        s.plans = [bura.bura_setup((n, n), a, k) for n, a, k in _problems(case)]
        s.batch = bura.BuraBatch(s.plans, s.f, s.u, case["tol"])
        return s
    shape = _shape(case)
    n = math.prod(shape)
    s.f = _rhs(n, seed)
    s.u = torch.empty_like(s.f)
    if kind == "csr":
        s.plans = [bura.bura_setup_csr(*_p1(case["nx"]), case["alpha"], case["k"])]
    elif kind == "sum":
        c, d = _quadrature(case["alpha"], case["kprime"], _scale(shape))
        s.plans = [bura.bura_setup_shifts(shape, c[i:i + 13], d[i:i + 13]) for i in range(0, len(c), 13)]
    else:
        faces = tuple(a.cpu().numpy() for a in _faces(shape, seed)) if case["var"] else None
        s.plans = [bura.bura_setup(shape, case["alpha"], case["k"], faces=faces, options=_options(case))]
    if kind == "serve":
        s.f = s.f.cpu().pin_memory().numpy()
        s.u = [torch.empty(n, dtype=torch.float64).pin_memory().numpy() for _ in range(2)]
    return s


def _serve_alphas(case):
    return case["alpha"], ALPHAS[(ALPHAS.index(case["alpha"]) + 2) % 5]


def run(s):
    kind, tol = s.case["kind"], s.case["tol"]
    if kind == "batch":
        s.batch.run()
        s.batch.wait()
    elif kind == "serve":
        for a, u in zip(_serve_alphas(s.case), s.u):
            bura.bura_retarget(s.plans[0], a)
            bura.bura_solve_host(s.plans[0], s.f, u, tol)
    elif kind == "sum":
        bura.bura_solve_sum(s.plans, s.f, s.u, tol)
    else:
        bura.bura_solve(s.plans[0], s.f, s.u, tol)
    return s.u


def work(case):
    """Every right-hand side and coefficient read once and every solution written once; one application of every shifted
    operator."""
    if case["kind"] == "batch":
        ps = _problems(case)
        return {"bytes": sum(16.0 * n * n for n, _, _ in ps), "flops": sum(10.0 * n * n * (k + 1) for n, _, k in ps)}
    shape = _shape(case)
    n, d = float(math.prod(shape)), len(shape)
    if case["kind"] == "sum":
        systems = len(_quadrature(case["alpha"], case["kprime"], 1.0)[0])
    else:
        systems = case["k"] + 1
    passes = 2 if case["kind"] == "serve" else 1
    coef = 12.0 * 7 * n if case["kind"] == "csr" else 8.0 * d * n if case["var"] else 0.0
    return {"bytes": passes * 16 * n + coef, "flops": passes * 2.0 * (2 * d + 1) * n * systems}


# ---------------------------------------------------------------------- the same values in 64 bits
def _scale(shape):
    return sum((2 + min(n - 1, 2)) * (n + 1.0) ** 2 for n in shape)


def _table(alpha, k):
    with open("tests/golden/bura_oracle_table.json") as fh:
        e = json.load(fh)["%.4f/%d" % (alpha, k)]
    return [float(x) for x in e["c"]], [float(x) for x in e["d"]]


def _sine_value(shape, f, c, d):
    """sum_j c_j (A - d_j I)^-1 f of the constant operator scaled by its largest row sum, in its sine eigenbasis."""
    S, lam = [], torch.zeros((1,) * len(shape), dtype=torch.float64, device=DEV)
    for ax, n in enumerate(shape):
        i = torch.arange(1, n + 1, dtype=torch.int64, device=DEV)
        ang = (i[:, None] * i[None, :]) % (2 * (n + 1))
        S.append(math.sqrt(2.0 / (n + 1)) * torch.sin(math.pi * ang.double() / (n + 1)))
        e = 4 * (n + 1.0) ** 2 / _scale(shape) * torch.sin(math.pi * i.double() / (2 * (n + 1))) ** 2
        lam = lam + e.reshape([-1 if len(shape) - 1 - ax == t else 1 for t in range(len(shape))])

    def transform(x):
        for ax in range(len(shape)):
            dim = len(shape) - 1 - ax
            x = torch.movedim(torch.tensordot(x, S[ax], dims=([dim], [0])), -1, dim)
        return x

    g = transform(f.reshape(shape[::-1]))
    return transform(g * sum(cj / (lam - dj) for cj, dj in zip(c, d))).reshape(-1)


def _cg_value(apply, diag, f, c, d):
    """sum_j c_j (A - d_j I)^-1 f by diagonally scaled conjugate gradients on every shifted system."""
    c, d = (torch.tensor(v, dtype=torch.float64, device=DEV)[:, None] for v in (c, d))
    inv = 1 / (diag[None, :] - d)
    x = torch.zeros((len(c), f.numel()), dtype=torch.float64, device=DEV)
    r = f.expand_as(x).clone()
    z = inv * r
    p = z.clone()
    rz = (r * z).sum(1, keepdim=True)
    small = 1e-26 * float((f * f).sum())
    for it in range(20000):
        q = apply(p) - d * p
        a = rz / (p * q).sum(1, keepdim=True).clamp(min=1e-300)
        x += a * p
        r -= a * q
        z = inv * r
        new = (r * z).sum(1, keepdim=True)
        p = z + new / rz.clamp(min=1e-300) * p
        rz = new
        if it % 50 == 49 and float((r * r).sum(1).max()) <= small:
            break
    return (c * x).sum(0)


def _grid_apply(shape, seed):
    """The scaled operator of a variable field as a function of (systems, N) arrays, and its diagonal."""
    d = len(shape)
    w = [a * (shape[ax] + 1.0) ** 2 for ax, a in enumerate(_faces(shape, seed))]
    lo = [a.narrow(d - 1 - ax, 0, shape[ax]) for ax, a in enumerate(w)]
    hi = [a.narrow(d - 1 - ax, 1, shape[ax]) for ax, a in enumerate(w)]
    diag = sum(lo) + sum(hi)
    rows = diag.clone()  # absolute row sums: the faces to the boundary have no neighbour
    for ax in range(d):
        dim, n = d - 1 - ax, shape[ax]
        rows.narrow(dim, 1, n - 1).add_(lo[ax].narrow(dim, 1, n - 1))
        rows.narrow(dim, 0, n - 1).add_(hi[ax].narrow(dim, 0, n - 1))
    lam = rows.max()
    diag = diag / lam
    mid = [(w[ax].narrow(d - 1 - ax, 1, shape[ax] - 1) / lam) for ax in range(d)]

    def apply(p):
        x = p.reshape((-1,) + shape[::-1])
        y = diag * x
        for ax in range(d):
            dim, n = d - ax, shape[ax]
            y.narrow(dim, 1, n - 1).sub_(mid[ax] * x.narrow(dim, 0, n - 1))
            y.narrow(dim, 0, n - 1).sub_(mid[ax] * x.narrow(dim, 1, n - 1))
        return y.reshape(p.shape)

    return apply, diag.reshape(-1)


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        return [_sine_value((n, n), _rhs(n * n, seed, 10 + i), *_table(a, k)) for i, (n, a, k) in enumerate(_problems(case))]
    shape = _shape(case)
    n = math.prod(shape)
    f = _rhs(n, seed)
    if kind == "sum":
        return _sine_value(shape, f, *_quadrature(case["alpha"], case["kprime"], _scale(shape)))
    if kind == "serve":
        return [_sine_value(shape, f, *_table(a, case["k"])) for a in _serve_alphas(case)]
    if not case["var"]:
        return _sine_value(shape, f, *_table(case["alpha"], case["k"]))
    if n > 1500000:
        return None  # the plain conjugate gradients would take minutes
    if kind == "csr":
        ptr, col, val = _p1(case["nx"])
        rows = np.repeat(np.arange(n), np.diff(ptr))
        lam = np.bincount(rows, np.abs(val), n).max()
        A = torch.sparse_csr_tensor(torch.from_numpy(ptr).long(), torch.from_numpy(col).long(), torch.from_numpy(val / lam), (n, n)).to(DEV)
        diag = torch.from_numpy(np.bincount(rows, np.where(col == rows, val, 0.0), n) / lam).to(DEV)
        return _cg_value(lambda p: (A @ p.t()).t().contiguous(), diag, f, *_table(case["alpha"], case["k"]))
    return _cg_value(*_grid_apply(shape, seed), f, *_table(case["alpha"], case["k"]))
