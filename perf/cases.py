"""What a user of this package has it do, as cases that can be timed.

A case is a dict of plain values:

  path      factor_refine  factor a point set, then solve A x = b to a 1e-10
                           relative residual (GMRES-IR): the main call chain
            factor_solve   factor, then one plain solve with the factor
            refine, cg     refined / conjugate-gradient solves with a factor
                           that the program keeps
            solve, apply   one plain solve / apply with a kept factor
            matvec         the exact FP64 operator of a kept factor
            network        loss, gradient and prediction of the rank-proposal
                           network
  points    grid (side^dim cell centres) or random (iid uniform points)
  prec      mixed (FP32 factor) or fp64

Points of a grid are fixed by its side; right-hand sides, scattered points
and network inputs are drawn on the GPU from the seed.
"""
from __future__ import annotations

import math

import torch

import paper_1609_08130_gb300 as pkg
from paper_1609_08130_gb300 import inputs, rss

TOL = 1e-10
DEFAULTS = dict(points="grid", dim=2, problems=1, prec="mixed", eps=1e-6, leaf=64, nrhs=1, colours=3)


def listed():
    return [
        # the smallest configuration (64^2 grid, one right-hand side), library
        # defaults: launches, host work and latency count
        dict(name="grid2d_64_refine", path="factor_refine", side=64),
        # the benchmark's default workload: 512^2 grid, four right-hand sides,
        # the 2^d-colour schedule
        dict(name="grid2d_512_refine", path="factor_refine", side=512, nrhs=4, colours=2),
        # the 3D workload of the paper's second example, 32^3 at eps 1e-3
        dict(name="grid3d_32_refine", path="factor_refine", dim=3, side=32, eps=1e-3, colours=2),
        # many independent scattered problems in one handle, sizes spread over
        # the batched workload's 1024..16384
        dict(name="batch_32_refine", path="factor_refine", points="random", problems=32, n_lo=1024, n_hi=16384,
             colours=2),
        # one scattered problem of an odd size, library defaults
        dict(name="random2d_20011_refine", path="factor_refine", points="random", n=20011, nrhs=3),
        # a ragged grid (no power of two) with a leaf size of its own, FP64
        # throughout: the direct solver
        dict(name="grid2d_100_fp64_solve", path="factor_solve", side=100, leaf=40, prec="fp64", nrhs=2),
        # one more right-hand side for a kept FP64 factor: the shortest call
        dict(name="solve_fp64_128", path="solve", side=128, prec="fp64"),
        # a kept FP32 factor as preconditioner for a block of right-hand sides
        dict(name="refine_256_16rhs", path="refine", side=256, nrhs=16, colours=2),
        # the paper's iterative solver (CG) with a kept factor
        dict(name="cg_256_2rhs", path="cg", side=256, nrhs=2),
        # the forward operator through the factor
        dict(name="apply_fp64_256_8rhs", path="apply", side=256, prec="fp64", nrhs=8),
        # the exact operator on scattered 3D points
        dict(name="matvec_random3d_20000", path="matvec", points="random", dim=3, n=20000, eps=1e-3, nrhs=2),
        # training signal of the rank-proposal network over the boxes of a
        # large factorization
        dict(name="network_20000", path="network", n=20000),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    path = rng.choice(["factor_refine"] * 5 + ["factor_solve", "solve", "refine", "cg", "apply", "matvec", "network"])
    if path == "network":
        return dict(path=path, n=_log_int(rng, 300, 20000))
    c = dict(path=path)
    kind = rng.choice(["grid2d", "grid2d_pow2", "random2d", "grid3d", "random3d", "batch"])
    if path == "matvec" and kind == "batch":
        kind = "random2d"
    if path in ("solve", "apply", "factor_solve"):
        c["prec"] = "fp64"
    elif rng.random() < 0.15 and path == "factor_refine":
        c["prec"] = "fp64"
    fp64 = c.get("prec") == "fp64"
    c["colours"] = rng.choice([2, 3])
    c["nrhs"] = rng.choice([1, 1, 2, 3, 4] if path.startswith("factor") else [1, 2, 4, 5, 8, 16])
    if kind == "grid2d":
        c.update(side=_log_int(rng, 20, 150), leaf=rng.choice([25, 40, 64]))
    elif kind == "grid2d_pow2":
        c.update(side=rng.choice([32, 64, 128, 256]))
    elif kind == "random2d":
        c.update(points="random", n=_log_int(rng, 500, 20000), leaf=rng.choice([30, 64]))
    elif kind == "grid3d":
        c.update(dim=3, side=rng.randint(8, 16 if fp64 else 32), eps=1e-3)
    elif kind == "random3d":
        c.update(points="random", dim=3, n=_log_int(rng, 500, 4000 if fp64 else 20000), eps=1e-3)
    else:
        c.update(points="random", problems=rng.randint(2, 12), n_lo=rng.randint(300, 1024),
                 n_hi=_log_int(rng, 1100, 4000 if fp64 else 16384))
    return c


def _sizes(c):
    """Points of each problem: fixed by the case, so that its cost is."""
    if c["points"] == "grid":
        return [c["side"] ** c["dim"]]
    if c["problems"] == 1 and "n" in c:
        return [c["n"]]
    lo, hi, p = c["n_lo"], c["n_hi"], c["problems"]
    return [lo + int((hi - lo) * (((i * 0.6180339887498949) + 0.31) % 1.0)) for i in range(p)]


def _full(case):
    return {**DEFAULTS, **case}


def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _points(c, g):
    if c["points"] == "grid":
        return [torch.from_numpy(inputs.grid_points(c["side"], c["dim"])).cuda()]
    return [torch.rand(n, c["dim"], generator=g, device="cuda", dtype=torch.float64) for n in _sizes(c)]


def _kernel_kind(c):
    return pkg.LAPLACE2D_LOG if c["dim"] == 2 else pkg.LAPLACE3D_INV


def _factor(c, pts):
    kw = dict(leaf=c["leaf"], prec=pkg.FP64 if c["prec"] == "fp64" else pkg.MIXED,
              flags=rss.FLAG_COLOUR_2D if c["colours"] == 2 else 0)
    if c["problems"] > 1:
        return pkg.Factorization.batched(pts, _kernel_kind(c), c["eps"], **kw)
    return pkg.Factorization(pts[0], _kernel_kind(c), c["eps"], **kw)


def _network_data(case, g):
    """Features in the ranges that boxes have (leaf and upper boxes of 2D and
    3D trees) and rank fractions."""
    n = case["n"]
    u = torch.rand(n, 13, generator=g, device="cuda")
    X = torch.zeros(n, 16, device="cuda")
    dim3 = (u[:, 0] < 0.5).float()
    X[:, 0] = dim3
    X[:, 1] = dim3
    X[:, 2] = 0.3 + 0.3 * (u[:, 2] < 0.5).float()
    X[:, 3:6] = torch.log2(1 + torch.exp(u[:, 3:6] * 4 + torch.tensor([2.5, 4.0, 5.0], device="cuda"))) / 10
    X[:, 6:8] = 0.5 + 0.5 * torch.round(u[:, 6:8] * 8) / 8
    X[:, 8] = (u[:, 8] < 0.7).float()
    X[:, 9] = torch.where(X[:, 8] > 0, torch.ones_like(u[:, 9]), 0.3 + 0.6 * u[:, 9])
    X[:, 10] = torch.floor(2 + 5 * u[:, 10]) / 10
    X[:, 11] = torch.where(dim3 > 0, 0.9003, 0.6022)
    X[:, 12] = 0.5
    y = 0.25 + 0.6 * torch.rand(n, generator=g, device="cuda")
    return X, y


def prepare(case, seed):
    g = _generator(seed)
    if case["path"] == "network":
        X, y = _network_data(case, g)
        return dict(case=case, X=X, y=y, net=pkg.Mlp(seed=int(seed)))
    c = _full(case)
    pts = _points(c, g)
    n = sum(_sizes(c))
    b = torch.randn(c["nrhs"], n, generator=g, device="cuda", dtype=torch.float64)
    if c["nrhs"] == 1:
        b = b[0]
    state = dict(case=c, b=b)
    if c["path"].startswith("factor"):
        state["pts"] = pts
    else:
        state["factor"] = _factor(c, pts)
    return state


def run(state):
    c = state["case"]
    path = c["path"]
    if path == "network":
        grad, loss = state["net"].grad(state["X"], state["y"])
        return dict(grad=grad, loss=loss, predict=state["net"].predict(state["X"]))
    b = state["b"]
    f = _factor(c, state["pts"]) if path.startswith("factor") else state["factor"]
    if path in ("factor_refine", "refine"):
        return f.solve_refined(b, tol=TOL)[0]
    if path == "cg":
        return f.solve_cg(b, tol=TOL)[0]
    if path in ("factor_solve", "solve"):
        return f.solve(b)
    if path == "apply":
        return f.apply(b)
    return f.matvec(b)


def work(case):
    """Inputs read once and outputs written once (a kept factor is an input),
    and the method's arithmetic counted per point: in 2D about 1.5e5 flops to
    compress and eliminate a point at the leaves and as much again above, in
    3D about 1e6; two flops per stored entry and column for a solve."""
    if case["path"] == "network":
        n = case["n"]
        return {"bytes": n * (16 + 1 + 1) * 4.0 + 9473 * 6.0, "flops": n * 9408 * 2.0 * 4}
    c = _full(case)
    n = sum(_sizes(c))
    vectors = n * 8.0 * (c["dim"] + 2 * c["nrhs"])
    elem = 8 if c["prec"] == "fp64" else 4
    entries = n * (600.0 if c["dim"] == 2 else 2500.0)
    operator = n * 20.0 * max(math.log2(max(n, 2)), 1.0) * c["nrhs"]
    path = c["path"]
    if path == "matvec":
        return {"bytes": vectors, "flops": operator}
    if path.startswith("factor"):
        return {"bytes": vectors, "flops": n * (3e5 if c["dim"] == 2 else 1e6) + 2 * entries * c["nrhs"]}
    return {"bytes": vectors + elem * entries, "flops": 2 * entries * c["nrhs"] + operator}


# --- the same in 64 bits, without the package's kernels --------------------

def _kernel_of_r2(dim, r2):
    return -torch.log(r2) / (4 * math.pi) if dim == 2 else 1 / (4 * math.pi * torch.sqrt(r2))


class _GridOperator:
    """A = I + K / n on an s^dim grid of cell centres, x fastest, by a
    circulant of side 2 s."""

    def __init__(self, s, dim):
        self.s, self.dim, self.n = s, dim, s ** dim
        i = torch.arange(2 * s, device="cuda", dtype=torch.float64)
        d = torch.where(i < s, i, i - 2 * s) / s
        r2 = sum(a * a for a in torch.meshgrid(*([d] * dim), indexing="ij"))
        corner = (0,) * dim
        r2[corner] = 1.0
        k = _kernel_of_r2(dim, r2) / self.n
        k[corner] = 0.0
        self.spectrum = torch.fft.rfftn(k)

    def __call__(self, x):
        s, dim = self.s, self.dim
        dims = tuple(range(1, dim + 1))
        v = x.reshape((-1,) + (s,) * dim)
        y = torch.fft.irfftn(torch.fft.rfftn(v, s=(2 * s,) * dim, dim=dims) * self.spectrum, s=(2 * s,) * dim, dim=dims)
        return x + y[(slice(None),) + (slice(0, s),) * dim].reshape(x.shape)


class _DenseOperator:
    """A = I + K / n on any points, the matrix formed in slabs."""

    def __init__(self, pts):
        n, dim = pts.shape
        self.K = torch.empty(n, n, device="cuda", dtype=torch.float64)
        for i in range(0, n, 2048):
            r2 = sum((pts[i:i + 2048, d, None] - pts[None, :, d]) ** 2 for d in range(dim))
            rows = torch.arange(i, min(i + 2048, n), device="cuda")
            r2[rows - i, rows] = 1.0
            k = _kernel_of_r2(dim, r2) / n
            k[rows - i, rows] = 1.0
            self.K[i:i + 2048] = k

    def __call__(self, x):
        return x @ self.K.T


def _solve_cg(A, b):
    x = torch.zeros_like(b)
    r = b.clone()
    p = r.clone()
    rs = (r * r).sum(1, keepdim=True)
    bs = rs.clone()
    for _ in range(200):
        q = A(p)
        x += rs / (p * q).sum(1, keepdim=True) * p
        r = b - A(x)
        new = (r * r).sum(1, keepdim=True)
        if float((new / bs).max()) < 1e-29:
            break
        p = r + new / rs * p
        rs = new
    return x


def _exact_network(case, seed):
    s = prepare(case, seed)
    th = torch.from_numpy(s["net"].params()).to(torch.bfloat16).double().cuda().requires_grad_(True)
    X, y, H = s["X"].double(), s["y"].double(), 64
    sizes = [H * 16, H, H * H, H, H * H, H, H, 1]
    W1, b1, W2, b2, W3, b3, w4, b4 = torch.split(th, sizes)
    h = torch.tanh(X @ W1.view(H, 16).T + b1)
    h = torch.tanh(h @ W2.view(H, H).T + b2)
    h = torch.tanh(h @ W3.view(H, H).T + b3)
    p = h @ w4 + b4
    loss = ((p - y) ** 2).mean()
    loss.backward()
    return dict(grad=th.grad, loss=float(loss), predict=p.detach())


def exact(case, seed):
    if case["path"] == "network":
        return _exact_network(case, seed)
    c = _full(case)
    g = _generator(seed)
    pts = _points(c, g)
    n = sum(_sizes(c))
    b = torch.randn(c["nrhs"], n, generator=g, device="cuda", dtype=torch.float64)
    forward = c["path"] in ("apply", "matvec")
    out, at = [], 0
    for p in pts:
        part = b[:, at:at + len(p)]
        at += len(p)
        A = _GridOperator(c["side"], c["dim"]) if c["points"] == "grid" else _DenseOperator(p)
        out.append(A(part) if forward else _solve_cg(A, part))
        del A
    out = torch.cat(out, dim=1)
    return out[0] if c["nrhs"] == 1 else out
