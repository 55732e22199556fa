"""Solves with ill-conditioned top blocks (first-kind matrices, eps 0: the whole
matrix is the top block).  Several problems, more than 1024 DOFs or more than
four columns correct the product with the inverse by its residual, and are then
as accurate as triangular solves; a narrow solve of one small block is the plain
product, of the same factors.

Tolerance: against triangular solves the plain product's forward error is 3 to 10
times larger here.  Half of it, in the geometric mean, is asked for, on
right-hand sides made with the factor's own matrix (column by column from
rss_apply), so that the roundings of its entries are in neither."""
import numpy as np
import pytest

from paper_1609_08130_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_1609_08130_gb300 as p
    p.build()
    return p


def _factor(pkg, pts, prec):
    return pkg.Factorization(torch.from_numpy(pts).cuda(), 0, 0.0, leaf=1024, diag=0.0,
                             prec=pkg.FP64 if prec == "fp64" else pkg.MIXED)


def _rhs(f, x):
    A = f.apply(torch.eye(x.shape[1], dtype=torch.float64, device="cuda")).cpu().numpy().T
    return (x.astype(np.longdouble) @ A.T.astype(np.longdouble)).astype(np.float64)


def _solve(f, b):
    return f.solve(torch.from_numpy(np.ascontiguousarray(b)).cuda()).cpu().numpy()


def _gmean_ratio(new, plain, x):
    e = [np.linalg.norm(z - x, axis=1) for z in (new, plain)]
    return float(np.exp(np.mean(np.log(e[0] / e[1]))))


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("n", [300, 900])
def test_wide_calls(pkg, prec, n):
    f = _factor(pkg, inputs.random_points(95, n, 2), prec)
    x = inputs.rhs(96, n, 12)
    b = _rhs(f, x)
    narrow = np.stack([_solve(f, b[c]) for c in range(12)])
    assert _gmean_ratio(_solve(f, b), narrow, x) <= 0.5


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
def test_several_problems(pkg, prec):
    sizes = [300 + 27 * i for i in range(12)]
    probs = [inputs.random_points(90 + i, n, 2) for i, n in enumerate(sizes)]
    f = pkg.Factorization.batched([torch.from_numpy(p).cuda() for p in probs], 0, 0.0, leaf=1024, diag=0.0,
                                  prec=pkg.FP64 if prec == "fp64" else pkg.MIXED)
    single = [_factor(pkg, p, prec) for p in probs]
    xs = [inputs.rhs(200 + i, n, 1) for i, n in enumerate(sizes)]
    bs = [_rhs(g, x) for g, x in zip(single, xs)]
    z, off = _solve(f, np.concatenate(bs, axis=1)), np.cumsum([0] + sizes)
    r = [_gmean_ratio(z[:, o:o + n], _solve(g, b), x) for g, b, x, o, n in zip(single, bs, xs, off, sizes)]
    assert np.exp(np.mean(np.log(r))) <= 0.5


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("dim,kind", [(2, 0), (3, 1)])
def test_well_conditioned_blocks_keep_the_plain_product(pkg, prec, dim, kind):
    """Second-kind matrices: a wide call gives each column the bits of a narrow
    one, since neither corrects anything."""
    n = 700
    f = pkg.Factorization(torch.from_numpy(inputs.random_points(97, n, dim)).cuda(), kind, 0.0, leaf=1024,
                          prec=pkg.FP64 if prec == "fp64" else pkg.MIXED)
    assert f.stats()["ntop"] == n
    b = inputs.rhs(98, n, 9)
    wide = _solve(f, b)
    assert all(np.array_equal(wide[c], _solve(f, b[c])) for c in range(9))
