"""The direct sum is as accurate as a sum in FP64: the kernel's part alone
(diag 0, as in first-kind matrices) against extended precision, for right-hand
sides of one sign and of both.

Tolerance: what the kernel adds up is good to about 2^-56 a term; the result is
rounded where the parts' sums go to FP64 and in three FP64 products, and the
kernel's constant and the weight are FP64: fewer than eight roundings of up to
2^-53, mostly of random sign, so 2^-51 in the norm.  A plain FP64 sum on the
same rows is measured beside it and has to be no better."""
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


def _rows(pts, kind, w, rows, T):
    """Rows of w K in the type T."""
    p = pts.astype(T)
    r2 = sum((p[rows][:, None, d] - p[None, :, d]) ** 2 for d in range(p.shape[1]))
    r2[np.arange(len(rows)), rows] = 1
    pi4 = np.arctan(T(1)) * 16
    K = T(w) * (-np.log(r2) / pi4 if kind == 0 else 1 / (pi4 * np.sqrt(r2)))
    K[np.arange(len(rows)), rows] = 0
    return K


def _errors(pkg, pts, kind, x):
    n = len(pts)
    f = pkg.Factorization(torch.from_numpy(pts).cuda(), kind, 1e-2, leaf=max(64, n // 8), prec=pkg.MIXED, diag=0.0)
    y = f.matvec(torch.from_numpy(x).cuda()).cpu().numpy()
    rows = np.arange(0, n, max(1, n // 200))
    ref = x.astype(np.longdouble) @ _rows(pts, kind, 1.0 / n, rows, np.longdouble).T
    K = _rows(pts, kind, 1.0 / n, rows, np.float64)
    # term after term, as one accumulator adds them
    plain = np.stack([np.cumsum(K * xc[None, :], axis=1)[:, -1] for xc in x])
    nrm = lambda a: float(np.sqrt((a * a).sum()))  # noqa: E731
    return nrm(y[:, rows] - ref) / nrm(ref), nrm(plain - ref) / nrm(ref)


@pytest.mark.parametrize("dim,kind", [(2, 0), (3, 1), (2, 1), (3, 0)])
@pytest.mark.parametrize("n,nrhs", [(300, 1), (4000, 3), (20000, 8)])
@pytest.mark.parametrize("sign", ["both", "one"])
def test_error_is_that_of_fp64(pkg, dim, kind, n, nrhs, sign):
    pts = inputs.random_points(61, n, dim)
    x = inputs.rhs(62, n, nrhs)
    new, plain = _errors(pkg, pts, kind, np.abs(x) if sign == "one" else x)
    assert new <= 2.0 ** -51 and new <= plain, (new, plain)


@pytest.mark.parametrize("dim,kind", [(2, 0), (3, 1)])
def test_cluster_at_the_origin(pkg, dim, kind):
    """Coordinates whose last bits are far below those of the others: half of
    the points in a cell of side 2^-24 at the origin."""
    pts = inputs.random_points(63, 600, dim)
    pts[:300] *= 2.0 ** -24
    new, plain = _errors(pkg, pts, kind, inputs.rhs(64, 600, 2))
    assert new <= 2.0 ** -51 and new <= plain, (new, plain)
