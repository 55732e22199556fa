"""The exact operator by direct summation (pairs of FP32 numbers) against the
same sum in extended precision, at the edges of its tiles and column groups,
for both kernels in both dimensions, several problems, extreme column scales,
values that are not finite and points that coincide.

Tolerance: a pair carries 48 bits and a term goes through fewer than eight
pair operations, the FP64 sums of 256 terms add 2^-50 relative to the sum of
magnitudes, the output rounds once: |y - ref| <= 2^-44 |K| |x| + 2^-51 |ref|."""
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


def _reference(pts, kind, w, diag, x):
    """(A x, |K| |x|) in numpy's extended precision; x: (nrhs, n)."""
    p = pts.astype(np.longdouble)
    r2 = sum((p[:, None, d] - p[None, :, d]) ** 2 for d in range(p.shape[1]))
    np.fill_diagonal(r2, 1)
    pi = np.arctan(np.longdouble(1)) * 4
    K = np.longdouble(w) * (-np.log(r2) / (4 * pi) if kind == 0 else 1 / (4 * pi * np.sqrt(r2)))
    np.fill_diagonal(K, 0)
    xl = x.astype(np.longdouble)
    return xl @ K.T + np.longdouble(diag) * xl, np.abs(xl) @ np.abs(K).T


def _check(y, ref, mag):
    err = np.abs(y.astype(np.longdouble) - ref)
    assert np.all(err <= 2.0 ** -44 * mag + 2.0 ** -51 * np.abs(ref)), float(np.max(err / (mag + np.abs(ref))))


@pytest.mark.parametrize("dim,kind", [(2, 0), (3, 1), (2, 1), (3, 0)])
@pytest.mark.parametrize("n,nrhs", [(1, 1), (2, 3), (255, 1), (256, 2), (257, 4), (700, 8), (300, 11), (130, 35)])
def test_direct_sum_matches_extended_precision(pkg, dim, kind, n, nrhs):
    pts = inputs.random_points(31, n, dim)
    f = pkg.Factorization(torch.from_numpy(pts).cuda(), kind, 1e-3, leaf=64, diag=0.0 if n > 2 else 1.0)
    x = inputs.rhs(32, n, nrhs)
    y = f.matvec(torch.from_numpy(x).cuda()).cpu().numpy()
    _check(y, *_reference(pts, kind, 1.0 / n, 0.0 if n > 2 else 1.0, x))


def test_many_tiles_and_batches(pkg):
    """Several problems in one handle: tiles that end inside a block, four
    threads per target (over 300 tiles), each problem's own weight."""
    sizes = [3000, 513, 64] + [1500] * 52
    probs = [inputs.batched_problem(40 + p, n) for p, n in enumerate(sizes)]
    f = pkg.Factorization.batched([torch.from_numpy(p).cuda() for p in probs], 0, 1e-6, prec=pkg.MIXED)
    x = inputs.rhs(33, sum(sizes), 1)
    y = f.matvec(torch.from_numpy(x).cuda()).cpu().numpy()
    o = 0
    for p, n in list(zip(probs, sizes))[:5]:
        _check(y[:, o:o + n], *_reference(p, 0, 1.0 / n, 1.0, x[:, o:o + n]))
        o += n


@pytest.mark.parametrize("scale", [1e-300, 1e-30, 1e30, 1e290])
def test_column_scales(pkg, scale):
    n = 600
    pts = inputs.random_points(34, n, 2)
    f = pkg.Factorization(torch.from_numpy(pts).cuda(), 0, 1e-3, leaf=64)
    x = inputs.rhs(35, n, 2)
    x[1] *= scale
    x[0, 256:] *= 1e-200  # tiles of one column at different scales
    y = f.matvec(torch.from_numpy(x).cuda()).cpu().numpy()
    _check(y, *_reference(pts, 0, 1.0 / n, 1.0, x))


def test_values_that_are_not_finite_and_points_that_coincide(pkg):
    n = 520
    pts = inputs.random_points(36, n, 2)
    pts[7] = pts[300] + 2.0 ** -52  # far closer than FP32 resolves
    f = pkg.Factorization(torch.from_numpy(pts).cuda(), 0, 1e-3, leaf=64)
    x = inputs.rhs(37, n, 3)
    x[1, 400] = np.inf
    x[2, 3] = np.nan
    y = f.matvec(torch.from_numpy(x).cuda()).cpu().numpy()
    ref, mag = _reference(pts, 0, 1.0 / n, 1.0, x[:1])
    _check(y[:1], ref, mag)
    assert np.all(np.isinf(y[1])) and np.all(np.isnan(y[2]))
