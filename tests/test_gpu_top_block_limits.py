"""The top block at the order where its kernels change hands: the largest that
the register panels and the blocked inverse take (FP64 2048, FP32 4096: full
8-wide panels, every thread's rows in use, the largest shared memory of the
inverse), the first past it (no inverse: triangular solves, also for several
groups of columns), alone and beside a small problem in one handle.

eps = 0 keeps every column, so F = A up to rounding.  Tolerance: LU with partial
pivoting and its solves are backward stable to n u, the second-kind matrices here
have condition numbers below 10: 100 n u for apply and solve."""
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


def _dense(pts):
    n = len(pts)
    r2 = (pts[:, None, 0] - pts[None, :, 0]) ** 2 + (pts[:, None, 1] - pts[None, :, 1]) ** 2
    np.fill_diagonal(r2, 1)
    return -np.log(r2) / (4 * np.pi * n) + np.eye(n)


def _check(f, mats, prec, nrhs):
    sizes = [len(A) for A in mats]
    x = inputs.rhs(52, sum(sizes), nrhs)
    off = np.cumsum([0] + sizes)
    b = np.concatenate([x[:, o:o + n] @ A.T for A, o, n in zip(mats, off, sizes)], axis=1)
    y = f.apply(torch.from_numpy(x).cuda()).cpu().numpy()
    z = f.solve(torch.from_numpy(b).cuda()).cpu().numpy()
    for o, n in zip(off, sizes):
        tol = 100 * n * (2.0 ** -53 if prec == "fp64" else 2.0 ** -24)
        part = slice(o, o + n)
        assert np.linalg.norm(y[:, part] - b[:, part]) <= tol * np.linalg.norm(b[:, part])
        assert np.linalg.norm(z[:, part] - x[:, part]) <= tol * np.linalg.norm(x[:, part])


@pytest.mark.parametrize("prec,n", [("fp64", 2048), ("fp64", 2049), ("mixed", 4096), ("mixed", 4097)])
def test_one_block(pkg, prec, n):
    pts = inputs.random_points(51, n, 2)
    f = pkg.Factorization(torch.from_numpy(pts).cuda(), 0, 0.0, leaf=n, prec=pkg.FP64 if prec == "fp64" else pkg.MIXED)
    assert f.stats()["ntop"] == n
    A = _dense(pts)
    for nrhs in (1, 9):
        _check(f, [A], prec, nrhs)


@pytest.mark.parametrize("sizes", [(2048, 40), (2049, 40)])
def test_several_blocks(pkg, sizes):
    probs = [inputs.random_points(60 + i, n, 2) for i, n in enumerate(sizes)]
    f = pkg.Factorization.batched([torch.from_numpy(p).cuda() for p in probs], 0, 0.0, leaf=4096, prec=pkg.FP64)
    mats = [_dense(p) for p in probs]
    for nrhs in (1, 9):
        _check(f, mats, "fp64", nrhs)
