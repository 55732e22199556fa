"""The top block's LU, inverse and product, and the grouped sweeps, at the
edges of their panels, thread rows and column groups.

eps = 0 keeps every column, so the whole matrix is the top block: F = A up to
rounding.  Tolerances: LU with partial pivoting and its inverse are backward
stable to n u; the second-kind matrices here have condition numbers below 10, so
100 n u bounds the relative error of apply and solve (u = 2^-53, or 2^-24 for
the FP32 factor)."""
import numpy as np
import pytest

import oracle
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


def _dense(pts, kind):
    return oracle.matvec(pts, kind, np.eye(len(pts))).T


@pytest.mark.parametrize("prec,n", [("fp64", n) for n in (1, 2, 31, 32, 33, 65, 500, 513, 1030)] +
                         [("mixed", n) for n in (1, 33, 320, 513, 1025, 2060)])
def test_top_block_alone(pkg, prec, n):
    pts = inputs.random_points(51, n, 2)
    f = pkg.Factorization(torch.from_numpy(pts).cuda(), 0, 0.0, leaf=max(n, 1),
                          prec=pkg.FP64 if prec == "fp64" else pkg.MIXED)
    assert f.stats()["ntop"] == n
    A = _dense(pts, 0)
    tol = 100 * n * (2.0 ** -53 if prec == "fp64" else 2.0 ** -24)
    for nrhs in (1, 3, 9):
        x = inputs.rhs(52, n, nrhs)
        b = x @ A.T
        y = f.apply(torch.from_numpy(x).cuda()).cpu().numpy()
        z = f.solve(torch.from_numpy(b).cuda()).cpu().numpy()
        assert np.linalg.norm(y - b) <= tol * np.linalg.norm(b)
        assert np.linalg.norm(z - x) <= tol * np.linalg.norm(x)
    ld = np.linalg.slogdet(A)[1]
    assert abs(float(f.logdet()[0]) - ld) <= tol * n


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
def test_top_blocks_of_several_problems(pkg, prec):
    """One launch over blocks of different orders, some done before others."""
    sizes = [40, 700, 1, 33, 260, 32]
    probs = [inputs.random_points(60 + i, n, 2) for i, n in enumerate(sizes)]
    f = pkg.Factorization.batched([torch.from_numpy(p).cuda() for p in probs], 0, 0.0, leaf=1024,
                                  prec=pkg.FP64 if prec == "fp64" else pkg.MIXED)
    x = inputs.rhs(53, sum(sizes), 2)
    y = f.apply(torch.from_numpy(x).cuda()).cpu().numpy()
    z = f.solve(torch.from_numpy(x).cuda()).cpu().numpy()
    o = 0
    for p, n in zip(probs, sizes):
        A = _dense(p, 0)
        xs = x[:, o:o + n]
        tol = 100 * n * (2.0 ** -53 if prec == "fp64" else 2.0 ** -24)
        assert np.linalg.norm(y[:, o:o + n] - xs @ A.T) <= tol * np.linalg.norm(xs @ A.T)
        ref = np.linalg.solve(A, xs.T).T
        assert np.linalg.norm(z[:, o:o + n] - ref) <= tol * np.linalg.norm(ref)
        o += n


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("flags", [0, 4, 16])
@pytest.mark.parametrize("nrhs", [5, 8, 67])
def test_column_groups_equal_single_columns(pkg, prec, flags, nrhs):
    """Groups of four columns (a ragged last group, more than one pass of 64)
    give what each column gives alone, for solve and apply, both schedules and
    symmetric storage."""
    pts = torch.from_numpy(inputs.random_points(54, 3000, 2)).cuda()
    f = pkg.Factorization(pts, 0, 1e-6, leaf=64, prec=pkg.FP64 if prec == "fp64" else pkg.MIXED, flags=flags)
    B = torch.from_numpy(inputs.rhs(55, 3000, nrhs)).cuda()
    tol = 1e-13 if prec == "fp64" else 2e-6
    for fn in (f.solve, f.apply):
        Y = fn(B)
        for c in (0, 3, 4, nrhs - 1):
            y = fn(B[c])
            assert float(torch.linalg.norm(Y[c] - y)) <= tol * float(torch.linalg.norm(y))
