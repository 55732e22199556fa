"""FP32 boxes of more than 128 DOFs: pair blocks assembled in several pieces,
LU and inverse of X_RR in registers at its two widths (up to 192 and up to 224
rows) and the blocked form beyond.  Apply against the exact operator and solve
against apply, both at the suite's 10 eps bar (the operator's eigenvalues are
near 1, so the FP32 factor's own rounding stays below it)."""
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


# points, leaf, least and most redundant DOFs of the widest box
CASES = {
    "r_to_160": (2300, 185, 129, 160),
    "r_to_192": (2700, 210, 150, 192),
    "r_to_224": (3150, 240, 193, 224),
    "blocked": (3500, 260, 193, 260),
}


@pytest.mark.parametrize("case", list(CASES))
def test_wide_boxes(pkg, case):
    n, leaf, rmin, rmax = CASES[case]
    eps = 1e-4  # ranks of about 10: r stays near the box's size
    pts = torch.from_numpy(inputs.random_points(31, n, 2)).cuda()
    f = pkg.Factorization(pts, 0, eps, leaf=leaf, prec=pkg.MIXED, flags=pkg.rss.FLAG_NO_AUTOTUNE)
    s = f.stats()
    r = s["b"] - s["k"]
    assert s["b"].max() > 128 and rmin <= r.max() <= rmax, (s["b"].max(), r.max())
    x = torch.from_numpy(np.ascontiguousarray(inputs.rhs(32, n, 3))).cuda()
    ax, y = f.matvec(x), f.apply(x)
    assert float(torch.linalg.norm(y - ax) / torch.linalg.norm(ax)) <= 10 * eps
    z = f.solve(y)
    assert float(torch.linalg.norm(z - x) / torch.linalg.norm(x)) <= 10 * eps
    for m in (1, 2):  # narrow groups: the box's CTAs share the last product
        z = f.solve(y[:m].contiguous())
        assert float(torch.linalg.norm(z - x[:m]) / torch.linalg.norm(x[:m])) <= 10 * eps
