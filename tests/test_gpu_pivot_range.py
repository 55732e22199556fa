"""FP64 factors of matrices far from unit scale: pivots are compared over the
whole FP64 range.  Scaling a first-kind matrix (diag 0, so that every diagonal
block starts with zeros on its diagonal) by a power of two scales every number
of the factorization exactly, so what solve makes of apply's output has the same
error as at scale 1; a factor of two is left for kernels that add in no fixed
order."""
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


def _round_trip(pkg, pts, eps, leaf, weight):
    f = pkg.Factorization(torch.from_numpy(pts).cuda(), 0, eps, leaf=leaf, prec=pkg.FP64, diag=0.0, weight=weight)
    x = torch.from_numpy(inputs.rhs(81, len(pts), 2)).cuda()
    b = f.apply(x)
    assert float(torch.linalg.norm(b / weight)) > 0
    return float(torch.linalg.norm(f.solve(b) - x) / torch.linalg.norm(x))


@pytest.mark.parametrize("scale", [2.0 ** -166, 2.0 ** 166, 2.0 ** -400])
@pytest.mark.parametrize("case", ["top_only", "top_panels", "grid", "random"])
def test_far_scales_pivot_like_unit_scale(pkg, scale, case):
    pts, eps, leaf = {"top_only": (inputs.random_points(82, 40, 2), 0.0, 40),
                      "top_panels": (inputs.random_points(83, 1100, 2), 0.0, 1100),
                      "grid": (inputs.grid_points(40, 2), 1e-10, 32),
                      "random": (inputs.random_points(84, 1500, 2), 1e-10, 32)}[case]
    unit = _round_trip(pkg, pts, eps, leaf, 1.0)
    assert unit <= 1e-8
    assert _round_trip(pkg, pts, eps, leaf, scale) <= 2 * unit
