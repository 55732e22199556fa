"""The FP32 factor's ID from the exact Gram matrix (tensor cores, pivoted
Cholesky) at the edges of its block widths and row chunks, against the
Householder reduction of the same rows (the forced large-box path) and the
exact operator.  Both IDs truncate at the same tolerance, so ranks agree up
to ties at the threshold, and each factor's apply error meets the suite's
10 eps bar."""
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


# points, kind, eps, leaf, extra flags, least and most |B| the case is for
CASES = {
    "narrow_leaf": (lambda: inputs.grid_points(64, 2), 0, 1e-6, 9, 0, 1, 80),
    "one_block_full": (lambda: inputs.grid_points(64, 2), 0, 1e-6, 64, 0, 64, 96),
    "one_block_plus_one": (lambda: inputs.random_points(4, 4000, 2), 0, 1e-6, 65, 0, 65, 96),
    "wide_block_full": (lambda: inputs.random_points(5, 5500, 2), 0, 1e-6, 96, 0, 90, 128),
    "two_blocks": (lambda: inputs.random_points(6, 7000, 2), 0, 1e-6, 128, 0, 100, 128),
    "three_blocks": (lambda: inputs.random_points(7, 2600, 2), 0, 1e-6, 200, 0, 129, 192),
    "five_blocks": (lambda: inputs.random_points(8, 6000, 2), 0, 1e-6, 500, 0, 257, 512),
    "octree": (lambda: inputs.random_points(9, 6000, 3), 1, 1e-3, 64, 0, 65, 256),
    "weak_rows": (lambda: inputs.random_points(10, 3000, 2), 0, 1e-6, 64, 32, 60, 128),
    "coarse_eps": (lambda: inputs.random_points(11, 3000, 2), 0, 1e-2, 64, 4, 30, 64),
    "smallest_eps": (lambda: inputs.grid_points(48, 2), 0, 5e-7, 40, 0, 36, 96),
}


@pytest.mark.parametrize("case", list(CASES))
def test_gram_id_matches_householder_and_operator(pkg, case):
    mk, kind, eps, leaf, flags, bmin, bmax = CASES[case]
    pts = torch.from_numpy(mk()).cuda()
    n = pts.shape[0]
    F = lambda fl: pkg.Factorization(pts, kind, eps, leaf=leaf, prec=pkg.MIXED,  # noqa: E731
                                     flags=flags | pkg.rss.FLAG_NO_AUTOTUNE | fl)
    f, g = F(0), F(pkg.rss.FLAG_LARGE_BOX_PATH)
    s, t = f.stats(), g.stats()
    assert bmin <= s["b"].max() <= bmax, s["b"].max()
    same_b = s["b"] == t["b"]  # boxes whose children kept the same ranks
    assert same_b.any()
    dk = np.abs(s["k"][same_b] - t["k"][same_b])
    assert dk.max() <= max(2, 0.1 * s["b"].max()) and np.mean(dk <= 1) > 0.9, (dk.max(), np.mean(dk <= 1))
    x = torch.from_numpy(inputs.rhs(12, n, 2)).cuda()
    ax = f.matvec(x)
    err = [float(torch.linalg.norm(h.apply(x) - ax) / torch.linalg.norm(ax)) for h in (f, g)]
    assert err[0] <= 10 * eps and err[1] <= 10 * eps, err
    # the same bits again: integer sums do not depend on the order
    h = F(0)
    assert np.array_equal(h.stats()["k"], s["k"])
    if flags != 4:  # (2^d colours add shared blocks atomically)
        assert torch.equal(h.apply(x), f.apply(x))


def test_tolerances_below_the_quantisation_take_the_householder_id(pkg):
    """eps 1e-7 is below what the Gram form resolves: the factor is the one
    that the Householder shapes give, bit for bit, with and without a table."""
    pts = torch.from_numpy(inputs.grid_points(32, 2)).cuda()
    x = torch.from_numpy(inputs.normal(3, 1024)).cuda()
    lib = pkg.lib()
    try:
        lib.rss_autotune_clear()
        for width in (64, 128):
            for cls in range(20):
                assert lib.rss_autotune_set(4, width, cls, 1, 1, 1, 1) == 0
        pinned = pkg.Factorization(pts, 0, 1e-7, leaf=64, prec=pkg.MIXED)
        ax = pinned.matvec(x)
        assert float(torch.linalg.norm(pinned.apply(x) - ax) / torch.linalg.norm(ax)) <= 1e-5
        again = pkg.Factorization(pts, 0, 1e-7, leaf=64, prec=pkg.MIXED)
        assert torch.equal(again.apply(x), pinned.apply(x))
    finally:
        lib.rss_autotune_clear()
