"""A table of ID shapes saved from one run and set in another gives the same
factor, bit for bit: which phases take the Gram form is a rule of sizes.  And the
Householder shapes, which FP32 factors take below the Gram form's tolerance, each
against the exact operator."""
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


@pytest.fixture
def lib(pkg):
    lib = pkg.lib()
    lib.rss_autotune_clear()
    yield lib
    lib.rss_autotune_clear()


def _restore(lib, table):
    lib.rss_autotune_clear()
    for t in table:
        assert lib.rss_autotune_set(t["elem_bytes"], t["width"], t["phase_class"], t["tpc"], t["groups"], t["ctas"],
                                    t["rows"]) == 0


# (a leaf of 9 has boxes below the Gram form's widths, eps 1e-7 takes none)
@pytest.mark.parametrize("leaf,eps", [(64, 1e-6), (9, 1e-6), (64, 1e-7)])
def test_saved_table_gives_the_same_factor(pkg, lib, leaf, eps):
    pts = torch.from_numpy(inputs.grid_points(72, 2)).cuda()
    x = torch.from_numpy(inputs.rhs(11, 72 * 72, 2)).cuda()
    for e in (1e-6, 1e-7):  # the keys of both forms are in the table
        pkg.Factorization(pts, 0, e, leaf=leaf, prec=pkg.MIXED)
    f = pkg.Factorization(pts, 0, eps, leaf=leaf, prec=pkg.MIXED)
    table = pkg.autotune_table()
    assert table
    _restore(lib, table)
    g = pkg.Factorization(pts, 0, eps, leaf=leaf, prec=pkg.MIXED)
    assert np.array_equal(f.stats()["k"], g.stats()["k"])
    assert torch.equal(f.apply(x), g.apply(x))


@pytest.mark.parametrize("leaf,n,width", [(64, 3000, (64, 128)), (200, 2600, (256,))])
def test_householder_shapes_of_the_fp32_factor(pkg, lib, leaf, n, width):
    """Tolerance: the suite's bar of ten times eps for FP32 factors at their
    smallest tolerances, 10 x 4e-7."""
    eps = 4e-7
    pts = torch.from_numpy(inputs.random_points(93, n, 2)).cuda()
    x = torch.from_numpy(inputs.rhs(94, n, 2)).cuda()
    for tpc, g, c, rows in pkg.rss.AUTOTUNE_SHAPES:
        fits = [w for w in width if pkg.rss.shape_fits(w, tpc, g, rows) and not (w == 256 and c > 1 and tpc != 2)]
        if not fits:
            continue
        lib.rss_autotune_clear()
        for w in fits:
            for cls in range(20):
                assert lib.rss_autotune_set(4, w, cls, tpc, g, c, rows) == 0
        f = pkg.Factorization(pts, 0, eps, leaf=leaf, prec=pkg.MIXED)
        ax = f.matvec(x)
        assert float(torch.linalg.norm(f.apply(x) - ax) / torch.linalg.norm(ax)) <= 10 * eps, (tpc, g, c, rows)
