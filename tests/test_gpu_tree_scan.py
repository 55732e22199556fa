"""The tree's scans at the edges of their rounds (8192 counts in one block, then
131072 a round over a cluster): the tree of n points equals the oracle's for
sizes whose digit counts, node counts and lists fall on either side."""
import numpy as np
import pytest

import oracle
from paper_1609_08130_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,dim,leaf", [(8191, 2, 64), (8192, 2, 8), (8193, 3, 64), (131072, 2, 64), (131073, 2, 500),
                                        (300001, 3, 300)])
def test_tree_of_many_points_matches_oracle(n, dim, leaf):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_1609_08130_gb300 as pkg
    pkg.build()
    pts = inputs.random_points(71, n, dim)
    t, o = pkg.Tree(torch.from_numpy(pts).cuda(), leaf), oracle.Tree(pts, leaf)
    assert t.nnode == o.nnode and t.maxdepth == o.maxdepth
    np.testing.assert_array_equal(t.perm(), o.perm())
    a, b = t.nodes(), o.nodes()
    for key in ("depth", "parent", "start", "count"):
        np.testing.assert_array_equal(np.asarray(a[key]), np.asarray(b[key]))
