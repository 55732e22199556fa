"""An rss_solve_noalloc captured in the caller's own CUDA graph keeps working
whatever other calls the factor serves between its replays: the memory its
launches refer to stays the factor's until rss_free, also when a call with
more columns than any before makes the factor take larger workspaces."""
import ctypes as C

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


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("cols", [1, 4])
def test_replay_after_wide_calls(pkg, prec, cols):
    lib = pkg.lib()
    p64 = prec == "fp64"
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        pts = torch.from_numpy(inputs.random_points(71, 6000, 2)).cuda()
        n = pts.shape[0]
        make = lambda: pkg.Factorization(pts, 0, 1e-6, leaf=64, prec=pkg.FP64 if p64 else pkg.MIXED,  # noqa: E731
                                         stream=s, flags=pkg.rss.FLAG_ASYNC)
        f = make()
        b = torch.from_numpy(inputs.rhs(72, n, cols)).cuda()
        wide = torch.from_numpy(inputs.rhs(73, n, 70)).cuda()
        x = torch.zeros_like(b)
        solve = lambda: lib.rss_solve_noalloc(f.h, C.c_void_p(b.data_ptr()), C.c_void_p(x.data_ptr()), cols)  # noqa: E731
        assert solve() == pkg.rss.RSS_OK  # the first call looks up the array and sets attributes
        assert lib.rss_sync(f.h) == pkg.rss.RSS_OK
        want = x.clone()
        torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s, capture_error_mode="relaxed"):
        assert solve() == pkg.rss.RSS_OK
    with torch.cuda.stream(s):
        for k in (5, 9, 70):
            x.fill_(float("nan"))
            g.replay()
            assert torch.equal(x, want)
            y = f.solve(wide[:k])
            f.apply(wide[:k])
            make()  # takes what memory the calls gave back to the pool
            x.fill_(float("nan"))
            g.replay()
            assert torch.equal(x, want)
            assert torch.equal(f.solve(wide[:k]), y)
        assert lib.rss_sync(f.h) == pkg.rss.RSS_OK
    torch.cuda.synchronize()
