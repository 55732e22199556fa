"""rss_matvec on scattered points under stream capture: an asynchronous factor's
call records kernels only (no allocation, so the graph can be instantiated more
than once), and calls from several threads do not disturb one another."""
import ctypes as C
import threading

import pytest

from paper_1609_08130_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

KERNEL_NODE = 0  # CU_GRAPH_NODE_TYPE_KERNEL


@pytest.fixture(scope="module")
def pkg():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_1609_08130_gb300 as p
    p.build()
    return p


def _factor(pkg, stream, n=1500, flags=0):
    pts = torch.from_numpy(inputs.random_points(41, n, 2)).cuda()
    return pkg.Factorization(pts, 0, 1e-4, leaf=64, prec=pkg.MIXED, stream=stream, flags=flags)


@pytest.mark.parametrize("cols", [1, 20])
def test_capture_records_kernels_only(pkg, cols):
    cu = C.CDLL("libcuda.so.1")
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        f = _factor(pkg, s, flags=pkg.rss.FLAG_ASYNC)
        x = torch.from_numpy(inputs.rhs(42, f.n, cols)).cuda()
        y = torch.zeros_like(x)
        call = lambda: pkg.lib().rss_matvec(f.h, C.c_void_p(x.data_ptr()), C.c_void_p(y.data_ptr()), cols)  # noqa: E731
        assert call() == pkg.rss.RSS_OK
        assert pkg.lib().rss_sync(f.h) == pkg.rss.RSS_OK
        st, graph, num = C.c_void_p(s.cuda_stream), C.c_void_p(), C.c_size_t()
        assert cu.cuStreamBeginCapture_v2(st, 2) == 0  # relaxed
        status = call()
        assert cu.cuStreamEndCapture(st, C.byref(graph)) == 0
        assert status == pkg.rss.RSS_OK
        assert cu.cuGraphGetNodes(graph, None, C.byref(num)) == 0 and num.value > 0
        nodes = (C.c_void_p * num.value)()
        assert cu.cuGraphGetNodes(graph, nodes, C.byref(num)) == 0
        kinds = []
        for node in nodes:
            k = C.c_int(-1)
            assert cu.cuGraphNodeGetType(C.c_void_p(node), C.byref(k)) == 0
            kinds.append(k.value)
        assert cu.cuGraphDestroy(graph) == 0
        assert all(k == KERNEL_NODE for k in kinds), kinds
        assert pkg.lib().rss_sync(f.h) == pkg.rss.RSS_OK


def test_calls_from_several_threads(pkg):
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        f = _factor(pkg, s)
        xs = [torch.from_numpy(inputs.rhs(50 + t, f.n, 3)).cuda() for t in range(4)]
        want = [f.matvec(x) for x in xs]
    torch.cuda.synchronize()
    bad = []

    def work(t):
        with torch.cuda.stream(s):
            for _ in range(20):
                if not torch.equal(f.matvec(xs[t]), want[t]):
                    bad.append(t)

    threads = [threading.Thread(target=work, args=(t,)) for t in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad
