"""What may come between two solves of one context: a timed solve, another stream,
a stream that is gone, a graph of the caller's.  Every result has to be the one
that a context of its own gives: the same bits on 64 x 64; above, where the sums
of y are added up by FP64 atomics in any order, lambda to 1e-9 (a last bit of T,
1e-16, times the condition number of Eq. 11, up to 1e6) and u to 2e-5, the bar on
u for a change of rounding."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import synthetic as S  # noqa: E402
import paper_1609_01839_gb300 as gfd  # noqa: E402

DEV = torch.device("cuda:0")


def problem(seed, M=64, N=64, k=5, sigma=0.02):
    rng = np.random.default_rng(seed)
    u = S.image_polygons(seed, M, N, n_poly=6, rng=rng)
    h = S.psf_uniform(k)
    y = S.blur_circular(u, h) + sigma * rng.standard_normal((M, N))
    f = lambda a: torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).to(DEV)  # noqa: E731
    return {"y": f(y), "h": f(h), "sigma": sigma, "w": 5, "eps": 1e-3}


def alone(item, iters):
    with gfd.Context(0) as c:
        u, lam, _ = c.solve(item["y"], item["h"], item["sigma"], item["w"], item["eps"], iters)
        torch.cuda.synchronize()
    return u, lam


def close(p, want):
    u, lam = want
    return (float((u - p["u"]).abs().max()) < 2e-5 and
            float((p["lam"] / lam - 1.0).abs().max()) < 1e-9)


@pytest.mark.parametrize("use_graphs", [True, False])
def test_timed_solves_between(use_graphs):
    a, b = problem(1), problem(2)
    want = {id(a): alone(a, 4), id(b): alone(b, 4)}
    with gfd.Context(0, use_graphs=use_graphs) as c:
        arr = {id(p): c.make_images([p], 4) for p in (a, b)}
        for p, timed in ((a, True), (a, False), (b, False), (b, True), (a, True), (b, False),
                         (b, True), (b, False), (a, False)):
            p["u"].zero_()
            torch.cuda.synchronize()
            if timed:
                c.solve_batched_timed(arr[id(p)], 4)
            else:
                c.solve_batched_images(arr[id(p)], 4)
            torch.cuda.synchronize()
            u, lam = want[id(p)]
            assert torch.equal(u, p["u"]) and torch.equal(lam, p["lam"])
            assert c.status(1) == [0]


def test_streams_without_a_wait_between():
    """Solves on streams in turn, of the same and of other buffers: the shared
    workspace is handed on in order."""
    items = [problem(10 + i, 128, 128) for i in range(4)]
    want = [alone(p, 6) for p in items]
    streams = [torch.cuda.Stream() for _ in range(3)]
    with gfd.Context(0) as c:
        arr = [c.make_images([p], 6) for p in items]
        torch.cuda.synchronize()
        for k in range(24):
            c.solve_batched_images(arr[(k // 2) % 4], 6, stream=streams[k % 3])
        torch.cuda.synchronize()
    assert all(close(p, w) for p, w in zip(items, want))


def test_streams_that_are_gone():
    """Streams destroyed with work pending, whose handles may be given again."""
    rt = torch.cuda.cudart()
    items = [problem(20 + i, 256, 256) for i in range(6)]
    want = [alone(p, 8) for p in items]
    with gfd.Context(0) as c:
        arr = [c.make_images([p], 8) for p in items]
        torch.cuda.synchronize()
        for a in arr:
            h = ctypes.c_void_p()
            assert int(rt.cudaStreamCreate(ctypes.addressof(h))) == 0
            rc = gfd.lib.gfdeconv_solve_batched(c._h, 1, a, 8, h)
            assert int(rt.cudaStreamDestroy(h.value)) == 0
            assert rc == 0
        torch.cuda.synchronize()
    assert all(close(p, w) for p, w in zip(items, want))


def test_solve_in_a_graph_of_the_callers():
    """A context without graphs of its own: a caller captures a solve."""
    a = problem(31, 256, 256)
    want = alone(a, 8)
    with gfd.Context(0, use_graphs=False) as c:
        arr = c.make_images([a], 8)
        c.solve_batched_images(arr, 8)
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            c.solve_batched_images(arr, 8)
        for _ in range(2):
            a["u"].zero_()
            g.replay()
            torch.cuda.synchronize()
            assert close(a, want)
