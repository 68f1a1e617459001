"""What may come between two solves of one context: a timed solve, another stream,
a stream that is gone, a graph of the caller's.  Every result has to be the one
that a context of its own gives."""
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
