"""The fallback passes of small canvases run as one cluster of blocks per image.
A batch whose clusters outnumber what is resident at once, so that they start
one after another, has to give every image what it gets alone: lambda_0 comes
out of the same sums in the same order, so it is the same number."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import synthetic as S  # noqa: E402
import paper_1609_01839_gb300 as gfd  # noqa: E402

DEV = torch.device("cuda:0")


@pytest.mark.parametrize("M,N,n", [(64, 64, 250), (16, 32, 1500)])
def test_more_clusters_than_fit(M, N, n):
    rng = np.random.default_rng(M)
    f = lambda a: torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).to(DEV)  # noqa: E731
    h = S.psf_uniform(5)
    make = [{"y": f(S.blur_circular(rng.random((M, N)), h) + 0.02 * rng.standard_normal((M, N))),
             "h": f(h), "sigma": 0.02, "w": 3, "eps": 1e-3} for _ in range(n)]
    items = [dict(it) for it in make]
    with gfd.Context(0) as c:
        c.solve_batched(items, 2)
        torch.cuda.synchronize()
        assert set(c.status(n)) == {0}
    with gfd.Context(0) as c:
        for i in (0, 1, n // 2, n - 1):
            u, lam, _ = c.solve(make[i]["y"], make[i]["h"], 0.02, 3, 1e-3, 2)
            torch.cuda.synchronize()
            assert float(lam[0]) == float(items[i]["lam"][0])
            assert float((u - items[i]["u"]).abs().max()) < 2e-5
