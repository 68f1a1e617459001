"""A context that solves images of one shape in different buffers keeps its
captured graph and refreshes the descriptors: every result has to be the one
that a context of its own gives, whatever changed between the calls (buffers,
PSF size, sigma, eps, start values, clean image, stream, window, size)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import synthetic as S  # noqa: E402
import paper_1609_01839_gb300 as gfd  # noqa: E402

DEV = torch.device("cuda:0")


def problem(seed, M, N, k, sigma):
    rng = np.random.default_rng(seed)
    u = S.image_polygons(seed, M, N, n_poly=6, rng=rng)
    h = S.psf_uniform(k)
    y = S.blur_circular(u, h) + sigma * rng.standard_normal((M, N))
    f = lambda a: torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).to(DEV)  # noqa: E731
    return f(y), f(h), f(u)


def test_calls_of_one_shape_in_other_buffers():
    calls = []  # (M, N, psf, sigma, w, eps, iters, init, clean, stream)
    side = torch.cuda.Stream()
    for i, (M, N, k, sg, w, eps, it, init, clean, st) in enumerate([
            (64, 64, 5, 0.02, 5, 1e-3, 4, False, False, None),
            (64, 64, 5, 0.02, 5, 1e-3, 4, False, False, None),
            (64, 64, 9, 0.01, 5, 1e-3, 4, False, True, None),
            (64, 64, 3, 0.03, 5, 1e-2, 4, True, False, side),
            (64, 64, 5, 0.02, 5, 1e-3, 4, False, False, None),
            (64, 64, 5, 0.02, 7, 1e-3, 4, False, False, None),
            (32, 64, 5, 0.02, 7, 1e-3, 4, False, True, side),
            (32, 64, 5, 0.02, 7, 1e-3, 3, False, False, None)]):
        y, h, u = problem(100 + i, M, N, k, sg)
        calls.append((y, h, sg, w, eps, it, u if clean else None, y.clone() if init else None, st))
    torch.cuda.synchronize()
    got = []
    with gfd.Context(0) as c:
        for y, h, sg, w, eps, it, uo, ui, st in calls:  # no wait between the calls
            got.append(c.solve(y, h, sg, w, eps, it, u_orig=uo, u_init=ui, stream=st))
        torch.cuda.synchronize()
    for (y, h, sg, w, eps, it, uo, ui, _), (u, lam, isnr) in zip(calls, got):
        with gfd.Context(0) as c:
            u1, lam1, isnr1 = c.solve(y, h, sg, w, eps, it, u_orig=uo, u_init=ui)
            torch.cuda.synchronize()
        assert torch.equal(u, u1) and torch.equal(lam, lam1)
        assert (isnr is None) == (isnr1 is None)
        if isnr is not None:
            assert float((isnr - isnr1).abs().max()) < 1e-6


def test_batches_of_one_shape_in_other_order_of_buffers():
    probs = [problem(7 + i, 32 << (i % 2), 64, 3 + 2 * i, 0.02) for i in range(4)]
    make = lambda order: [{"y": probs[i][0], "h": probs[i][1], "sigma": 0.02, "w": 5,  # noqa: E731
                           "eps": 1e-3} for i in order]
    with gfd.Context(0) as c:
        a = c.solve_batched(make([0, 1, 2, 3]), 3)
        b = c.solve_batched(make([2, 3, 0, 1]), 3)
        torch.cuda.synchronize()
        for i, j in ((0, 2), (1, 3), (2, 0), (3, 1)):
            assert torch.equal(a[i]["u"], b[j]["u"]) and torch.equal(a[i]["lam"], b[j]["lam"])
        assert c.status(4) == [0] * 4
