"""The colour filter over what its arithmetic must hold: every window radius at
tile edges, near-equal channels (a nearly singular covariance), a large offset,
a constant image.  Tolerance: 4 ulp of the output's size plus what the FP32
storage of a and b allows (|a . I| + |b| at 2^-24, averaged over w^2 windows: 1
ulp of that size), i.e. 5 * 2^-24 * (max|u| + max|a.I| + max|b|); the FP64
formula of the same reading is the reference."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import oracle as O  # noqa: E402
import paper_1609_01839_gb300 as gfd  # noqa: E402

DEV = torch.device("cuda:0")


@pytest.mark.parametrize("boundary", ("periodic", "truncated"))
@pytest.mark.parametrize("M,N,w,kind", [
    (16, 32, 1, "scene"), (32, 64, 3, "scene"), (64, 32, 5, "grey"), (16, 64, 7, "offset"),
    (8, 8, 17, "scene"), (32, 32, 11, "grey"), (64, 64, 13, "offset"), (128, 16, 15, "scene"),
    (32, 64, 9, "constant")])
def test_color_every_radius(M, N, w, kind, boundary):
    rng = np.random.default_rng(100 * w + M)
    I = rng.random((3, M, N))
    if kind == "grey":
        I = I[:1] + 1e-3 * rng.random((3, M, N))
    elif kind == "offset":
        I = 4.0 + 0.01 * I
    elif kind == "constant":
        I = np.full((3, M, N), 0.7)
    I = I.astype(np.float32)
    p = (I.mean(0) + 0.05 * rng.standard_normal((M, N))).astype(np.float32)
    eps = 1e-3
    ref = O.guided_filter_color(np.moveaxis(I, 0, -1), p, w, eps, boundary)
    b = gfd.BOUNDARY_TRUNCATED if boundary == "truncated" else gfd.BOUNDARY_PERIODIC
    with gfd.Context(0, boundary=b) as c:
        u = c.guidfilter_color(torch.from_numpy(I).to(DEV), torch.from_numpy(p).to(DEV), w, eps)
    err = np.abs(u.cpu().numpy().astype(np.float64) - ref).max()
    size = np.abs(ref).max() + 3.0 * np.abs(I).max() + np.abs(p).max()  # |a| is of order 1 here
    assert err <= 5.0 * 2.0 ** -24 * size, (err, size)
