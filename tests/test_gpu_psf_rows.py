"""The PSF's transform reads only the canvas rows that the PSF reaches: PSFs of
one row, the neighbours of the canvas height, and beyond (the rows wrap).  ||h * u - y||^2 of the start values against the FP64 oracle to the
bar of the other residual tests, 1e-5 relative; y is unrelated to h * u, so the
residual is as large as the planes and far above the FP32 floor."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import oracle as O  # noqa: E402
import paper_1609_01839_gb300 as gfd  # noqa: E402

DEV = torch.device("cuda:0")


@pytest.mark.parametrize("M,N", [(8, 8), (16, 64), (256, 8)])
def test_psf_heights(M, N):
    rng = np.random.default_rng(M + N)
    f = lambda a: torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).to(DEV)  # noqa: E731
    items, refs = [], []
    for kh in (1, 3, M - 1, min(M + 1, 253), min(2 * M + 3, 251)):
        for kw in (1, 5, N + 1):
            h = rng.random((kh, kw)).astype(np.float32)
            h /= h.sum(dtype=np.float64).astype(np.float32)
            y, u = (rng.random((M, N)).astype(np.float32) for _ in range(2))
            items.append({"y": f(y), "h": f(h), "sigma": 0.02, "w": 3, "eps": 1e-3, "u_init": f(u)})
            d = np.fft.fft2(u.astype(np.float64)) * O.psf_spectrum(h.astype(np.float64), M, N)
            refs.append((np.abs(d - np.fft.fft2(y.astype(np.float64))) ** 2).sum() / (M * N))
    with gfd.Context(0) as c:
        c.solve_batched(items, 1, want_res=True)
        torch.cuda.synchronize()
    got = [float(it["res"][0]) for it in items]
    assert got == pytest.approx(refs, rel=1e-5)
