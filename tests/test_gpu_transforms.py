"""Every transform length of the library's row and column passes against the
FP64 DFT, forward and inverse, and every tile width of the fused column passes
against the default one.  Tolerance: 1e-6 of the spectrum's (image's) norm, the
bar of the other transform tests: an FP32 transform of up to 24 binary stages
carries about sqrt(24) * 6e-8 = 3e-7."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1609_01839_gb300 as gfd  # noqa: E402

DEV = torch.device("cuda:0")
SIZES = [8, 16, 32, 64, 128, 256, 512, 1024, 2048, 4096]


@pytest.fixture(scope="module")
def ctx():
    c = gfd.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("M,N", [(s, 8) for s in SIZES] + [(8, s) for s in SIZES[1:]] + [(512, 2048)])
def test_every_length_round_trip(ctx, M, N):
    g = torch.Generator(device=DEV)
    g.manual_seed(M * 5000 + N)
    x = torch.rand(M, N, generator=g, device=DEV)
    X = ctx.fft2_r2c(x)
    F = torch.fft.rfft2(x.double())
    ref = F[:, :-1].clone()
    ref[:, 0] = F[:, 0] + 1j * F[:, -1]
    assert float((X.to(torch.complex128) - ref).norm() / ref.norm()) < 1e-6
    back = ctx.fft2_c2r(X)
    assert float((back.double() - x.double()).norm() / x.double().norm()) < 1e-6


def observation(rng, M, N, kh, kw, sigma):
    """8 x 8 blocks of random brightness, a kh x kw mean, Gaussian noise."""
    u = np.kron(rng.random((M // 8, N // 8)), np.ones((8, 8)))
    b = sum(np.roll(u, (i, j), (0, 1)) for i in range(-(kh // 2), kh // 2 + 1)
            for j in range(-(kw // 2), kw // 2 + 1)) / (kh * kw)
    y = b + sigma * rng.standard_normal((M, N))
    return torch.from_numpy(y.astype(np.float32)).to(DEV)


@pytest.mark.parametrize("M,N,n", [(256, 2048, 3), (512, 4096, 1), (1024, 2048, 1), (2048, 8, 1),
                                   (256, 64, 1), (1024, 512, 1), (32, 16, 1), (8, 16, 2)])
def test_every_tile_width(tmp_path, M, N, n):
    """A solve with each tile width that the column passes are compiled for, and
    canvases whose column passes are the short ones: 2e-5 of each other's
    results (the per-iteration bar on u)."""
    rng = np.random.default_rng(M + N)
    y = [observation(rng, M, N, 3, 3, 0.02) for _ in range(n)]
    h = torch.full((3, 3), 1.0 / 9.0, device=DEV)
    ref = None
    for threads in (256, 128, 64, 32):
        path = tmp_path / f"t{threads}.txt"
        path.write_text(f"chains 1\nclass {M} {N} col_threads {threads} row_threads 64 gf_rows 16\n")
        with gfd.Context(0, tune_cache=str(path)) as c:
            items = [{"y": v, "h": h, "sigma": 0.02, "w": 5, "eps": 1e-3} for v in y]
            c.solve_batched(items, 6)
            torch.cuda.synchronize()
            assert c.status(n) == [0] * n
        u = torch.stack([it["u"] for it in items])
        ref = u if ref is None else ref
        assert float((u - ref).abs().max()) < 2e-5


@pytest.mark.parametrize("M,N", [(8, 32), (16, 16), (64, 128), (512, 256), (1024, 64)])
def test_short_columns_equal_persistent(M, N):
    """The short column passes (one image) against the persistent ones (the same
    image in a batch large enough for them): lambda_0 to 1e-6, u to 2e-5."""
    rng = np.random.default_rng(M * N)
    n = (1 << 20) // (M * N) + 1
    y = observation(rng, M, N, 3, 5, 0.02)
    h = torch.full((3, 5), 1.0 / 15.0, device=DEV)
    with gfd.Context(0) as c:
        one = [{"y": y, "h": h, "sigma": 0.02, "w": 3, "eps": 1e-3}]
        c.solve_batched(one, 5)
        many = [{"y": y, "h": h, "sigma": 0.02, "w": 3, "eps": 1e-3} for _ in range(n)]
        c.solve_batched(many, 5)
        torch.cuda.synchronize()
        assert set(c.status(n)) == {0}
    assert abs(float(one[0]["lam"][0] / many[0]["lam"][0]) - 1.0) < 1e-6
    for it in (many[0], many[-1]):
        assert float((one[0]["u"] - it["u"]).abs().max()) < 2e-5
