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


@pytest.mark.parametrize("M,N", [(256, 64), (512, 16), (1024, 32), (2048, 8), (64, 256)])
def test_every_tile_width(tmp_path, M, N):
    """A solve with each tile width the column passes are compiled for: 2e-5 of
    the default's result (the per-iteration bar on u)."""
    rng = np.random.default_rng(M + N)
    y = torch.from_numpy(rng.random((M, N)).astype(np.float32)).to(DEV)
    h = torch.full((3, 3), 1.0 / 9.0, device=DEV)
    ref = None
    for threads in (256, 128, 64, 32):
        path = tmp_path / f"t{threads}.txt"
        path.write_text(f"chains 1\nclass {M} {N} col_threads {threads} row_threads 64 gf_rows 16\n")
        with gfd.Context(0, tune_cache=str(path)) as c:
            u, lam, _ = c.solve(y, h, 0.05, 5, 1e-3, 6)
            torch.cuda.synchronize()
            assert c.status(1) == [0]
        ref = u if ref is None else ref
        assert float((u - ref).abs().max()) < 2e-5
