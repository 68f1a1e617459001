"""Gradients over window sizes and canvas shapes: the adjoint's tiles (32 x 16
pixels and a halo of 2 r) larger than the canvas, windows wider than it, canvases
that are not square, one and 17 pixels of window, several windows in one call.

Reference: the oracle's FP64 gradient.  Tolerance: 1e-4 relative in norm, the bar
of the other gradient tests, and 30 times what the gradient moves by when the
image moves by 1e-7 of itself (FP32 rounds at 6e-8, some tens of times over)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import synthetic as S  # noqa: E402
import paper_1609_01839_gb300 as gfd  # noqa: E402
from oracle import adjoint as A  # noqa: E402

DEV = torch.device("cuda:0")


def problem(M, N, w, seed=11):
    rng = np.random.default_rng(seed)
    u0 = S.image_polygons(seed, M, N, n_poly=8, texture_std=0.02, rng=rng)
    h = S.psf_gaussian(5 if min(M, N) < 16 else 9, 1.0)
    y = S.blur_circular(u0, h) + rng.standard_normal((M, N)) / 255
    return y.astype(np.float32), h.astype(np.float32), 1.0 / 255, w, 1e-3, u0.astype(np.float32)


def check(ctx, probs, iters):
    t = lambda a: torch.from_numpy(a).to(DEV)  # noqa: E731
    items = [{"y": t(y), "h": t(h), "sigma": s, "w": w, "eps": e} for y, h, s, w, e, _ in probs]
    ctx.solve_batched(items, iters, want_checkpoints=True)
    got = ctx.backward_batched(
        items, iters, [2.0 * (i["u"] - t(p[5])) / p[5].size for i, p in zip(items, probs)])
    noise = np.random.default_rng(0)
    for (y, h, s, w, e, uc), g in zip(probs, got):
        ref = A.solve_with_grad(y, h, s, w, e, iters, uc)
        assert np.isfinite(ref["lam"]).all()
        near = A.solve_with_grad(y * (1 + 1e-7 * noise.standard_normal(y.shape)), h, s, w, e, iters, uc)
        for key, v in zip(("g_y", "g_h", "g_eps"), g):
            r = np.atleast_1d(ref[key])
            d = np.linalg.norm(np.atleast_1d(v.cpu().numpy().astype(np.float64)) - r)
            tol = 1e-4 * np.linalg.norm(r) + 30 * np.linalg.norm(np.atleast_1d(near[key]) - r)
            assert d <= tol, (key, y.shape, w, d / np.linalg.norm(r))


@pytest.mark.parametrize("M, N", [(8, 8), (16, 64), (64, 16), (128, 32)])
@pytest.mark.parametrize("w", [1, 3, 9, 17])
def test_windows_and_canvases(M, N, w):
    """(With w = 1 the filter returns u_p, which meets the constraint by itself:
    a second step would rest on the rounding of its residual.)"""
    with gfd.Context(0) as c:
        check(c, [problem(M, N, w)], 1 if w == 1 else 3)


def test_several_windows_in_one_call():
    with gfd.Context(0) as c:
        check(c, [problem(64, 16, w, 20 + w) for w in (9, 3, 17, 3, 5)], 2)
