"""Roots of Eq. 11 far from where an iteration expects them: problems (tiny eps,
wide windows, misjudged sigma) whose lambda jumps by factors of 16 to 88 up or
14 to 48 down between the third and the fifth iteration.  Every iteration has to
resolve its root: status 0, and lambda within the bound that its condition
number gives (test_gpu_parity.lambda_tolerance) of the oracle's root for the
same iterate."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import oracle as O  # noqa: E402
import synthetic as S  # noqa: E402
import paper_1609_01839_gb300 as gfd  # noqa: E402
from test_gpu_parity import lambda_tolerance  # noqa: E402

DEV = torch.device("cuda:0")
PSF = {"g": lambda: S.psf_gaussian(25, 1.6), "u5": lambda: S.psf_uniform(5), "u9": lambda: S.psf_uniform(9), "m": S.psf_motion}
# seed, PSF, BSNR, sigma's factor, window, eps, texture, rho (0: Eq. 12), the jump
CASES = [(31, "u5", 7.2, 0.94, 9, 1.1883357636221632e-05, 0.1, 1.0, 16.3),
         (29, "m", 22.4, 1.678, 17, 1.3468658156013927e-05, 0.1, 0.0, 88.1),
         (32, "m", 14.5, 1.731, 17, 2.1108186724396855e-05, 0.1, 0.0, 0.070),
         (5, "m", 18.8, 1.42, 17, 2.0819191614853472e-05, 0.02, 1.0, 0.021)]
# a second lambda 23 000 times the first (2400 times is the far end of the bracket
# tried beside the expected one)
FAR = (21, "g", 25.6, 2.174, 17, 1.13e-05, 0.02, 1.0, 23000.0)


def problem(seed, psf, bsnr, fac, w, eps, tex, rho, jump):
    rng = np.random.default_rng(seed)
    u = S.image_polygons(seed, 64, 64, n_poly=6, texture_std=tex, rng=rng)
    h = PSF[psf]()
    b = S.blur_circular(u, h)
    sg = math.sqrt(b.var() / 10.0 ** (bsnr / 10.0))
    y = (b + sg * rng.standard_normal((64, 64))).astype(np.float32)
    return y, h.astype(np.float32), fac * sg


@pytest.mark.parametrize("rows,cols", [(1, 1), (32, 32)])
@pytest.mark.parametrize("case", CASES, ids=lambda c: f"x{c[8]}")
def test_jumping_lambda(case, rows, cols):
    """On 64 x 64, and on 2048 x 2048 canvases holding the same image 32 x 32
    times (the same roots), whose fallback passes are launched otherwise."""
    y, h, sigma = problem(*case)
    _, _, _, _, w, eps, _, rho, jump = case
    f = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(DEV)  # noqa: E731
    iters = 6
    item = {"y": f(np.tile(y, (rows, cols))), "h": f(h), "sigma": sigma, "w": w, "eps": eps}
    with gfd.Context(0, rho=rho) as c:
        c.solve_batched([item], iters, want_checkpoints=True)
        torch.cuda.synchronize()
        status = c.status(1)
    lam = item["lam"].cpu().numpy()
    H = O.psf_spectrum(h.astype(np.float64), 64, 64)
    Y = np.fft.fft2(y.astype(np.float64))
    T = O.discrepancy_target(y.astype(np.float64), h.astype(np.float64), sigma, rho or None)
    a = np.abs(H) ** 2
    ratios = []
    for k in range(iters):
        UE = np.fft.fft2(item["u_iters"][k, :64, :64].cpu().numpy().astype(np.float64))
        ref, res, _ = O.solve_lambda(H, Y, UE, T)
        r = np.abs(H * UE - Y) ** 2
        f1, f0 = O.f_lambda(ref * 1.001, a, r, 4096), O.f_lambda(ref / 1.001, a, r, 4096)
        kappa = 2 * math.log(1.001) / abs(math.log(f1) - math.log(f0))
        assert abs(lam[k] / ref - 1) < lambda_tolerance(kappa, 1e-6), (k, lam[k], ref, kappa)
        ratios.append(lam[k] / lam[k - 1] if k >= 3 else 1.0)
    assert status == [0]
    assert max(ratios) > 0.8 * jump if jump > 1 else min(ratios) < 1.25 * jump  # it did jump


@pytest.mark.parametrize("passes", [2, 3, 4, 16])
def test_far_second_lambda(passes):
    """Resolved by two passes: [150, 2400] lambda_0 is tried first only where
    enough passes are left for a root beyond it."""
    y, h, sigma = problem(*FAR)
    f = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(DEV)  # noqa: E731
    with gfd.Context(0, rho=FAR[7], lambda_max_passes=passes) as c:
        item = {"y": f(y), "h": f(h), "sigma": sigma, "w": FAR[4], "eps": FAR[5]}
        c.solve_batched([item], 2, want_checkpoints=True)
        torch.cuda.synchronize()
        assert c.status(1) == [0]
    H = O.psf_spectrum(h.astype(np.float64), 64, 64)
    Y = np.fft.fft2(y.astype(np.float64))
    T = O.discrepancy_target(y.astype(np.float64), h.astype(np.float64), sigma, FAR[7])
    lam = item["lam"].cpu().numpy()
    a = np.abs(H) ** 2
    for k in range(2):
        UE = np.fft.fft2(item["u_iters"][k].cpu().numpy().astype(np.float64))
        ref, _, _ = O.solve_lambda(H, Y, UE, T)
        r = np.abs(H * UE - Y) ** 2
        f1, f0 = O.f_lambda(ref * 1.001, a, r, 4096), O.f_lambda(ref / 1.001, a, r, 4096)
        kappa = 2 * math.log(1.001) / abs(math.log(f1) - math.log(f0))
        assert abs(lam[k] / ref - 1) < lambda_tolerance(kappa, 1e-6), (k, lam[k], ref, kappa)
    assert lam[1] > 0.8 * FAR[8] * lam[0]
