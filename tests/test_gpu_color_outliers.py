"""The colour filter where values are not alike: bright pixels in a dark image, tiny
eps, scales far from one, values that are not finite.  A pixel may touch the
windows that hold it and no others.

The reference is the formula in extended precision.  Tolerance, pixel by pixel: 5
roundings of s + |u| with s = sum box(|a_c|) |I_c| + box(|b|) (FP32 storage of a
and b, their products, the output), and what FP64 sums allow, 16 * 2^-53 * s
times the largest I^2 that the pixel's windows hold over eps."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1609_01839_gb300 as gfd  # noqa: E402

DEV = torch.device("cuda:0")
LD = np.longdouble


def shifts(x, r):
    for i in range(-r, r + 1):
        for j in range(-r, r + 1):
            yield np.roll(x, (i, j), (0, 1))


def box(x, r):
    return sum(shifts(x, r)) / LD((2 * r + 1) ** 2)


def widest(x, r):
    return np.max(np.stack(list(shifts(x, r))), axis=0)


def reference(I, p, w, eps):
    """u and the tolerance, pixel by pixel (periodic windows)."""
    r = (w - 1) // 2
    I, p, eps = I.astype(LD), p.astype(LD), LD(eps)
    mu, pb = [box(c, r) for c in I], box(p, r)
    S = [[box(I[i] * I[j], r) - mu[i] * mu[j] + (eps if i == j else 0) for j in range(3)]
         for i in range(3)]
    v = [box(I[i] * p, r) - mu[i] * pb for i in range(3)]
    cof = [[S[(i + 1) % 3][(j + 1) % 3] * S[(i + 2) % 3][(j + 2) % 3] -
            S[(i + 1) % 3][(j + 2) % 3] * S[(i + 2) % 3][(j + 1) % 3] for j in range(3)]
           for i in range(3)]
    det = sum(S[0][j] * cof[0][j] for j in range(3))
    a = [sum(cof[i][j] * v[j] for j in range(3)) / det for i in range(3)]
    b = pb - sum(a[i] * mu[i] for i in range(3))
    u = sum(box(a[i], r) * I[i] for i in range(3)) + box(b, r)
    s = sum(box(abs(a[i]), r) * abs(I[i]) for i in range(3)) + box(abs(b), r)
    cond = widest((I * I).max(0), 2 * r) / eps
    return u, 5 * LD(2) ** -24 * (s + abs(u)) + 16 * LD(2) ** -53 * cond * s


def gpu(I, p, w, eps):
    with gfd.Context(0) as c:
        u = c.guidfilter_color(torch.from_numpy(I).to(DEV), torch.from_numpy(p).to(DEV), w, eps)
    return u.cpu().numpy()


def inputs(seed, top=0.1, M=64, N=64):
    rng = np.random.default_rng(seed)
    I = (top * rng.random((3, M, N))).astype(np.float32)
    p = (I.mean(0) + 0.1 * top * rng.standard_normal((M, N))).astype(np.float32)
    return I, p


def check(I, p, w, eps, where=None):
    u, tol = reference(I, p, w, eps)
    err = abs(gpu(I, p, w, eps).astype(LD) - u)
    bad = ~(err <= tol)
    if where is not None:
        bad &= where
    assert not bad.any(), (float((err / tol)[bad].max()), np.argwhere(bad)[:5])


@pytest.mark.parametrize("w", [1, 3, 9, 17])
@pytest.mark.parametrize("bright", [10.0, 1e3, 1e4])
@pytest.mark.parametrize("at", [(8, 16), (24, 48), (3, 5), (16, 32)])  # two of them tile centres
def test_bright_pixel(w, bright, at):
    I, p = inputs(1)
    I[:, at[0], at[1]] = bright
    p[at] = bright
    check(I, p, w, 1e-3)
    I, p = inputs(2)
    p[at] = bright
    check(I, p, w, 1e-3)


@pytest.mark.parametrize("eps", [1e-4, 1e-6, 1e-8, 1e-10])
def test_small_eps(eps):
    I, p = inputs(3, top=1.0)
    I = (I[:1] + 1e-3 * I).astype(np.float32)
    check(I, p, 5, eps)


@pytest.mark.parametrize("si,sp", [(1e20, 1.0), (1e-20, 1.0), (1.0, 1e30), (1.0, 3e38), (1.0, 1e-30),
                                   (1e18, 1e18), (1e-18, 1e18)])
def test_scales(si, sp):
    """GF(s I, t p, s^2 eps) = t GF(I, p, eps)."""
    I, p = inputs(4, top=1.0)
    check((I * np.float32(si)).astype(np.float32), np.minimum(p, 1.1).astype(np.float32) * np.float32(sp),
          3, 1e-3 * si * si)


@pytest.mark.parametrize("value", [np.nan, np.inf, -np.inf])
@pytest.mark.parametrize("plane", [0, 3])
@pytest.mark.parametrize("at", [(8, 16), (0, 0), (31, 33), (17, 63)])
def test_not_finite(value, plane, at):
    w, r = 5, 2
    I, p = inputs(5, top=1.0)
    J, q = I.copy(), p.copy()
    if plane < 3:
        J[plane][at] = value
    else:
        q[at] = value
    dist = np.maximum(*[np.minimum(abs(np.arange(64) - c), 64 - abs(np.arange(64) - c)).reshape(s)
                        for c, s in zip(at, ((64, 1), (1, 64)))])
    u, tol = reference(I, p, w, 1e-3)  # beyond 2 r the value does not matter
    got = gpu(J, q, w, 1e-3)
    assert not np.isfinite(got[dist <= 2 * r]).any()
    assert (abs(got.astype(LD) - u) <= tol)[dist > 2 * r].all()


@pytest.mark.parametrize("eps", [1e-5, 1e-4, 1e-2])
@pytest.mark.parametrize("low", [0.0, 1e-3, 0.05])
def test_two_levels(eps, low):
    """Tiles half dark, half bright: the dark windows keep their own accuracy."""
    I, p = inputs(6, top=0.01)
    edge = (np.add.outer(np.arange(64), 2 * np.arange(64)) % 90) < 40
    I = (I + np.where(edge, 0.9, low)).astype(np.float32)
    p = (abs(p) + np.where(edge, 0.8, low)).astype(np.float32)
    check(I, p, 9, eps)


@pytest.mark.parametrize("w", [1, 3, 9, 17])
@pytest.mark.parametrize("level", [1.0, 1000.0])
@pytest.mark.parametrize("spread", [2.0 ** -23, 1e-6, 1e-4, 3e-3])
def test_nearly_flat_planes(w, level, spread):
    """Planes that hardly move about a value far from zero (clipped highlights), some or
    all of them: the grid is then as coarse as the value asks for."""
    I, p = inputs(31, top=level)
    rng = np.random.default_rng(32)
    near = lambda: (level * (1 - spread * rng.random(p.shape))).astype(np.float32)  # noqa: E731
    for flat in ([2], [0, 1, 2, 3]):
        J, q = I.copy(), p.copy()
        for k in flat:
            if k < 3:
                J[k] = near()
            else:
                q = near()
        eps = 1e-3 * level ** 2
        u, tol = reference(J, q, w, eps)
        assert (np.abs(gpu(J, q, w, eps) - u) <= tol).all(), flat


@pytest.mark.parametrize("seed", [41, 42])
def test_black_and_grey_fields(seed):
    """A grey image in three channels (a matrix singular but for eps), black fields beside
    bright ones, eps at the end of the split's range (R^2 = 2^16 eps): the remainders
    are half a grid step at most, so that the black fields keep the tolerance."""
    rng = np.random.default_rng(seed)
    i, j = np.mgrid[:64, :64]
    g = np.where((i // 13 + j // 17) % 2 == 0, 0.6, 0.0) + 1e-3 * rng.standard_normal((64, 64))
    I = np.stack([np.clip(g, 0, 1).astype(np.float32)] * 3)
    p = (I[0] + 0.03 * rng.standard_normal((64, 64))).astype(np.float32)
    check(I, p, 9, 1e-5)
